// Stage 2 of the two-stage scheme: the classical parallel circuit of
// Section 2 (Eqs. 1-3, Fig. 1(c)) that turns the stage-1 quantities into the
// solutions z = y ^ z^a, y in Col(A), one after another.
//
// On the GPU the paper's binary counter over R^(r) becomes the reflected Gray
// code over the RREF basis (the reading stated in hlf.h):
//     z(i) = z0 ^ XOR_{k in g(i)} B_k,  g(i) = i ^ (i >> 1),
// so consecutive solutions differ by one basis row, z(i+1) = z(i) ^ B_ctz(i+1),
// and any window can be seeded independently with <= 64 row XORs.
//
// Kernels
//   reduce_kernel        each thread seeds its own contiguous run of indices
//                        and walks it one XOR per solution; blocks of 2^U
//                        solutions are unrolled so that the first U basis
//                        rows are compile-time register operands. The
//                        per-thread (count, hash sum, XOR-fold) is reduced by
//                        warp shuffles, shared memory and, where several
//                        CTAs share a window, one 64-bit atomic per quantity
//                        per CTA. One window or many (a result per chunk).
//                        Windows too short to give a full wave long runs are
//                        bound by how many threads walk them: runs go down
//                        to one Gray block.
//   store_kernel         coalesced materialisation by groups of 64 or 32
//                        consecutive solutions a warp step (store_groups): one
//                        XOR per solution, 512 B a step at W = 1; at W > 1 the
//                        lanes' solutions are restaged in shared memory so that
//                        the warp writes its 32*W words with consecutive lanes
//                        on consecutive words. Bound by HBM stores.
//   sample_kernel        z(i) at arbitrary indices, straight from the formula.

#include "enum_impl.cuh"

namespace hlf {
namespace {



// The reduce of n_chunks windows of `chunk` indices, window c starting at
// offset + c * chunk (hlf_enumerate_reduce is one window). A window is cut into
// `parts` CTAs of blockDim.x threads, each thread walking `per` consecutive
// indices that start at a multiple of 2^U, so that only the window's two ends
// have partial Gray blocks. Items (window, part) are taken grid-stride. With
// one part per window the CTA writes the result; otherwise it adds to it.
template <int W, int U, int T>
__global__ void __launch_bounds__(T, min_ctas_for(W))
    reduce_kernel(const uint64_t* __restrict__ table, uint64_t offset, uint64_t chunk, uint64_t n_chunks,
                  uint32_t parts, uint64_t per, uint64_t runs, uint64_t align, int ntab,
                  hlf_reduce* __restrict__ out)
{
    __shared__ Table<W> t;
    __shared__ SeedTable<W> st;
    const bool mixed = __syncthreads_or(load_table_hash_domain<W, U>(t, table));
    build_seed_table<W>(st, t, ntab);
    __syncthreads();
    for (uint64_t item = blockIdx.x; item < n_chunks * parts; item += gridDim.x) {
        const uint64_t c = item / parts;
        const uint64_t first = offset + c * chunk;
        const uint64_t skip = first & align;  // indices before the window in its first block
        const uint64_t run = (item - c * parts) * blockDim.x + threadIdx.x;
        const uint64_t a = run * per;  // counted from that block's start
        Acc<W> acc;
        acc.zero();
        uint64_t cnt = 0;
        const uint64_t lo = max(a, skip);
        if (run < runs && lo - skip < chunk) {
            cnt = min(per - (lo - a), chunk - (lo - skip));
            uint64_t z[W];
            const uint64_t i = first + (lo - skip);
            seed_lookup<W>(st, ntab, i, z);
            reduce_run_from<W, U>(t, mixed, i, cnt, z, acc);
        }
        block_reduce<W, T>(cnt, acc);
        if (threadIdx.x != 0) continue;
        hlf_reduce& r = out[c];
        if (parts == 1) {
            r.count = cnt;
            r.hsum = acc.hs;
#pragma unroll
            for (int w = 0; w < HLF_MAX_W; ++w) r.xor_fold[w] = w < W ? acc.fold_word(w < W ? w : 0) : 0ull;
        } else if (cnt) {
            atomicAdd(reinterpret_cast<unsigned long long*>(&r.count), (unsigned long long)cnt);
            atomicAdd(reinterpret_cast<unsigned long long*>(&r.hsum), (unsigned long long)acc.hs);
#pragma unroll
            for (int w = 0; w < W; ++w) {
                const uint64_t f = acc.fold_word(w);
                if (f) atomicXor(reinterpret_cast<unsigned long long*>(&r.xor_fold[w]), (unsigned long long)f);
            }
        }
    }
}

struct StorePlan {
    uint64_t offset, count;
    GroupPlan g;
    uint64_t per_warp;  // groups per warp
};

template <int W>
__global__ void __launch_bounds__(kThreads) store_kernel(const uint64_t* __restrict__ table,
                                                         const __grid_constant__ StorePlan pl,
                                                         uint64_t* __restrict__ out)
{
    constexpr int M = Groups<W>::kLog2;
    extern __shared__ __align__(16) uint64_t s_stage[];  // W > 1: [warps][stage_words<W>()]
    __shared__ Table<W> t;
    __shared__ uint64_t s_C[kTableRows - M][W];  // C_j = B_{M-1} ^ B_{M+j}
    load_table<W>(t, table);
    __syncthreads();
    for (int i = threadIdx.x; i < (kTableRows - M) * W; i += blockDim.x) {
        const int j = i / W, w = i % W;
        s_C[j][w] = t.B[M - 1][w] ^ t.B[M + j][w];
    }
    __syncthreads();

    const uint64_t gt = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    // ragged head and tail, one index per thread, from the definition
    if (gt < pl.g.n_head + pl.g.n_tail) {
        const uint64_t i = gt < pl.g.n_head ? pl.offset + gt : pl.g.tail_first + (gt - pl.g.n_head);
        uint64_t z[W];
        seed<W>(t, i, z);
        if (HLF_IN_BOUNDS(i - pl.offset, pl.count, kSiteStore)) {
#pragma unroll
            for (int w = 0; w < W; ++w) out[(i - pl.offset) * W + w] = z[w];
        }
    }
    __syncwarp();

    const uint64_t wg = gt >> 5;
    const int lane = threadIdx.x & 31;
    const uint64_t h0 = pl.g.h_first + wg * pl.per_warp;
    if (wg * pl.per_warp >= pl.g.h_end - pl.g.h_first) return;
    const uint64_t h1 = min(h0 + pl.per_warp, pl.g.h_end);
    uint64_t z[W];
    seed_group<W>([&](int k) { return k == kTableZ0Row ? t.z0 : t.B[k]; }, h0, lane, z);
    store_groups<W>(
        z, h0, h1, pl.g.odd, t.B[0][0], out - pl.offset * W, s_stage + (threadIdx.x >> 5) * stage_words<W>(), lane,
        [&](int j) { return s_C[j]; },
        [&](uint64_t i, uint64_t len) { return HLF_RANGE_IN_BOUNDS(i - pl.offset, len, pl.count, kSiteStore); });
}

// ----------------------------------------------------------------- sample

// An index is ceil(nb / 4) lookups a word in the seed tables. Walking its set Gray
// bits instead, each lane its own rows, 2^20 indices at W = 1 and r = 54 took 33 us.
template <int W>
__global__ void __launch_bounds__(kThreads) sample_kernel(const uint64_t* __restrict__ table, int nb,
                                                          const uint64_t* __restrict__ idx, uint64_t m,
                                                          uint64_t* __restrict__ out, int32_t* info)
{
    __shared__ Table<W> t;
    __shared__ SeedTable<W> st;
    load_table<W>(t, table);
    __syncthreads();
    const int ntab = nb ? (nb + 3) / 4 : 1;
    build_seed_table<W>(st, t, ntab);
    __syncthreads();
    for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < m; j += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t i = idx[j];
        uint64_t z[W];
        if (nb < 64 && (i >> nb)) {
            *reinterpret_cast<volatile int32_t*>(info) = HLF_ERR_RANGE;  // host-mapped status word
#pragma unroll
            for (int w = 0; w < W; ++w) z[w] = 0;
        } else {
            seed_lookup<W>(st, ntab, i, z);
        }
        if (HLF_IN_BOUNDS(j, m, kSiteStore)) {
#pragma unroll
            for (int w = 0; w < W; ++w) out[j * W + w] = z[w];
        }
    }
}

// ------------------------------------------------------------- launchers


// CTAs of `kernel` that fit on one SM at once (at least 1): grids are sized
// to one wave, since every kernel here gives its CTAs equal work and a
// partial second wave would cost a whole extra wave.
template <typename K>
int blocks_per_sm(K kernel, size_t smem)
{
    int fit = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, kernel, kThreads, smem) != cudaSuccess || fit < 1) {
        cudaGetLastError();
        return 1;
    }
    return fit;
}

// How a reduce of n_chunks windows of `chunk` indices is cut: CTAs of
// `threads`, `parts` of them per window, `per` indices per thread.
struct ReduceShape {
    unsigned threads, blocks;
    uint32_t parts;
    uint64_t per, runs;
    uint64_t align;  // runs start at multiples of align + 1
};

// The threads a window can use are one per Gray block of 2^U indices; a seed
// costs a few tens of solutions (kSeedCost), so short runs are worth it
// whenever they fill idle SMs. One window: one CTA if that holds them all (the
// result then needs no clearing), else all of them, up to one wave, in CTAs no
// larger than spreading them over every SM takes. Several windows: the largest
// CTA a window fills, and the cut whose waves cost least.
// With runs of at least 2048 indices and one CTA per window instead, 2^20
// four-word solutions took 694 us on one SM (now 12.4, two launches and the
// host's call among it), and 64 windows of 2^24 at W = 1 took 2.16 ms on 64
// CTAs of 256 threads (now 0.79).
template <int W, int U, int T>
ReduceShape reduce_shape(uint64_t chunk, uint64_t n_chunks)
{
    constexpr uint64_t kSeedCost = 48;
    const uint64_t sms = (uint64_t)sm_count();
    const uint64_t runs = ((chunk - 1) >> U) + 2;  // Gray blocks the window touches, at most
    const uint64_t room = (uint64_t)min_ctas_for(W) * T;  // threads an SM holds
    ReduceShape sh{};
    uint64_t want;  // threads for the window
    if (n_chunks == 1) {
        want = runs < sms * room ? runs : sms * room;
        uint64_t bd = want <= T ? want : (want + sms - 1) / sms;
        bd = (bd + 31) / 32 * 32;
        bd = bd > T ? T : (want > T && bd < 128 ? 128 : bd);
        sh.threads = (unsigned)bd;
        sh.parts = (uint32_t)((want + bd - 1) / bd);
    } else {
        uint64_t bd = T;
        while (bd > 64 && bd > runs) bd /= 2;
        sh.threads = (unsigned)bd;
        const uint64_t slots = sms * (room / bd);
        uint64_t best = ~0ull;
        for (uint64_t k = 1; k <= 64 && (k == 1 || (k - 1) * bd < runs); ++k) {
            const uint64_t waves = (n_chunks * k + slots - 1) / slots;
            const uint64_t cost = waves * (kSeedCost + (chunk + k * bd - 1) / (k * bd));
            if (cost < best) {
                best = cost;
                sh.parts = (uint32_t)k;
            }
            if (n_chunks > (~0ull >> 8)) break;  // a window each is enough
        }
    }
    want = (uint64_t)sh.parts * sh.threads;
    // chunk + 2^U - 1 indices at most, counted from the window's first block;
    // past 2^63 that count could wrap, so such windows start their runs at the
    // window's own start
    sh.align = chunk <= 1ull << 63 ? (1ull << U) - 1 : 0;
    sh.per = chunk / want + (chunk % want + sh.align + want - 1) / want;
    sh.per = (sh.per + (1ull << U) - 1) & ~((1ull << U) - 1);
    sh.runs = sh.align ? want : (chunk - 1) / sh.per + 1;
    const uint64_t items = n_chunks * sh.parts;
    const uint64_t cap = sms * (room / sh.threads);
    sh.blocks = (unsigned)(items < cap ? items : cap);
    return sh;
}

template <int W, int U>
hlf_status launch_reduce_u(const uint64_t* table, uint64_t offset, uint64_t chunk, uint64_t n_chunks,
                           hlf_reduce* out, cudaStream_t s)
{
    constexpr int T = reduce_threads(W);
    const ReduceShape sh = reduce_shape<W, U, T>(chunk, n_chunks);
    if (sh.parts > 1 && cudaMemsetAsync(out, 0, sizeof(hlf_reduce) * n_chunks, s) != cudaSuccess)
        return HLF_ERR_CUDA;
    const int ntab = seed_tables_for(offset + (chunk * n_chunks - 1));
    reduce_kernel<W, U, T><<<sh.blocks, sh.threads, 0, s>>>(table, offset, chunk, n_chunks, sh.parts, sh.per, sh.runs,
                                                           sh.align, ntab, out);
    return cudaGetLastError() == cudaSuccess ? HLF_OK : HLF_ERR_CUDA;
}

// W = 1 has two unrolls: 2^6 solutions per Gray block where every thread of a
// full wave has at least 16 blocks, else 2^3, whose finer cut balances and
// fills the SMs better than the deeper unroll saves.
template <int W>
hlf_status launch_reduce_w(const uint64_t* table, uint64_t offset, uint64_t chunk, uint64_t n_chunks,
                           hlf_reduce* out, cudaStream_t s)
{
    if constexpr (W == 1) {
        const uint64_t wave = (uint64_t)sm_count() * min_ctas_for(1) * reduce_threads(1);
        if (chunk * n_chunks < wave * 1024) return launch_reduce_u<1, 3>(table, offset, chunk, n_chunks, out, s);
    }
    return launch_reduce_u<W, reduce_unroll(W)>(table, offset, chunk, n_chunks, out, s);
}

// One wave of warps, each with consecutive groups; short windows give a warp one
// group and spread the warps over the SMs (2^14 solutions of two words on one CTA
// took 13 us, a group a warp on 64 CTAs takes 4).
template <int W>
hlf_status launch_store_w(const uint64_t* table, uint64_t offset, uint64_t count, uint64_t* out,
                          cudaStream_t s)
{
    StorePlan pl{};
    pl.offset = offset;
    pl.count = count;
    // W = 1: pairs on 16 bytes, whichever the parity of the window's first word
    const uint32_t odd = W == 1 ? ((reinterpret_cast<uintptr_t>(out) >> 3) ^ offset) & 1 : 0;
    pl.g = plan_groups(offset, count, Groups<W>::kSize, odd);
    const uint64_t groups = pl.g.h_end - pl.g.h_first;
    constexpr size_t smem_warp = W == 1 ? 0 : stage_words<W>() * sizeof(uint64_t);
    constexpr size_t smem_max = smem_warp * (kThreads / 32);
    static int fit[64] = {0};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 64) return HLF_ERR_CUDA;
    if (fit[dev] == 0) {
        if (W > 1 && cudaFuncSetAttribute(store_kernel<W>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)smem_max) != cudaSuccess)
            return HLF_ERR_CUDA;
        fit[dev] = blocks_per_sm(store_kernel<W>, smem_max);
    }
    const uint64_t sms = (uint64_t)sm_count();
    const uint64_t max_warps = sms * fit[dev] * (kThreads / 32);
    uint64_t warps = groups < max_warps ? groups : max_warps;
    if (warps == 0) warps = 1;
    pl.per_warp = groups ? (groups + warps - 1) / warps : 1;
    if (groups) warps = (groups + pl.per_warp - 1) / pl.per_warp;
    const uint64_t ragged = pl.g.n_head + pl.g.n_tail;
    uint64_t threads = warps * 32;
    if (threads < ragged) threads = ragged;
    uint64_t bd = (threads / sms + 31) / 32 * 32;
    bd = bd < 64 ? 64 : (bd > kThreads ? kThreads : bd);
    const unsigned blocks = (unsigned)((threads + bd - 1) / bd);
    store_kernel<W><<<blocks, (unsigned)bd, smem_warp * (bd / 32), s>>>(table, pl, out);
    return cudaGetLastError() == cudaSuccess ? HLF_OK : HLF_ERR_CUDA;
}

template <int W>
hlf_status launch_sample_w(const uint64_t* table, int nb, const uint64_t* idx, uint64_t m, uint64_t* out,
                           int32_t* info, cudaStream_t s)
{
    // CTAs of at least a few indices a thread, so that the tables are worth building
    const uint64_t cap = (uint64_t)sm_count() * 4;
    uint64_t blocks = (m + kThreads - 1) / kThreads;
    if (blocks > cap) blocks = cap;
    sample_kernel<W><<<(unsigned)blocks, kThreads, 0, s>>>(table, nb, idx, m, out, info);
    return cudaGetLastError() == cudaSuccess ? HLF_OK : HLF_ERR_CUDA;
}

#define HLF_DISPATCH_W(W, CALL)                     \
    switch (W) {                                    \
    case 1: return CALL(1);                         \
    case 2: return CALL(2);                         \
    case 3: return CALL(3);                         \
    case 4: return CALL(4);                         \
    case 5: return CALL(5);                         \
    case 6: return CALL(6);                         \
    case 7: return CALL(7);                         \
    case 8: return CALL(8);                         \
    case 9: return CALL(9);                         \
    case 10: return CALL(10);                       \
    case 11: return CALL(11);                       \
    case 12: return CALL(12);                       \
    case 13: return CALL(13);                       \
    case 14: return CALL(14);                       \
    case 15: return CALL(15);                       \
    case 16: return CALL(16);                       \
    default: return HLF_ERR_SIZE;                   \
    }

}  // namespace

hlf_status launch_reduce(const uint64_t* table, int W, uint64_t offset, uint64_t chunk, uint64_t n_chunks,
                         hlf_reduce* out, cudaStream_t s)
{
#define CALL(w) launch_reduce_w<w>(table, offset, chunk, n_chunks, out, s)
    HLF_DISPATCH_W(W, CALL)
#undef CALL
}

hlf_status launch_store(const uint64_t* table, int W, uint64_t offset, uint64_t count, uint64_t* out,
                        cudaStream_t s)
{
#define CALL(w) launch_store_w<w>(table, offset, count, out, s)
    HLF_DISPATCH_W(W, CALL)
#undef CALL
}

hlf_status launch_sample(const uint64_t* table, int W, int nb, const uint64_t* idx, uint64_t m,
                         uint64_t* out, int32_t* info, cudaStream_t s)
{
#define CALL(w) launch_sample_w<w>(table, nb, idx, m, out, info, s)
    HLF_DISPATCH_W(W, CALL)
#undef CALL
}

HLF_DEBUG_TAKE(enumerate)

}  // namespace hlf
