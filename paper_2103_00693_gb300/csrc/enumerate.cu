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
//                        to one Gray block, and below that to single indices
//                        (reduce_cut.h).
//   store_kernel         coalesced materialisation by groups of 64 or 32
//                        consecutive solutions a warp step (store_groups): one
//                        XOR per solution, 512 B a step at W = 1; at W > 1 the
//                        lanes' solutions are restaged in shared memory so that
//                        the warp writes its 32*W words with consecutive lanes
//                        on consecutive words. Bound by HBM stores.
//   sample_kernel        z(i) at arbitrary indices, by lookups in seed tables.

#include "enum_impl.cuh"
#include "reduce_cut.h"

namespace hlf {
namespace {

// The reduce of n_chunks windows of `chunk` indices, window c starting at
// offset + c * chunk (hlf_enumerate_reduce is one window). A window is cut into
// `parts` CTAs of blockDim.x threads, each thread walking `per` consecutive
// indices that start at a multiple of 2^U, so that only the window's two ends
// have partial Gray blocks; a window of few blocks (align = 0) is dealt from its own
// start. Items (window, part) are taken grid-stride. With
// one part per window the CTA writes the result unless asked to add; otherwise it
// adds to it, once the kernel that clears the results (clear_results_kernel, which this
// one may start beside) has ended.
template <int W, int U, int T>
__global__ void __launch_bounds__(T, min_ctas_for(W))
    reduce_kernel(const uint64_t* __restrict__ table, uint64_t offset, uint64_t chunk, uint64_t n_chunks,
                  uint32_t parts, uint64_t per, uint64_t runs, uint64_t align, int ntab, bool add,
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
        asm volatile("griddepcontrol.wait;" ::: "memory");
        hlf_reduce& r = out[c];
        if (parts == 1 && !add) {
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

// Results to zero. The reduce that follows is launched as this kernel's dependent and
// fills its tables and walks beside it; only its additions wait. Everything else the
// reduce reads was complete before this kernel began. 2^20 four-word solutions:
// 10.8 us a call, 12.3 with a memset before the reduce.
__global__ void clear_results_kernel(uint64_t* __restrict__ out, uint64_t words)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint64_t step = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < words; i += step) out[i] = 0ull;
}

// ------------------------------------------------ large windows at W = 1
// The reduce of one aligned region [base, base + 2^m) of indices, m >= kRegionMin.
// Its solutions are z(base) ^ span(B_0 .. B_{m-1}) in whatever basis, so the walk may
// choose one. In the L domain every vector has a low and a high 32-bit word, and at
// least m - 32 dimensions of the span have a zero low word. With UH of these as the
// innermost rows, the low word y_lo of 2^UH solutions in a row is the same, and with
// it the low word of the hash's first product and most of the high one:
//     y * M1 = y_lo * M1 + (y_hi * M1_lo << 32),
// so a solution costs one 32-bit multiply-add where the product took a wide and two
// narrow ones; the step XOR is one word; and since the product's low word p is fixed,
// x ^= x >> 27 is a rotation of the high word by 5 and two masked XORs:
//     lo' = (p ^ (p >> 27)) ^ (rot & ~31),  hi' = hi ^ (rot & 31).
// 10 operations of the ALU pipe instead of 12, and 4 multiplies instead of 6.
// 2^35 solutions (a rank-35 grid): 19.1 ms, 23.9 before; in a bare loop over 2^34,
// UH = 4: 9.5 ms, 3: 9.5, 2: 9.8, the plain walk 12.5. Rows with a zero high word
// inside gave 2%; the hash's last shift or its sum on the multiply pipe lost 1-10%.

constexpr int kRegionMin = 33;
static_assert(kRegionMin > 32, "a region's basis has a row of zero low word");

// x = (lo, hi) behind the second shift: the last product and shift, added to hs.
__device__ __forceinline__ void region_tail(uint32_t lo, uint32_t hi, uint64_t& hs)
{
    uint64_t y = (((uint64_t)hi << 32) | lo) * 0x94D049BB133111EBull;
    hs += y ^ (y >> 31);
}

// 2^L solutions whose low words agree: p is the product's low word, kx = p ^ (p >> 27),
// c the part of its high word that y_lo gives.
template <int L, int UH>
__device__ __forceinline__ void region_inner(uint32_t& yh, uint32_t kx, uint32_t c, const uint32_t (&BH)[UH],
                                             uint64_t& hs)
{
    if constexpr (L == 0) {
        const uint32_t h = yh * 0x1CE4E5B9u + c;
        const uint32_t rot = __funnelshift_l(h, h, 5);
        region_tail(kx ^ (rot & ~31u), h ^ (rot & 31u), hs);
    } else {
        region_inner<L - 1, UH>(yh, kx, c, BH, hs);
        yh ^= BH[L - 1];
        region_inner<L - 1, UH>(yh, kx, c, BH, hs);
    }
}

// 2^(L + UH) solutions: the Gray walk over L general rows around the inner blocks.
template <int L, int UH, int UL>
__device__ __forceinline__ void region_block(uint32_t& yl, uint32_t& yh, const uint64_t (&BL)[UL],
                                             const uint32_t (&BH)[UH], uint64_t& hs)
{
    if constexpr (L == 0) {
        const uint64_t p = yl * 0xBF58476D1CE4E5B9ull;
        const uint32_t pl = (uint32_t)p;
        region_inner<UH, UH>(yh, pl ^ (pl >> 27), (uint32_t)(p >> 32), BH, hs);
    } else {
        region_block<L - 1, UH, UL>(yl, yh, BL, BH, hs);
        yl ^= (uint32_t)BL[L - 1];
        yh ^= (uint32_t)(BL[L - 1] >> 32);
        region_block<L - 1, UH, UL>(yl, yh, BL, BH, hs);
    }
}

constexpr int kRegionBlock = 6;  // log2 of the solutions unrolled

// The run [j, j + len) of the region, whole blocks, from z(j) = y.
template <int UH>
__device__ __forceinline__ void region_run(const Table<1>& t, uint64_t j, uint64_t len, uint64_t y, uint64_t& hs)
{
    constexpr int UL = kRegionBlock - UH;
    uint32_t BH[UH];
    uint64_t BL[UL];
#pragma unroll
    for (int k = 0; k < UH; ++k) BH[k] = (uint32_t)(t.B[k][0] >> 32);
#pragma unroll
    for (int k = 0; k < UL; ++k) BL[k] = t.B[UH + k][0];
    uint32_t yl = (uint32_t)y, yh = (uint32_t)(y >> 32);
    const uint64_t end = j + len;
    for (;;) {
        region_block<UL, UH, UL>(yl, yh, BL, BH, hs);
        j += 1ull << kRegionBlock;
        if (j >= end) break;
        const uint64_t r = t.B[ctz64(j)][0];
        yl ^= (uint32_t)r;
        yh ^= (uint32_t)(r >> 32);
    }
}

// Table in the L domain -> the region's: z0 = z(base), rows 0 .. m - 1 a basis of the
// same span with the vectors of zero low word first, the others zero. Returns how
// many those are. One warp reduces the low words as the elimination does (warp
// maxima; lane l has rows l and l + 32): a row that becomes a pivot leaves the rest
// and is a later row of the basis, what is left at the end has zero low words.
__device__ int region_basis(Table<1>& t, uint64_t base, int m, int* s_u)
{
    const int lane = threadIdx.x & 31;
    if (warp_uniform(threadIdx.x >> 5) == 0) {
        const uint64_t g = base ^ (base >> 1);
        const uint64_t seed_part = ((g >> lane) & 1u ? t.B[lane][0] : 0ull) ^
                                   ((g >> (lane + 32)) & 1u ? t.B[lane + 32][0] : 0ull);
        const uint64_t zb = (((uint64_t)__reduce_xor_sync(0xffffffffu, (uint32_t)(seed_part >> 32)) << 32) |
                             __reduce_xor_sync(0xffffffffu, (uint32_t)seed_part)) ^
                            t.z0[0];
        uint64_t r0 = lane < m ? t.B[lane][0] : 0ull, r1 = lane + 32 < m ? t.B[lane + 32][0] : 0ull;
        bool live0 = lane < m, live1 = lane + 32 < m;
        __syncwarp();
        int at = m;  // pivots fill the rows from the end
        for (;;) {
            const uint32_t q = __reduce_max_sync(0xffffffffu, max((uint32_t)r0, (uint32_t)r1));
            if (!q) break;
            // a row whose low word is q: the pivot. Any of them; lane `src`'s first.
            const bool e0 = (uint32_t)r0 == q, e1 = (uint32_t)r1 == q;
            const int src = __ffs(__ballot_sync(0xffffffffu, e0 || e1)) - 1;
            const uint64_t p = __shfl_sync(0xffffffffu, e0 ? r0 : r1, src);
            --at;
            if (lane == src) {
                t.B[at][0] = p;
                if (e0) live0 = false, r0 = 0ull;
                else live1 = false, r1 = 0ull;
            }
            const uint32_t top = 0x80000000u >> __clz(q);
            if ((uint32_t)r0 & top) r0 ^= p;
            if ((uint32_t)r1 & top) r1 ^= p;
        }
        const unsigned m0 = __ballot_sync(0xffffffffu, live0), m1 = __ballot_sync(0xffffffffu, live1);
        const unsigned below = (1u << lane) - 1u;
        if (live0) t.B[__popc(m0 & below)][0] = r0;
        if (live1) t.B[__popc(m0) + __popc(m1 & below)][0] = r1;
        for (int k = m + lane; k < kTableRows; k += 32) t.B[k][0] = 0ull;
        if (lane == 0) {
            t.z0[0] = zb;
            *s_u = at;
        }
    }
    __syncthreads();
    return *s_u;
}

__global__ void __launch_bounds__(1024, 1) reduce_region_kernel(const uint64_t* __restrict__ table, uint64_t base,
                                                                int m, uint64_t per, hlf_reduce* __restrict__ out)
{
    __shared__ Table<1> t;
    __shared__ SeedTable<1> st;
    __shared__ int s_u;
    load_table_hash_domain<1, 2>(t, table);
    __syncthreads();
    const int u = region_basis(t, base, m, &s_u);
    const int ntab = (m + 3) / 4;
    build_seed_table<1>(st, t, ntab);
    __syncthreads();
    const uint64_t size = 1ull << m;
    const uint64_t j = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) * per;
    Acc<1> acc;
    acc.zero();  // the fold of a whole region is zero
    uint64_t cnt = 0;
    if (j < size) {
        cnt = min(per, size - j);
        uint64_t z[1];
        seed_lookup<1>(st, ntab, j, z);
        // u >= m - 32 >= 1: at most 32 of the m rows are pivots on the 32-bit low word
        if (u >= 4) region_run<4>(t, j, cnt, z[0], acc.hs);
        else if (u == 3) region_run<3>(t, j, cnt, z[0], acc.hs);
        else if (u == 2) region_run<2>(t, j, cnt, z[0], acc.hs);
        else region_run<1>(t, j, cnt, z[0], acc.hs);
    }
    block_reduce<1, 1024>(cnt, acc);
    if (threadIdx.x == 0 && cnt) {
        atomicAdd(reinterpret_cast<unsigned long long*>(&out->count), (unsigned long long)cnt);
        atomicAdd(reinterpret_cast<unsigned long long*>(&out->hsum), (unsigned long long)acc.hs);
    }
}

struct StorePlan {
    uint64_t offset, count;
    GroupPlan g;
    uint64_t warps;     // with groups, per_warp each (the last may have fewer)
    uint64_t per_warp;
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

    const uint64_t wg = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    auto row = [&](int k) { return k == kTableZ0Row ? t.z0 : t.B[k]; };
    auto ok = [&](uint64_t i, uint64_t len) { return HLF_RANGE_IN_BOUNDS(i - pl.offset, len, pl.count, kSiteStore); };
    if (wg >= pl.warps) {  // the last warps have the ragged ends
        if (wg - pl.warps < ragged_shares(pl.g)) store_ragged<W>(row, pl.g, pl.offset, wg - pl.warps, out, lane, ok);
        return;
    }
    const uint64_t h0 = pl.g.h_first + wg * pl.per_warp;
    const uint64_t h1 = min(h0 + pl.per_warp, pl.g.h_end);
    uint64_t z[W];
    seed_group<W>(row, h0, lane, z);
    store_groups<W>(z, h0, h1, pl.g.phase, t.B[0][0], out - pl.offset * W,
                    s_stage + (threadIdx.x >> 5) * stage_words<W>(), lane, [&](int j) { return s_C[j]; }, ok);
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

// add: *out is a sum in progress (one window).
template <int W, int U>
hlf_status launch_reduce_u(const uint64_t* table, uint64_t offset, uint64_t chunk, uint64_t n_chunks,
                           hlf_reduce* out, cudaStream_t s, bool add = false)
{
    constexpr int T = reduce_threads(W);
    const ReduceShape sh = reduce_shape(chunk, n_chunks, U, T, (uint64_t)sm_count(), (uint64_t)min_ctas_for(W) * T,
                                        sizeof(Table<W>) + sizeof(SeedTable<W>) + sizeof(uint64_t) * (T / 32) * (2 + W));
    const int ntab = seed_tables_for(offset + (chunk * n_chunks - 1));
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = sh.blocks;
    cfg.blockDim = sh.threads;
    cfg.stream = s;
    cudaLaunchAttribute beside{};
    beside.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    beside.val.programmaticStreamSerializationAllowed = 1;
    if (sh.parts > 1 && !add) {
        static_assert(sizeof(hlf_reduce) % sizeof(uint64_t) == 0, "cleared by words");
        const uint64_t words = sizeof(hlf_reduce) / sizeof(uint64_t) * n_chunks;
        const uint64_t ctas = (words + kThreads - 1) / kThreads, most = (uint64_t)sm_count();
        clear_results_kernel<<<(unsigned)(ctas < most ? ctas : most), kThreads, 0, s>>>(
            reinterpret_cast<uint64_t*>(out), words);
        if (cudaGetLastError() != cudaSuccess) return HLF_ERR_CUDA;
        cfg.attrs = &beside;
        cfg.numAttrs = 1;
    }
    return cudaLaunchKernelEx(&cfg, reduce_kernel<W, U, T>, table, offset, chunk, n_chunks, sh.parts, sh.per, sh.runs,
                              sh.align, ntab, add, out) == cudaSuccess
               ? HLF_OK
               : HLF_ERR_CUDA;
}

// W = 1 has two unrolls: 2^6 solutions per Gray block where every thread of a
// full wave has at least 16 blocks, else 2^3, whose finer cut balances and
// fills the SMs better than the deeper unroll saves.
hlf_status launch_reduce_1(const uint64_t* table, uint64_t offset, uint64_t chunk, uint64_t n_chunks,
                           hlf_reduce* out, cudaStream_t s, bool add)
{
    const uint64_t wave = (uint64_t)sm_count() * min_ctas_for(1) * reduce_threads(1);
    if (chunk * n_chunks < wave * 1024) return launch_reduce_u<1, 3>(table, offset, chunk, n_chunks, out, s, add);
    return launch_reduce_u<1, reduce_unroll(1)>(table, offset, chunk, n_chunks, out, s, add);
}

// One window of at least 2^kRegionMin solutions at W = 1: its aligned regions of that
// size and more, the largest that fit (at most two of each size), and what lies
// before and after them.
hlf_status launch_reduce_regions(const uint64_t* table, uint64_t offset, uint64_t count, hlf_reduce* out,
                                 cudaStream_t s)
{
    if (cudaMemsetAsync(out, 0, sizeof(hlf_reduce), s) != cudaSuccess) return HLF_ERR_CUDA;
    const uint64_t threads = (uint64_t)sm_count() * 1024;
    for (uint64_t a = offset, left = count; left;) {
        int m = 63;
        while (m >= kRegionMin && ((1ull << m) > left || (a & ((1ull << m) - 1)))) --m;
        uint64_t size;
        if (m >= kRegionMin) {
            size = 1ull << m;
            uint64_t per = (size + threads - 1) / threads;
            per = (per + (1ull << kRegionBlock) - 1) & ~((1ull << kRegionBlock) - 1);
            reduce_region_kernel<<<(unsigned)((size + per * 1024 - 1) / (per * 1024)), 1024, 0, s>>>(table, a, m, per,
                                                                                                  out);
            if (cudaGetLastError() != cudaSuccess) return HLF_ERR_CUDA;
        } else {  // up to the next multiple of 2^kRegionMin, or the end
            size = (1ull << kRegionMin) - (a & ((1ull << kRegionMin) - 1));
            if (size > left) size = left;
            const hlf_status st = launch_reduce_1(table, a, size, 1, out, s, true);
            if (st != HLF_OK) return st;
        }
        a += size;
        left -= size;
    }
    return HLF_OK;
}

template <int W>
hlf_status launch_reduce_w(const uint64_t* table, uint64_t offset, uint64_t chunk, uint64_t n_chunks,
                           hlf_reduce* out, cudaStream_t s)
{
    if constexpr (W == 1) {
        if (n_chunks == 1 && chunk >= 1ull << kRegionMin) return launch_reduce_regions(table, offset, chunk, out, s);
        return launch_reduce_1(table, offset, chunk, n_chunks, out, s, false);
    } else {
        return launch_reduce_u<W, reduce_unroll(W)>(table, offset, chunk, n_chunks, out, s);
    }
}

template <int W>
hlf_status launch_store_w(const uint64_t* table, uint64_t offset, uint64_t count, uint64_t* out,
                          cudaStream_t s)
{
    StorePlan pl{};
    pl.offset = offset;
    pl.count = count;
    pl.g = plan_groups(offset, count, Groups<W>::kSize, W == 1 ? store_phase(out, offset) : 0);
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
    pl.per_warp = groups ? (groups + max_warps - 1) / max_warps : 1;
    pl.warps = (groups + pl.per_warp - 1) / pl.per_warp;
    const uint64_t threads = 32 * (pl.warps + ragged_shares(pl.g));
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
