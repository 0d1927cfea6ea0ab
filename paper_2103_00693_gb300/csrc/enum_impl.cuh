// Device helpers of stage 2 (the classical parallel circuit of Section 2,
// Eqs. 1-3, Fig. 1(c)), shared by the single-instance kernels and the batched
// persistent kernel: the shared-memory enumeration table, seeding a run from
// the definition z(i) = z0 ^ XOR_{k in g(i)} B_k, the reflected-Gray walk of a
// run with its reduce, the per-thread reduce accumulator and the block
// reduction.
#pragma once

#include "hlf_internal.cuh"

namespace hlf {

constexpr int kThreads = 256;

// Solutions unrolled per Gray block (2^U) in the per-thread walks: 2^6 at
// W = 1, 2^4 at W = 2, 2^3 at W = 3, 4, and 2^2 beyond, where each solution is
// already 20W - 2 operations and deeper unrolling only costs registers.
// Shape of the single-instance reduce: at W <= 4 one CTA of 1024 threads per
// SM with up to 64 registers each; with the deeper unroll, measured 7-10%
// faster than several 256-thread CTAs with 40-44 registers each.
constexpr int reduce_unroll(int W) { return W == 1 ? 6 : (W == 2 ? 4 : (W <= 4 ? 3 : 2)); }
constexpr int reduce_threads(int W) { return W <= 4 ? 1024 : kThreads; }
constexpr int min_ctas_for(int W) { return W <= 4 ? 1 : 2; }

template <int W>
struct Table {
    uint64_t B[kTableRows][W];  // B_0..B_63, zero rows beyond min(r,64), row 64 zero
    uint64_t z0[W];
};

template <int W>
__device__ __forceinline__ void load_table(Table<W>& t, const uint64_t* __restrict__ g)
{
    uint64_t* d = &t.B[0][0];
    for (int i = threadIdx.x; i < kTableTotalRows * W; i += blockDim.x) d[i] = g[i];
}

// The first layer of the SplitMix64 finalizer, L(x) = x ^ (x >> 30), is
// linear over GF(2), so it commutes with the walk's XORs and with the XOR that
// chains the words: L(z(i+1)) = L(z(i)) ^ L(B_ctz(i+1)) and
// L(h ^ w) = L(h) ^ L(w). The reduce therefore walks y = L(z) on every word, with a
// table whose entries are L(B_k) and L(z0): word 0 skips the layer, and a later
// word joins the layer of the chained hash as the third operand of its XORs.
// Hash values are bit-identical to mix64 over z; the XOR-fold is taken in the L
// domain and mapped back once with L^-1(y) = y ^ (y >> 30) ^ (y >> 60). Two of the
// 16 ALU-pipe operations of a later word go away (cycles a warp of solutions
// costs a scheduler: W = 2 64 -> 60, with the steps below; W = 7 253 -> 227,
// W = 11 452 -> 358; 1024 grids of 1 to 4 words, batched: 2.10 -> 1.97 ms).
__device__ __forceinline__ uint64_t mix_head(uint64_t x) { return x ^ (x >> 30); }
__device__ __forceinline__ uint64_t mix_head_inv(uint64_t y) { return y ^ (y >> 30) ^ (y >> 60); }
__device__ __forceinline__ uint64_t mix_tail(uint64_t y)
{
    y *= 0xBF58476D1CE4E5B9ull;
    y ^= y >> 27;
    y *= 0x94D049BB133111EBull;
    y ^= y >> 31;
    return y;
}

// Table for the reduce: every word of every row (and of z0) taken through L.
// Returns whether this thread saw a row below U with a bit past word 0 (see
// reduce_run_from); the callers OR it over the CTA while they synchronise.
template <int W, int U>
__device__ __forceinline__ bool load_table_hash_domain(Table<W>& t, const uint64_t* __restrict__ g)
{
    uint64_t* d = &t.B[0][0];
    bool mixed = false;
    for (int i = threadIdx.x; i < kTableTotalRows * W; i += blockDim.x) {
        const uint64_t v = __ldcg(g + i);
        d[i] = mix_head(v);
        mixed |= i < U * W && i % W != 0 && v != 0ull;
    }
    return mixed;
}

// 64-bit shifts with PTX semantics: amounts of 64 give 0.
__device__ __forceinline__ uint64_t shl64(uint64_t x, uint32_t s)
{
    uint64_t r;
    asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
    return r;
}
__device__ __forceinline__ uint64_t shr64(uint64_t x, uint32_t s)
{
    uint64_t r;
    asm("shr.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
    return r;
}
template <int W>
__device__ __forceinline__ void xor_row(uint64_t (&z)[W], const uint64_t* __restrict__ b)
{
#pragma unroll
    for (int w = 0; w < W; ++w) z[w] ^= b[w];
}

// z(i) from its definition (seed of a run).
template <int W>
__device__ __forceinline__ void seed(const Table<W>& t, uint64_t i, uint64_t (&z)[W])
{
    uint64_t g = i ^ (i >> 1);
#pragma unroll
    for (int w = 0; w < W; ++w) z[w] = t.z0[w];
    while (g) {
        const int k = __ffsll((long long)g) - 1;
        g &= g - 1;
        xor_row<W>(z, t.B[k]);
    }
}

// Seeds by table lookup. z(i) is linear in the bits of g(i), so 16 tables of
// the combinations of four rows each give it in one lookup and one row XOR per
// four bits, where seed() walks the set bits one by one (a chain of about 30
// dependent shared-memory reads for a 60-bit index). z0 is folded into the
// first table. An entry of one word per table: the 16 entries of a table lie in
// 16 distinct bank pairs, so lanes with different indices read without
// conflicts.
constexpr int kSeedTables = 16;

template <int W>
struct SeedTable {
    uint64_t t[W][kSeedTables][16];
};

// Tables covering the index bits that [0, last] uses.
__host__ __device__ inline int seed_tables_for(uint64_t last)
{
#ifdef __CUDA_ARCH__
    const int bits = 64 - __clzll((long long)(last | 1));
#else
    const int bits = 64 - __builtin_clzll(last | 1);
#endif
    return (bits + 3) / 4;
}

// Built by the whole CTA from a loaded table; the caller synchronises after.
template <int W>
__device__ __forceinline__ void build_seed_table(SeedTable<W>& st, const Table<W>& t, int ntab)
{
    for (int e = threadIdx.x; e < W * ntab * 16; e += blockDim.x) {
        const int x = e & 15;
        const int q = (e >> 4) % ntab;
        const int w = (e >> 4) / ntab;
        uint64_t v = q == 0 ? t.z0[w] : 0ull;
#pragma unroll
        for (int b = 0; b < 4; ++b)
            if ((x >> b) & 1) v ^= t.B[4 * q + b][w];
        st.t[w][q][x] = v;
    }
}

template <int W>
__device__ __forceinline__ void seed_lookup(const SeedTable<W>& st, int ntab, uint64_t i, uint64_t (&z)[W])
{
    uint64_t g = i ^ (i >> 1);
#pragma unroll
    for (int w = 0; w < W; ++w) z[w] = st.t[w][0][g & 15];
    for (int q = 1; q < ntab; ++q) {
        g >>= 4;
#pragma unroll
        for (int w = 0; w < W; ++w) z[w] ^= st.t[w][q][g & 15];
    }
}

// Per-thread accumulator of the reduce, fed with solutions in the L domain (see
// load_table_hash_domain): sum of hashes and XOR-fold.
template <int W>
struct Acc {
    uint64_t hs;
    uint64_t fold[W];
    __device__ __forceinline__ void zero()
    {
        hs = 0;
#pragma unroll
        for (int w = 0; w < W; ++w) fold[w] = 0;
    }
    // The hash alone: for the solutions of whole aligned Gray blocks, whose
    // XOR is zero (see reduce_run_from).
    __device__ __forceinline__ void consume_hash(const uint64_t (&z)[W])
    {
        uint64_t h = mix_tail(z[0]);  // = mix64 of the solution's word 0
#pragma unroll
        for (int w = 1; w < W; ++w) h = mix_tail(mix_head(h) ^ z[w]);
        hs += h;
    }
    __device__ __forceinline__ void consume(const uint64_t (&z)[W])
    {
        consume_hash(z);
#pragma unroll
        for (int w = 0; w < W; ++w) fold[w] ^= z[w];
    }
    // XOR-fold back in the solution domain (after all XOR reductions).
    __device__ __forceinline__ uint64_t fold_word(int w) const { return mix_head_inv(fold[w]); }
};

// The accumulator seen by whole aligned Gray blocks: hash only.
template <int W>
struct HashOnly {
    Acc<W>& acc;
    __device__ __forceinline__ void consume(const uint64_t (&z)[W]) { acc.consume_hash(z); }
};

// 2^L consecutive solutions starting at an index that is a multiple of 2^L:
// the reflected Gray code is (first half, flip bit L-1, second half), so the
// step between the halves is row L-1, at a compile-time index. `Rows` holds the
// first NW words of each row: a register array where that is one word, else the
// shared-memory table (register copies of U rows of W words would cost more
// occupancy than they save). `Sink` consumes each solution.
template <int W, int L, int NW, typename Rows, typename Sink>
struct GrayBlock {
    static __device__ __forceinline__ void run(uint64_t (&z)[W], const Rows& Br, Sink& sink)
    {
        GrayBlock<W, L - 1, NW, Rows, Sink>::run(z, Br, sink);
#pragma unroll
        for (int w = 0; w < NW; ++w) z[w] ^= Br[L - 1][w];
        GrayBlock<W, L - 1, NW, Rows, Sink>::run(z, Br, sink);
    }
};
template <int W, int NW, typename Rows, typename Sink>
struct GrayBlock<W, 0, NW, Rows, Sink> {
    static __device__ __forceinline__ void run(uint64_t (&z)[W], const Rows&, Sink& sink) { sink.consume(z); }
};

// The reduce of [i, i + len), len >= 1, with z = z(i) in the L domain.
// The solutions of an aligned block of 2^U consecutive indices (U >= 2) are
// z_s ^ XOR_{k in S} B_k over all subsets S of {0..U-1}: z_s and every B_k occur
// an even number of times, so their XOR is zero (in the L domain too, L being
// linear). Whole blocks therefore feed only the hash; the head and the tail of
// the run (partial blocks) feed hash and fold. The fold is exact, and one 64-bit
// XOR per solution lighter.
//
// `mixed`: some row below U has bits past word 0. Reduced rows are zero outside
// their pivot and the free columns, so on grids, whose dependencies are local,
// the first rows usually have none; the steps inside a block then touch word 0
// only, held in registers.
template <int W, int U>
__device__ __forceinline__ void reduce_run_from(const Table<W>& t, bool mixed, uint64_t i, uint64_t len,
                                                uint64_t (&z)[W], Acc<W>& acc)
{
    static_assert(U >= 2, "a block of 2^U solutions XORs to zero only for U >= 2");
    constexpr uint64_t kBlk = 1ull << U;
    while (len && (i & (kBlk - 1))) {  // head up to a multiple of 2^U
        acc.consume(z);
        --len;
        ++i;
        if (len) xor_row<W>(z, t.B[ctz64(i)]);
    }
    if (len >= kBlk) {
        HashOnly<W> ho{acc};
        if (W == 1 || !mixed) {
            uint64_t Br[U][1];
#pragma unroll
            for (int k = 0; k < U; ++k) Br[k][0] = t.B[k][0];
            do {
                GrayBlock<W, U, 1, uint64_t[U][1], HashOnly<W>>::run(z, Br, ho);
                len -= kBlk;
                i += kBlk;
                if (len) xor_row<W>(z, t.B[ctz64(i)]);  // ctz(i) >= U here
            } while (len >= kBlk);
        } else {
            do {
                GrayBlock<W, U, W, uint64_t[kTableRows][W], HashOnly<W>>::run(z, t.B, ho);
                len -= kBlk;
                i += kBlk;
                if (len) xor_row<W>(z, t.B[ctz64(i)]);
            } while (len >= kBlk);
        }
    }
    while (len) {  // tail
        acc.consume(z);
        --len;
        ++i;
        if (len) xor_row<W>(z, t.B[ctz64(i)]);
    }
}

// Table in the L domain -> the table of an aligned region [base, base + 2^m) of
// indices, 0 < m <= 32, whose solutions are z(base) ^ span(B_0 .. B_{m-1}) in any
// basis: z0 = z(base), rows 0 .. m - 1 a basis with the vectors of zero words past
// word 0 first. Returns how many those are. The region's index counts from base.
// One warp reduces the later words, lane l holding row l: a warp maximum names a
// pivot, which leaves the rest and becomes a later row of the basis; what is left at
// the end has word 0 only. Called by the whole CTA.
template <int W>
__device__ int low_basis(Table<W>& t, uint64_t base, int m, int* s_low)
{
    const int lane = threadIdx.x & 31;
    if (warp_uniform(threadIdx.x >> 5) == 0) {
        const uint64_t g = base ^ (base >> 1);
        const bool lo = (g >> lane) & 1u, hi = (g >> (lane + 32)) & 1u;
        uint64_t r[W];
#pragma unroll
        for (int w = 0; w < W; ++w) {
            const uint64_t a = (lo ? t.B[lane][w] : 0ull) ^ (hi ? t.B[lane + 32][w] : 0ull);
            const uint32_t al = __reduce_xor_sync(0xffffffffu, (uint32_t)a);
            const uint32_t ah = __reduce_xor_sync(0xffffffffu, (uint32_t)(a >> 32));
            if (lane == 0) t.z0[w] ^= ((uint64_t)ah << 32) | al;
            r[w] = lane < m ? t.B[lane][w] : 0ull;
        }
        bool live = lane < m;
        __syncwarp();
        int at = m;  // pivots fill the rows from the end
#pragma unroll
        for (int w = 1; w < W; ++w) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                for (;;) {
                    const uint32_t v = (uint32_t)(r[w] >> (32 * h));
                    const uint32_t q = __reduce_max_sync(0xffffffffu, v);
                    if (!q) break;
                    const int src = __ffs(__ballot_sync(0xffffffffu, v == q)) - 1;
                    const bool has = v & (0x80000000u >> __clz(q));
                    --at;
#pragma unroll
                    for (int x = 0; x < W; ++x) {
                        const uint64_t p = __shfl_sync(0xffffffffu, r[x], src);
                        if (lane == src) t.B[at][x] = p;
                        r[x] ^= has ? p : 0ull;  // the pivot's own row becomes zero
                    }
                    if (lane == src) live = false;
                }
            }
        }
        const unsigned mask = __ballot_sync(0xffffffffu, live);
        if (live) {
            const int k = __popc(mask & ((1u << lane) - 1u));
#pragma unroll
            for (int x = 0; x < W; ++x) t.B[k][x] = x ? 0ull : r[0];
        }
        if (lane == 0) *s_low = at;
    }
    __syncthreads();
    return *s_low;
}

// Block-wide (count, hsum, fold) reduction over a CTA of THREADS threads;
// the result is valid in thread 0.
template <int W, int THREADS = kThreads>
__device__ __forceinline__ void block_reduce(uint64_t& cnt, Acc<W>& acc)
{
    static_assert(THREADS % 32 == 0 && THREADS <= 1024, "one partial per warp, reduced by one warp");
    __shared__ uint64_t s_part[THREADS / 32][2 + W];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
        acc.hs += __shfl_xor_sync(0xffffffffu, acc.hs, o);
#pragma unroll
        for (int w = 0; w < W; ++w) acc.fold[w] ^= __shfl_xor_sync(0xffffffffu, acc.fold[w], o);
    }
    if (lane == 0) {
        s_part[warp][0] = cnt;
        s_part[warp][1] = acc.hs;
#pragma unroll
        for (int w = 0; w < W; ++w) s_part[warp][2 + w] = acc.fold[w];
    }
    __syncthreads();
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
        cnt = lane < nw ? s_part[lane][0] : 0;
        acc.hs = lane < nw ? s_part[lane][1] : 0;
#pragma unroll
        for (int w = 0; w < W; ++w) acc.fold[w] = lane < nw ? s_part[lane][2 + w] : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
            acc.hs += __shfl_xor_sync(0xffffffffu, acc.hs, o);
#pragma unroll
            for (int w = 0; w < W; ++w) acc.fold[w] ^= __shfl_xor_sync(0xffffffffu, acc.fold[w], o);
        }
    }
    __syncthreads();  // s_part may be reused by the caller
}

// Streaming (evict-first) global stores: the solutions are written once and
// not read back by this kernel.

__device__ __forceinline__ void st_cs_v2(uint64_t* p, uint64_t a, uint64_t b)
{
    asm volatile("st.global.cs.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ void st_cs(uint64_t* p, uint64_t a)
{
    asm volatile("st.global.cs.u64 [%0], %1;" ::"l"(p), "l"(a) : "memory");
}

// 32 consecutive solutions of W > 1 words, one per lane (lane l holds the
// solution whose W words start at dst + l*W), written out coalesced: each lane
// stages its words in shared memory with an odd row stride (W | 1, so the
// lane-strided writes of one word index fall in distinct banks), then
// consecutive lanes store consecutive words of the 32*W-word block. `stage`
// holds 32*(W|1) words for this warp. With W even, dst must be 16-byte
// aligned and each lane stores word pairs.
template <int W>
constexpr int stage_words()
{
    return 32 * (W | 1);
}

template <int W, bool Pairs>
__device__ __forceinline__ void store_warp_coalesced(uint64_t* dst, const uint64_t (&z)[W], uint64_t* stage,
                                                     int lane)
{
    static_assert(W > 1, "W = 1 stores pairs of solutions straight from registers");
    constexpr int SW = W | 1;
#pragma unroll
    for (int w = 0; w < W; ++w) stage[lane * SW + w] = z[w];
    __syncwarp();
    if constexpr (Pairs && W % 2 == 0) {
#pragma unroll 4
        for (int k = 0; k < W / 2; ++k) {
            const int q = 2 * (lane + 32 * k);  // even, so q % W is even and q, q + 1 share a row
            const int l = q / W, w = q - l * W;
            st_cs_v2(dst + q, stage[l * SW + w], stage[l * SW + w + 1]);
        }
    } else {
#pragma unroll 4
        for (int k = 0; k < W; ++k) {
            const int q = lane + 32 * k;
            const int l = q / W, w = q - l * W;
            st_cs(dst + q, stage[l * SW + w]);
        }
    }
    __syncwarp();  // the stage is rewritten by the next call
}

// ------------------------------------------------------- storing by groups
// A window is stored in groups of G consecutive solutions, one group a warp step:
// G = 64 at W = 1 (a lane holds the pair z, z ^ B_0), 32 beyond. With m = log2 G,
// g(G h + t) = (g(h) << m) ^ ((h & 1) << (m - 1)) ^ g(t), so stepping h -> h + 1
// XORs the same row C_j = B_{m-1} ^ B_{m+j}, j = ctz(h + 1), into every lane.

template <int W>
struct Groups {
    static constexpr int kPerLane = W == 1 ? 2 : 1;
    static constexpr int kLog2 = W == 1 ? 6 : 5;
    static constexpr uint64_t kSize = 32 * kPerLane;
};

// Groups [h_first, h_end) of the window [offset, offset + count), group h being the
// indices G h + phase .. G h + phase + G - 1, and the indices before and after them.
struct GroupPlan {
    uint64_t n_head;      // [offset, offset + n_head)
    uint64_t tail_first;  // [tail_first, tail_first + n_tail)
    uint64_t n_tail;
    uint64_t h_first, h_end;
    uint32_t phase;
};

// phase < 4 (W = 1): where the groups start, such that they lie on 32 bytes whatever
// the window's offset: lane l then stores z(G h + 2 l + phase) and the one after it,
// which are its own or its neighbours'. 2^27 solutions take 171 us at every offset; with
// groups at multiples of G they took 190 at offsets 2 mod 4 (a sector in two pieces
// at each end of a step) and 234-246 at odd ones (8-byte stores). The window may end at
// 2^64 exactly, which wraps to 0.
inline uint32_t store_phase(const uint64_t* out, uint64_t offset)
{
    return (uint32_t)(offset - (reinterpret_cast<uintptr_t>(out) >> 3)) & 3;
}
inline GroupPlan plan_groups(uint64_t offset, uint64_t count, uint64_t G, uint32_t phase)
{
    GroupPlan pl{};
    pl.phase = phase;
    const uint64_t end = offset + count;  // 0 for 2^64
    const bool wraps = count != 0 && end == 0;
    // first group at or after offset, and one past the last that ends by `end`
    const uint64_t h_first = offset <= phase ? 0 : (offset - phase - 1) / G + 1;
    const uint64_t h_end = wraps && !phase ? (0ull - G) / G + 1 : (end < phase && !wraps ? 0 : (end - phase) / G);
    if (h_end <= h_first) {
        pl.n_head = count;
        return pl;
    }
    pl.h_first = h_first;
    pl.h_end = h_end;
    pl.n_head = h_first * G + phase - offset;
    pl.tail_first = h_end * G + phase;  // wraps to 0 only when the tail is empty
    pl.n_tail = count - pl.n_head - (h_end - h_first) * G;
    return pl;
}

// z(G h + kPerLane * lane) for the 32 lanes of a warp. `row(k)` points to the W words
// of B_k, z0 at row(kTableZ0Row). The part all lanes share is one XOR over the
// warp, lane l bringing rows l and l + 32; the lane's own part has at most m rows.
template <int W, typename Row>
__device__ __forceinline__ void seed_group(Row row, uint64_t h, int lane, uint64_t (&z)[W])
{
    constexpr int M = Groups<W>::kLog2;
    const uint64_t g = ((h ^ (h >> 1)) << M) ^ ((h & 1) << (M - 1));
    const bool lo = (g >> lane) & 1u, hi = (g >> (lane + 32)) & 1u;
#pragma unroll
    for (int w = 0; w < W; ++w) {
        const uint64_t a = (lo ? row(lane)[w] : 0ull) ^ (hi ? row(lane + 32)[w] : 0ull);
        z[w] = ((uint64_t)__reduce_xor_sync(0xffffffffu, (uint32_t)(a >> 32)) << 32) |
               __reduce_xor_sync(0xffffffffu, (uint32_t)a);
        z[w] ^= row(kTableZ0Row)[w];
    }
    const int t = Groups<W>::kPerLane * lane;
    const int gt = t ^ (t >> 1);
#pragma unroll
    for (int k = 0; k < M; ++k) {
        const bool in = (gt >> k) & 1;
#pragma unroll
        for (int w = 0; w < W; ++w) z[w] ^= in ? row(k)[w] : 0ull;
    }
}

// z(i) for lanes whose indices lie in [base, base + 64), base the same in all of them:
// i >> 6 is one of two consecutive values, so all but the last six rows and the step
// between the two are shared (as in seed_group).
template <int W, typename Row>
__device__ __forceinline__ void seed_near(Row row, uint64_t base, uint64_t i, int lane, uint64_t (&z)[W])
{
    const uint64_t H = base >> 6;
    const uint64_t g = ((H ^ (H >> 1)) << 6) ^ ((H & 1) << 5);
    const bool lo = (g >> lane) & 1u, hi = (g >> (lane + 32)) & 1u;
    const bool next = (i >> 6) != H;
    const int gt = (int)(i & 63) ^ ((int)(i & 63) >> 1);
    const int j = ctz64(H + 1);  // at most 58
#pragma unroll
    for (int w = 0; w < W; ++w) {
        const uint64_t a = (lo ? row(lane)[w] : 0ull) ^ (hi ? row(lane + 32)[w] : 0ull);
        z[w] = ((uint64_t)__reduce_xor_sync(0xffffffffu, (uint32_t)(a >> 32)) << 32) |
               __reduce_xor_sync(0xffffffffu, (uint32_t)a);
        z[w] ^= row(kTableZ0Row)[w] ^ (next ? row(5)[w] ^ row(6 + j)[w] : 0ull);
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const bool in = (gt >> k) & 1;
#pragma unroll
        for (int w = 0; w < W; ++w) z[w] ^= in ? row(k)[w] : 0ull;
    }
}

// The ragged ends of a window, 32 indices a warp: share `u` of ragged_shares(g).
__host__ __device__ inline uint64_t ragged_shares(const GroupPlan& g)
{
    return (g.n_head + 31) / 32 + (g.n_tail + 31) / 32;
}
template <int W, typename Row, typename Check>
__device__ __forceinline__ void store_ragged(Row row, const GroupPlan& g, uint64_t offset, uint64_t u, uint64_t* out,
                                             int lane, Check ok)
{
    const uint64_t heads = (g.n_head + 31) / 32;
    const bool head = u < heads;
    const uint64_t at = 32 * (head ? u : u - heads);
    const uint64_t left = (head ? g.n_head : g.n_tail) - at;
    const uint64_t base = (head ? offset : g.tail_first) + at;
    const uint64_t i = base + lane;
    uint64_t z[W];
    seed_near<W>(row, base, i, lane, z);
    if (lane < left && ok(i, 1)) {
#pragma unroll
        for (int w = 0; w < W; ++w) out[(i - offset) * W + w] = z[w];
    }
}

// Groups [h, h1) of a window, h < h1, by one warp from the lanes' seeds: `dst` is the
// output less offset * W words, `step(j)` points to C_j, `b0` is B_0's word (W = 1),
// `stage` holds stage_words<W>() words of the warp (W > 1, where phase is 0 and dst lies
// on 16 bytes).
template <int W, typename Step, typename Check>
__device__ __forceinline__ void store_groups(uint64_t (&z)[W], uint64_t h, uint64_t h1, uint32_t phase, uint64_t b0,
                                             uint64_t* dst, uint64_t* stage, int lane, Step step, Check ok)
{
    constexpr uint64_t G = Groups<W>::kSize;
    if constexpr (W == 1) {
        for (;;) {
            const uint64_t z1 = z[0] ^ b0;  // g(2t + 1) = g(2t) ^ 1
            const uint64_t zn = z[0] ^ step(ctz64(h + 1))[0];
            const uint64_t i = h * G + 2 * lane + phase;
            uint64_t a = z[0], b = z1;
            if (phase) {  // warp-uniform; the last lanes' neighbours are in the next group
                const uint64_t next = __shfl_sync(0xffffffffu, lane == 0 ? zn : z[0], (lane + 1) & 31);
                if (phase == 1) {
                    a = z1;
                    b = next;
                } else if (phase == 2) {
                    a = next;
                    b = next ^ b0;
                } else {
                    a = next ^ b0;
                    b = __shfl_sync(0xffffffffu, lane < 2 ? zn : z[0], (lane + 2) & 31);
                }
            }
            if (ok(i, 2)) st_cs_v2(dst + i, a, b);
            if (++h == h1) break;
            z[0] = zn;
        }
    } else {
        for (;;) {
            if (ok(h * G, G))  // warp-uniform
                store_warp_coalesced<W, true>(dst + h * G * W, z, stage, lane);
            if (++h == h1) break;
            xor_row<W>(z, step(ctz64(h)));
        }
    }
}

}  // namespace hlf
