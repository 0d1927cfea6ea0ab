// Stage 1 of the two-stage scheme as block-level device functions: the CLA
// module of Section 2 (Fig. 1(b)), steps (1)-(4), for one matrix per CTA.
//
//   (1) Gauss-Jordan elimination of A over GF(2). The reduced row echelon form
//       is unique, so any row with the column's bit may be the pivot; nothing
//       asks for the lowest one, and no exchange across the CTA is needed per
//       column: one warp finds the pivots alone.
//       W = 1 (eliminate_warp): the warp holds whole rows, two a lane, and
//       the pivot row of column c moves to position c. A pivot is one warp
//       maximum of the remaining words, with the columns from the top bit down.
//       W > 1 (eliminate_panels): panels of 32 columns. One warp, which owns no
//       rows, eliminates the 32-bit slices of the live rows (unused, slice not
//       zero); the row warps then apply what it found to whole rows. See there.
//   (2)-(4) Kernel basis, q and z^a. For a free column f the kernel vector is
//       x_f = e_f + sum_k B_k[f] e_{p_k}; q(x_f) = sum over i in supp(x_f) of
//       popcount(A_i & x_f), mod 4, which is x_f^T A x_f mod 4. With z^a
//       chosen to vanish on the pivots, z^a . x_f = z^a_f, so the equation
//       2 z^T x_f = q(x_f) (mod 4) gives z^a_f = q(x_f) / 2 directly. Bit p of
//       x_f is bit f of the row whose pivot is p, so 32 bits of x_f are one
//       ballot over 32 positions.
//
// Also checked here: padding bits (column >= n) are zero and A is symmetric
// (Section 1 defines the problem for symmetric A only), the latter by 64 x 64
// bit-block transposes in registers.
#pragma once

#include "hlf_internal.cuh"

namespace hlf {

// Transpose a 64 x 64 bit block held by one warp: lane l has rows l (x0) and
// l + 32 (x1), bit s of a row being column s. Stage j (j = 32, 16, ..., 1)
// swaps the row-index bit of weight j with the column-index bit of weight j:
// it exchanges the bits at column s + j of row t with those at column s of
// row t + j, for s and t with that bit clear. The six stages compose to the
// transpose. Stage 32 pairs the two rows of a lane, the others pair lanes l
// and l ^ j.
__device__ __forceinline__ void transpose64_warp(uint64_t& x0, uint64_t& x1, int lane)
{
    {
        const uint64_t t = ((x0 >> 32) ^ x1) & 0x00000000FFFFFFFFull;
        x1 ^= t;
        x0 ^= t << 32;
    }
#pragma unroll
    for (int j = 16; j >= 1; j >>= 1) {
        const uint64_t m = j == 16 ? 0x0000FFFF0000FFFFull
                         : j == 8  ? 0x00FF00FF00FF00FFull
                         : j == 4  ? 0x0F0F0F0F0F0F0F0Full
                         : j == 2  ? 0x3333333333333333ull
                                   : 0x5555555555555555ull;
        const bool upper = (lane & j) != 0;  // this lane's rows are the t + j of their pairs
        const uint64_t o0 = __shfl_xor_sync(0xffffffffu, x0, j);
        const uint64_t o1 = __shfl_xor_sync(0xffffffffu, x1, j);
        const uint64_t t0 = upper ? (((o0 >> j) ^ x0) & m) : (((x0 >> j) ^ o0) & m);
        const uint64_t t1 = upper ? (((o1 >> j) ^ x1) & m) : (((x1 >> j) ^ o1) & m);
        x0 ^= upper ? t0 : t0 << j;
        x1 ^= upper ? t1 : t1 << j;
    }
}

// ------------------------------------------------------------ elimination

constexpr int kPanelCap = 128;  // slices the searching warp takes at most (4 a lane)

// Slices a search takes when nl rows are live. Beyond the most that fit, 64: rows
// as many as that nearly always span the panel, and a shorter column costs less;
// where they do not, the panel is searched again for what the others still hold.
__device__ __forceinline__ int panel_cap(int nl)
{
    return nl <= 32 ? 32 : (nl <= 64 || nl > kPanelCap ? 64 : kPanelCap);
}

// Whether no row can hold further pivots of the panel: none was live, all that
// were have been searched, or every column has its pivot. (A live slice has a
// bit, so a search of any finds at least one pivot and this ends.)
__device__ __forceinline__ bool panel_done(int nl, uint32_t cols, int ncols)
{
    return cols == 0u || nl <= panel_cap(nl) || __popc(cols) == ncols;
}

// Shared memory of a factorisation of up to MAXN rows of W words. The arrays
// sized by n follow it: rows [W][stride] (word-major: a warp's rows are
// consecutive; the stride is odd, so the words of one row lie in distinct banks
// too) and T2 [8][W][16] (W > 1), and for factor_block a copy of A like rows.
template <int W, int MAXN>
struct FactorSmem {
    uint32_t list[kPanelCap];    // slices of the live rows
    int16_t listrow[kPanelCap];  // and the rows
    int16_t kres[kPanelCap];     // the column each searched slice became the pivot of, or -1
    __align__(8) int16_t prow[2][32];  // the pivot row of column b, -1 if free, by round parity
    int nlist[2];              // live rows, by round parity
    int nactive;               // rows that absorb pivots of the last panel
    uint32_t cols;             // the search's pivot columns
    __align__(16) uint32_t Hcol[32];  // reduced pivot row of column b as a set of pivot start rows, 0 if free
    uint32_t T1[8 * 16];       // XORs of Hcol over 4 columns
    int err;
    int rank;
    uint64_t z0[W];
    uint32_t pivmask[MAXN / 32];  // the pivot columns, one bit each
    int before[MAXN / 32];        // pivots in the mask words before
    uint2 active[MAXN];           // (row, coefficient set)
    int16_t rowof[MAXN];          // the row whose pivot is column c, -1 if c is free
    int16_t pivcol[MAXN];         // p_k
    int16_t rowk[MAXN];           // the row that holds B_k
};

template <int W>
__host__ __device__ constexpr int row_stride(int n) { return W == 1 ? 64 : (n | 1); }

template <int W, int MAXN>
__host__ __device__ constexpr size_t factor_smem_bytes(int n, bool with_copy)
{
    return (sizeof(FactorSmem<W, MAXN>) + 15) / 16 * 16 +
           sizeof(uint64_t) * W * ((size_t)row_stride<W>(n) * (with_copy ? 2 : 1) + (W > 1 ? 8 * 16 : 0));
}

template <int W, int MAXN>
__device__ __forceinline__ uint64_t* factor_rows(unsigned char* smem)
{
    return reinterpret_cast<uint64_t*>(smem + (sizeof(FactorSmem<W, MAXN>) + 15) / 16 * 16);
}

// The warps of an elimination (W > 1). An SM's four schedulers take a CTA's warps
// by their number mod 4. The searching warp is a serial chain of instructions, so
// it has a scheduler to itself: it is warp 3, the row warps are those whose number
// is not 3 mod 4, and the others stand idle until the elimination is done. Next to
// row warps on its scheduler the searches took a fifth longer (n = 1024: 181k cycles
// in all against 147k). A CTA of fewer than four warps has its last warp search.
__host__ __device__ constexpr int search_warp(int nwarps) { return nwarps >= 4 ? 3 : nwarps - 1; }
__host__ __device__ constexpr int row_warps(int nwarps) { return nwarps >= 4 ? nwarps - nwarps / 4 : nwarps - 1; }
// The threads of a CTA with at least `want` row threads.
__host__ __device__ constexpr int elim_threads(int want)
{
    const int rw = (want + 31) / 32;
    const int last = rw - 1 + (rw - 1) / 3;  // the last row warp's number
    return 32 * (last + 1 < 4 ? 4 : last + 1);
}

// A barrier of the row warps and the searching warp, reached from different code.
__device__ __forceinline__ void bar_elim(int rt)
{
    __syncwarp();
    asm volatile("bar.sync 1, %0;" ::"r"(rt + 32) : "memory");
}

// W = 1: one warp, the CTA's first, eliminates the whole matrix. Lane
// l's candidates are rows l and l + 32, columns 0..31 and 32..63 in a word each,
// bit-reversed so that the leftmost column is the top bit. The largest left word
// of all candidates has the column's bit if any has, so one warp maximum both
// tells whether the column has a pivot and broadcasts the pivot row's word; the
// right word is a second maximum over the rows that share the left one (any of
// them may be the pivot). The pivot row XORs itself to zero where it was and
// lives on at its column's position (lane c & 31), where later pivots clear their
// columns. No step branches: without a pivot no candidate has the bit.
template <int MAXN>
__device__ void eliminate_warp(const uint64_t* __restrict__ A, int n, unsigned char* smem, uint64_t* copy)
{
    using Smem = FactorSmem<1, MAXN>;
    Smem& sm = *reinterpret_cast<Smem*>(smem);
    uint64_t* s_rows = factor_rows<1, MAXN>(smem);  // by pivot column
    const int lane = threadIdx.x;
    uint64_t a0 = lane < n ? A[lane] : 0ull;
    uint64_t a1 = lane + 32 < n ? A[lane + 32] : 0ull;
    copy[lane] = a0;
    copy[lane + 32] = a1;
    a0 = __brevll(a0);
    a1 = __brevll(a1);
    uint32_t r0a = (uint32_t)(a0 >> 32), r0b = (uint32_t)a0, r1a = (uint32_t)(a1 >> 32), r1b = (uint32_t)a1;
    uint32_t z0a = 0, z0b = 0, z1b = 0;  // positions lane and lane + 32 (whose left words stay zero)
    uint32_t q = __reduce_max_sync(0xffffffffu, max(r0a, r1a));
#pragma unroll
    for (int c = 0; c < 32; ++c) {
        if (c % 8 == 0 && !q) break;
        const uint32_t L = 0x80000000u >> c;
        const bool piv = q & L;
        const uint32_t qb =
            __reduce_max_sync(0xffffffffu, max(r0a == q ? r0b : 0u, r1a == q ? r1b : 0u));
        const uint32_t qa = q;
        const bool h0 = r0a & L, h1 = r1a & L, hz = piv && (z0a & L);
        r0a ^= h0 ? qa : 0u;
        r1a ^= h1 ? qa : 0u;
        q = __reduce_max_sync(0xffffffffu, max(r0a, r1a));
        r0b ^= h0 ? qb : 0u;
        r1b ^= h1 ? qb : 0u;
        z0a ^= hz ? qa : 0u;
        z0b ^= hz ? qb : 0u;
        if (piv && lane == c) {
            z0a = qa;
            z0b = qb;
        }
    }
    q = __reduce_max_sync(0xffffffffu, max(r0b, r1b));
#pragma unroll
    for (int c = 0; c < 32; ++c) {
        if (c % 8 == 0 && !q) break;
        const uint32_t L = 0x80000000u >> c;
        const bool piv = q & L;
        const uint32_t qb = q;
        r0b ^= r0b & L ? qb : 0u;
        r1b ^= r1b & L ? qb : 0u;
        q = __reduce_max_sync(0xffffffffu, max(r0b, r1b));
        z0b ^= piv && (z0b & L) ? qb : 0u;
        z1b ^= piv && (z1b & L) ? qb : 0u;
        if (piv && lane == c) z1b = qb;
    }
    s_rows[lane] = __brevll(((uint64_t)z0a << 32) | z0b);
    s_rows[lane + 32] = __brevll((uint64_t)z1b);
    const unsigned m0 = __ballot_sync(0xffffffffu, z0a != 0u), m1 = __ballot_sync(0xffffffffu, z1b != 0u);
    if (lane == 0) {
        sm.pivmask[0] = m0;
        sm.pivmask[1] = m1;
    }
    sm.rowof[lane] = z0a ? (int16_t)lane : (int16_t)-1;
    sm.rowof[lane + 32] = z1b ? (int16_t)(lane + 32) : (int16_t)-1;
}

// One panel's search by one warp: Gauss-Jordan on up to 32 * NS slices of the
// list, bit-reversed so that the leftmost column is the top bit. As in
// eliminate_warp a warp maximum finds whether the column has a pivot and its
// slice at once, and no step branches. Each slice keeps the set (record) of
// pivots it absorbed, a pivot being named by its column: the pivot of column b
// publishes its record with bit b added. Of the slices equal to the maximum, the
// one with the largest record is the pivot (a second maximum, in flight together
// with the next column's first); of several equal in both any may be, and the
// one whose row ends up in prow is. The pivot's slice and set move to the pivot
// slot of lane b, where later pivots clear their columns; the set ends as H_b.
// A column takes 60, 77 or 109 cycles with 1, 2 or 4 slices a lane; with a ballot, a
// find-first and shuffles instead of the maxima it took 200. Two halves of 16 columns
// with slice and record in one word, one maximum a column, were slower (68, 91, 138):
// the maximum's result is held in a uniform register, and what is formed from it
// before it meets the slices lengthens the chain; joining the halves costs the rest.
//
// The loop runs eight columns per turn with the slices shifted up by eight after
// each (what they shift out is zero in every candidate), so that its code stays
// in the instruction cache (unrolled over 32, a first run took 1.4 times a warm one).
template <int NS, typename Smem>
__device__ __forceinline__ uint32_t panel_search(Smem& sm, int16_t* prow, int nl, int p, int lane)
{
    uint32_t s[NS], c[NS];
    uint32_t q = 0u;
#pragma unroll
    for (int j = 0; j < NS; ++j) {
        s[j] = 32 * j + lane < nl ? __brev(sm.list[32 * j + lane]) : 0u;
        c[j] = 0u;
        q = max(q, s[j]);
    }
    q = __reduce_max_sync(0xffffffffu, q);
    uint32_t ps = 0u, pc = 0u;  // lane b: the slice and set of column b's pivot
    prow[lane] = -1;
#pragma unroll 1
    for (int b0 = 0; b0 < 32 && q; b0 += 8) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const uint32_t L = 0x80000000u >> u;
            const bool piv = q & L;
            const uint32_t qs = q;
            uint32_t rc = 0u, mx = 0u;
            bool has[NS];
#pragma unroll
            for (int j = 0; j < NS; ++j) {
                has[j] = s[j] & L;
                rc = max(rc, s[j] == qs ? c[j] : 0u);
                s[j] ^= has[j] ? qs : 0u;
                mx = max(mx, s[j]);
            }
            const uint32_t own = __reduce_max_sync(0xffffffffu, rc);
            q = __reduce_max_sync(0xffffffffu, mx);
            const uint32_t qc = own ^ (1u << (b0 + u));
#pragma unroll
            for (int j = 0; j < NS; ++j) c[j] ^= has[j] ? qc : 0u;
            const bool clears = piv && (ps & L);
            ps ^= clears ? qs : 0u;
            pc ^= clears ? qc : 0u;
            if (piv && lane == b0 + u) {
                ps = qs;
                pc = qc;
            }
        }
#pragma unroll
        for (int j = 0; j < NS; ++j) s[j] <<= 8;
        ps <<= 8;
        q <<= 8;
    }
    const uint32_t cols = __ballot_sync(0xffffffffu, pc != 0u);
    sm.Hcol[lane] = pc;
#pragma unroll
    for (int j = 0; j < NS; ++j) {
        // a pivot absorbed itself, which leaves its own column alone in its record;
        // so does a row whose start slice equals a pivot's, which is as good
        const int col = __popc(c[j]) == 1 ? 31 - __clz(c[j]) : -1;
        sm.kres[32 * j + lane] = (int16_t)col;
        if (col >= 0) prow[col] = sm.listrow[32 * j + lane];
    }
    __syncwarp();
    if (pc && HLF_IN_BOUNDS(32 * p + lane, (int)(sizeof sm.rowof / sizeof sm.rowof[0]), kSiteFactorSmem))
        sm.rowof[32 * p + lane] = prow[lane];
    if (lane == 0) {
        sm.pivmask[p] |= cols;
        sm.cols = cols;
    }
    return cols;
}

template <int N>
struct Words {
    static constexpr int value = N;
};

// W > 1: the elimination by panels of 32 columns, in a CTA of row threads (R rows
// each: t, t + row threads, ...) and one more warp that searches.
//
// Per panel: (a) the row threads list the slices of the live rows; (b) the searching
// warp finds the panel's pivots (panel_search); (c) T2 gets the combinations of the
// pivots' start rows over 4 columns each; (d) every row is rebuilt as itself XOR
// the start rows in its coefficient set, eight lookups a word. The reduced pivot
// row of column b is the set H_b, and a row that is not one of the panel's
// pivots, searched or not, absorbs the XOR of H over the pivot columns its start
// slice has (nibble tables T1). The result has zeros on the panel's pivot columns
// outside each pivot's own row and the same row space. Rows left over when the
// search took only a part of the list can still hold bits in columns that got no
// pivot; the panel is then searched again for them. Pivot columns are those of
// the unique echelon form whatever the order, so nothing depends on the list's.
//
// The search of a panel needs one word of every row only, so (c) and (d) do that
// word first and leave the others until the search of the next panel has begun:
// the row threads finish them while the other warp searches.
// `copy` ([W][stride], or null) receives A as it came; `meanwhile(warp, warps)` is
// called by the row warps while the first panel is searched.
template <int W, int R, int MAXN, typename F>
__device__ void eliminate_panels(const uint64_t* __restrict__ A, int n, unsigned char* smem, uint64_t* copy,
                                 F&& meanwhile)
{
    using Smem = FactorSmem<W, MAXN>;
    Smem& sm = *reinterpret_cast<Smem*>(smem);
    const int S = row_stride<W>(n);
    uint64_t* rows = factor_rows<W, MAXN>(smem);  // [W][S]
    uint64_t* T2 = rows + (size_t)W * S;          // [8][W][16]
    const int lane = threadIdx.x & 31;
    const int warp = warp_uniform(threadIdx.x >> 5);
    const int rt = 32 * row_warps(blockDim.x >> 5);
    const int npanels = (n + 31) >> 5;

    for (int i = threadIdx.x; i < MAXN / 32; i += blockDim.x) sm.pivmask[i] = 0u;
    for (int i = threadIdx.x; i < n; i += blockDim.x) sm.rowof[i] = -1;
    if (threadIdx.x < 2) sm.nlist[threadIdx.x] = 0;
    if (threadIdx.x == 2) sm.nactive = 0;
    __syncthreads();

    if (warp == search_warp(blockDim.x >> 5)) {
        for (int p = 0, round = 0; p < npanels; ++round) {
            bar_elim(rt);  // the list is there
            const int nl = warp_uniform(sm.nlist[round & 1]);
            if (lane == 0) sm.nlist[(round + 1) & 1] = 0;
            const int ncols = n - 32 * p < 32 ? n - 32 * p : 32;
            uint32_t cols = 0u;
            if (nl) {
                const int cap = panel_cap(nl);
                cols = cap == 32   ? panel_search<1>(sm, sm.prow[round & 1], nl, p, lane)
                       : cap == 64 ? panel_search<2>(sm, sm.prow[round & 1], nl, p, lane)
                                   : panel_search<4>(sm, sm.prow[round & 1], nl, p, lane);
            }
            if (panel_done(nl, cols, ncols)) ++p;
            bar_elim(rt);             // the pivots are known
            if (cols) bar_elim(rt);  // T1 and T2's first word are built
        }
        bar_elim(rt);
        return;
    }
    if ((warp & 3) == 3) return;               // idle
    const int tid = 32 * (warp - (warp >> 2)) + lane;  // the row thread's number

    auto bar_rows = [&]() {
        __syncwarp();
        asm volatile("bar.sync 2, %0;" ::"r"(rt) : "memory");
    };
#pragma unroll 8
    for (int i = tid; i < n * W; i += rt) {  // consecutive threads, consecutive words
        const uint64_t x = A[i];
        const int row = i / W, v = i % W;
        rows[v * S + row] = x;
        if (copy) copy[v * S + row] = x;
    }
    bool used[R];      // the row is a pivot row
    uint32_t coef[R];  // the pivots it absorbs in the current panel
#pragma unroll
    for (int j = 0; j < R; ++j) {
        used[j] = false;
        coef[j] = 0u;
    }
    bar_rows();
    const int16_t* prow = sm.prow[0];  // the last panel's
    // T2[(t, v, x)]: XOR of word v of the pivot rows of columns 4t + i, i over the bits of x
    auto build = [&](int t, int v, int x) {
        const uint64_t pr = *reinterpret_cast<const uint64_t*>(prow + 4 * t);
        uint64_t acc = 0ull;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int row = (int16_t)(pr >> (16 * i));
            if (((x >> i) & 1) && row >= 0 && HLF_IN_BOUNDS(row, n, kSiteFactorSmem)) acc ^= rows[v * S + row];
        }
        if (HLF_IN_BOUNDS((t * W + v) * 16 + x, 128 * W, kSiteFactorSmem)) T2[(t * W + v) * 16 + x] = acc;
    };
    auto update = [&](int row, uint32_t cf, int v) {
        uint64_t* x = rows + v * S + row;
        uint64_t a[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) a[t] = T2[(t * W + v) * 16 + ((cf >> (4 * t)) & 15u)];
        *x ^= ((a[0] ^ a[1]) ^ (a[2] ^ a[3])) ^ ((a[4] ^ a[5]) ^ (a[6] ^ a[7]));
    };
    // Words w_from.. but w_done still lack the last panel's update. The rows that
    // need it (on a grid, those near the panel) are listed and their words dealt to
    // all row warps: 32 rows and kTaskWords words a task, whose loads are all in flight at
    // once (random symmetric n = 1024: 200 us; word by word 214, n = 700: 100 and 105).
    constexpr int kTaskWords = 4;
    int w_from = W, w_done = 0;
    auto finish = [&]() {
        if (w_from + (w_done == w_from) >= W) return;  // uniform
        for (int q = tid >> 4; q < 8 * (W - w_from); q += rt >> 4) {
            const int v = w_from + (q >> 3);
            if (v != w_done) build(q & 7, v, tid & 15);
        }
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const unsigned m = __ballot_sync(0xffffffffu, coef[j] != 0u);
            if (!m) continue;
            int base = 0;
            if (lane == 0) base = atomicAdd(&sm.nactive, __popc(m));
            base = __shfl_sync(0xffffffffu, base, 0) + __popc(m & ((1u << lane) - 1u));
            if (coef[j] && HLF_IN_BOUNDS(base, MAXN, kSiteFactorSmem))
                sm.active[base] = make_uint2((uint32_t)(tid + j * rt), coef[j]);
        }
        bar_rows();
        const int na = sm.nactive;
        const int chunks = (na + 31) >> 5;
        int ch = tid >> 5, v0 = w_from + 1;  // w_from itself is done, or takes w_from + 1's place, which is
        for (;;) {
            while (ch >= chunks && v0 < W) {
                ch -= chunks;
                v0 += kTaskWords;
            }
            if (v0 >= W || !chunks) break;
            const int e = 32 * ch + lane;
            if (e < na) {
                const uint2 rc = sm.active[e];
                const uint64_t* tb[8];
#pragma unroll
                for (int t = 0; t < 8; ++t) tb[t] = T2 + (t * W + v0) * 16 + ((rc.y >> (4 * t)) & 15u);
                uint64_t* x = rows + v0 * S + rc.x;
                const int first = v0 == w_done ? -1 : 0;
                auto task = [&](auto words) {  // all the loads in flight
                    constexpr int N = decltype(words)::value;
                    uint64_t acc[N];
#pragma unroll
                    for (int i = 0; i < N; ++i) acc[i] = x[(i ? i : first) * S];
#pragma unroll
                    for (int t = 0; t < 8; ++t)
#pragma unroll
                        for (int i = 0; i < N; ++i) acc[i] ^= tb[t][16 * (i ? i : first)];
#pragma unroll
                    for (int i = 0; i < N; ++i) x[(i ? i : first) * S] = acc[i];
                };
                if (v0 + kTaskWords <= W) task(Words<kTaskWords>{});
                else if (v0 + 3 == W) task(Words<3>{});
                else if (v0 + 2 == W) task(Words<2>{});
                else task(Words<1>{});
            }
            ch += rt >> 5;
        }
        w_from = W;
    };
    for (int p = 0, round = 0; p < npanels; ++round) {
        const int w = p >> 1;
        const int ncols = n - 32 * p < 32 ? n - 32 * p : 32;
        const uint32_t in_n = ncols == 32 ? ~0u : (1u << ncols) - 1u;  // bits past n may be set in faulty input
        uint32_t s[R];
        int pos[R];
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const int row = tid + j * rt;
            s[j] = row < n ? (uint32_t)(rows[w * S + row] >> (32 * (p & 1))) & in_n : 0u;
            pos[j] = kPanelCap;
            const bool live = s[j] != 0u && !used[j];
            const unsigned m = __ballot_sync(0xffffffffu, live);
            if (m) {
                int base = 0;
                if (lane == 0) base = atomicAdd(&sm.nlist[round & 1], __popc(m));
                base = __shfl_sync(0xffffffffu, base, 0);
                if (live) {
                    pos[j] = base + __popc(m & ((1u << lane) - 1u));
                    if (pos[j] < kPanelCap) {
                        sm.list[pos[j]] = s[j];
                        sm.listrow[pos[j]] = (int16_t)row;
                    }
                }
            }
        }
        bar_elim(rt);  // the list is there
        if (round == 0) meanwhile(tid >> 5, rt >> 5);
        finish();
        bar_elim(rt);  // the pivots are known
        const int nl = sm.nlist[round & 1];
        const uint32_t cols = nl ? sm.cols : 0u;
        if (panel_done(nl, cols, ncols)) ++p;
        if (!cols) continue;  // uniform: nothing absorbs anything
        prow = sm.prow[round & 1];
        if (tid == 0) sm.nactive = 0;
        w_from = w;
        w_done = (p >> 1) < W ? (p >> 1) : w;
        for (int e = tid; e < 128; e += rt) build(e >> 4, w_done, e & 15);
        for (int e = tid; e < 128; e += rt) {  // T1[(t, x)]: XOR of Hcol over the columns 4t + i, i over the bits of x
            const uint4 h = *reinterpret_cast<const uint4*>(&sm.Hcol[4 * (e >> 4)]);
            sm.T1[e] = ((e & 1 ? h.x : 0u) ^ (e & 2 ? h.y : 0u)) ^ ((e & 4 ? h.z : 0u) ^ (e & 8 ? h.w : 0u));
        }
        const int cap = panel_cap(nl);
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const int b = pos[j] < cap ? sm.kres[pos[j]] : -1;
            // a pivot, unless its equal took the place
            const bool now = b >= 0 && HLF_IN_BOUNDS(b, 32, kSiteFactorSmem) && prow[b] == tid + j * rt;
            used[j] |= now;
            coef[j] = now ? sm.Hcol[b] ^ (1u << b) : 0u;
            if (now) s[j] = 0u;  // its set is known, not looked up
        }
        bar_elim(rt);  // T1 and T2's first word are built
#pragma unroll
        for (int j = 0; j < R; ++j) {
            if (s[j]) {
#pragma unroll
                for (int t = 0; t < 8; ++t) coef[j] ^= sm.T1[(t << 4) | ((s[j] >> (4 * t)) & 15u)];
            }
            if (coef[j]) update(tid + j * rt, coef[j], w_done);
        }
    }
    finish();
    bar_elim(rt);
}

// The input checks: padding bits, then symmetry, by warp `warp` of `nwarps`. A
// warp takes the 64 x 64 blocks (I, J) and (J, I), I <= J, of the W x W block
// grid, transposes the first in registers and compares it with the second on the
// rows and columns below n. Returns this thread's verdict.
template <int W>
__device__ __forceinline__ int check_rows(const uint64_t* __restrict__ A, int n, int warp, int nwarps)
{
    const int lane = threadIdx.x & 31;
    int bad = 0;
    const int tail = n & 63;
    if (tail)
        for (int i = warp * 32 + lane; i < n; i += nwarps * 32)
            if (A[(size_t)i * W + W - 1] >> tail) bad = HLF_ERR_PADDING;
    for (int pr = warp; pr < W * (W + 1) / 2; pr += nwarps) {
        int I = 0, rest = pr;  // pair index -> (I, J), I <= J < W
        while (rest >= W - I) {
            rest -= W - I;
            ++I;
        }
        const int J = I + rest;
        const int ra = 64 * I + lane, rb = 64 * J + lane;
        uint64_t p0 = ra < n ? A[(size_t)ra * W + J] : 0ull;
        uint64_t p1 = ra + 32 < n ? A[(size_t)(ra + 32) * W + J] : 0ull;
        const uint64_t q0 = rb < n ? A[(size_t)rb * W + I] : 0ull;
        const uint64_t q1 = rb + 32 < n ? A[(size_t)(rb + 32) * W + I] : 0ull;
        transpose64_warp(p0, p1, lane);
        const int cols = n - 64 * I;
        const uint64_t cm = cols >= 64 ? ~0ull : ((1ull << cols) - 1ull);
        if ((rb < n && ((p0 ^ q0) & cm)) || (rb + 32 < n && ((p1 ^ q1) & cm))) bad = max(bad, HLF_ERR_NOT_SYMMETRIC);
    }
    return bad;
}

__device__ __forceinline__ void write_info(const FactorOut& o, int status, int r)
{
    o.info[0] = status;
    o.info[1] = r;
    if (o.work) {
        o.work[kFactorDevInfo] = status;
        o.work[kFactorDevInfo + 1] = r;
    }
}

// The rank, p_k and the rows of B_k from the pivot mask and rowof, by the whole CTA.
template <int W, int MAXN>
__device__ __forceinline__ int order_pivots(FactorSmem<W, MAXN>& sm, int n)
{
    const int lane = threadIdx.x & 31;
    if (threadIdx.x < 32) {
        const int cnt = 32 * lane < n ? __popc(sm.pivmask[lane]) : 0;
        int incl = cnt;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += t;
        }
        if (32 * lane < n) sm.before[lane] = incl - cnt;
        if (lane == 31) sm.rank = incl;
    }
    __syncthreads();
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
        const uint32_t m = sm.pivmask[c >> 5];
        if (!((m >> (c & 31)) & 1u)) continue;
        const int k = sm.before[c >> 5] + __popc(m & ((1u << (c & 31)) - 1u));
        sm.pivcol[k] = (int16_t)c;
        sm.rowk[k] = sm.rowof[c];
    }
    __syncthreads();
    return sm.rank;
}

// Step (1)'s outputs: B_k in pivot order and the pivots (where asked for), the
// enumeration table's rows below min(r, 64) and zeros from there to row `rows_to`.
template <int W, int MAXN>
__device__ __forceinline__ void write_basis(const FactorSmem<W, MAXN>& sm, const uint64_t* rows, int n, int r,
                                            const FactorOut& o, int rows_to)
{
    const int S = row_stride<W>(n);
    const int nb = r < HLF_MAX_VARYING ? r : HLF_MAX_VARYING;
    const int last = o.basis ? r : nb;
    for (int i = threadIdx.x; i < last * W; i += blockDim.x) {
        const int k = i / W, v = i % W;
        const int row = sm.rowk[k];
        if (!HLF_IN_BOUNDS(row, S, kSiteFactorSmem)) continue;
        const uint64_t x = rows[v * S + row];
        if (o.basis) o.basis[i] = x;
        if (k < nb) o.table[i] = x;
    }
    if (o.piv)
        for (int k = threadIdx.x; k < r; k += blockDim.x) o.piv[k] = sm.pivcol[k];
    for (int i = nb * W + threadIdx.x; i < rows_to * W; i += blockDim.x) o.table[i] = 0ull;
}

// Factor the n x n matrix A ([n][W] words, global) with the whole CTA. W > 1: R * 32
// * row_warps(blockDim.x / 32) >= n; blockDim.x is a multiple of 32, at least 64.
// n <= MAXN.
// `smem` points to factor_smem_bytes<W, MAXN>(n, true) bytes of shared memory.
// Writes o.table (always), o.basis, o.piv and o.ptable (when non-null) and
// o.info[0] = status, o.info[1] = r (or -1 on a fault). Returns r, or -1.
//
// The steps around the elimination are chains of memory latencies, so they are
// laid beside something else: the checks beside the elimination (a fault is seen
// after it), the paper-order table (the last warp) and the outputs (the first)
// beside the kernel vectors, and A is read from memory once.
template <int W, int R, int MAXN>
__device__ int factor_block(const uint64_t* __restrict__ A, int n, const FactorOut& o, unsigned char* smem)
{
    using Smem = FactorSmem<W, MAXN>;
    Smem& sm = *reinterpret_cast<Smem*>(smem);
    const int S = row_stride<W>(n);
    uint64_t* rows = factor_rows<W, MAXN>(smem);
    uint64_t* As = rows + (size_t)W * S + (W > 1 ? 8 * 16 * W : 0);  // A, [W][S]
    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int warp = tid >> 5;
    const int nwarps = blockDim.x >> 5;

    if (tid == 0) sm.err = 0;
    if (tid < W) sm.z0[tid] = 0;
    __syncthreads();
    auto check = [&](int w, int nw) {
        if (const int bad = check_rows<W>(A, n, w, nw)) atomicMax(&sm.err, bad);
    };
    if constexpr (W == 1) {
        if (warp_uniform(warp) == 0) eliminate_warp<MAXN>(A, n, smem, As);
        else check(warp - 1, nwarps - 1);
    } else {
        eliminate_panels<W, R, MAXN>(A, n, smem, As, check);
    }
    __syncthreads();
    if (sm.err) {
        const int e = sm.err;
        __syncthreads();
        if (tid == 0) write_info(o, e, -1);
        return -1;
    }
    const int r = order_pivots(sm, n);
    const int nb = r < HLF_MAX_VARYING ? r : HLF_MAX_VARYING;

    // ---- the paper's own order (Section 2, Eq. 3; the counter of Section 4):
    // counter value t sets R_{p_j} = bit (r - j) of t, y = A R, z = y ^ z^a.
    // Bit l of t selects T_l = column p_{r-1-l} of A (0-based pivots), which is
    // row p_{r-1-l} since A is symmetric. With P_k = T_0 ^ ... ^ T_k, the Gray
    // walk over P visits z(t) in counter order, because bit l of t is the XOR
    // of the Gray code's bits k >= l. Lane l has rows l and l + 32, whose prefix
    // XORs are two scans.
    if (o.ptable && warp == nwarps - 1) {
        for (int v = 0; v < W; ++v) {
            uint64_t t0 = lane < nb ? As[v * S + sm.pivcol[r - 1 - lane]] : 0ull;
            uint64_t t1 = lane + 32 < nb ? As[v * S + sm.pivcol[r - 33 - lane]] : 0ull;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint64_t u0 = __shfl_up_sync(0xffffffffu, t0, d);
                const uint64_t u1 = __shfl_up_sync(0xffffffffu, t1, d);
                if (lane >= d) {
                    t0 ^= u0;
                    t1 ^= u1;
                }
            }
            t1 ^= __shfl_sync(0xffffffffu, t0, 31);
            o.ptable[lane * W + v] = lane < nb ? t0 : 0ull;
            o.ptable[(lane + 32) * W + v] = lane + 32 < nb ? t1 : 0ull;
            if (lane == 0) o.ptable[64 * W + v] = 0ull;
        }
    }

    // ---- (2)-(4): one warp per free column f, from the last warp but one down
    int err = 0;
    for (int f = nwarps - 1 - warp; f < n; f += nwarps) {
        if ((sm.pivmask[f >> 5] >> (f & 31)) & 1u) continue;  // pivot column (uniform per warp)
        const int fw = f >> 6;
        const int fb = f & 63;
        uint32_t x[2 * W];  // x_f, 32 bits a word
#pragma unroll
        for (int t = 0; t < 2 * W; ++t) {
            const int c = 32 * t + lane;
            const int row = c < n ? sm.rowof[c] : -1;
            x[t] = __ballot_sync(0xffffffffu, row >= 0 && ((rows[fw * S + row] >> fb) & 1ull));
            if (t == f >> 5) x[t] |= 1u << (f & 31);
        }
        unsigned acc = 0;
#pragma unroll
        for (int t = 0; t < 2 * W; ++t) {
            if ((x[t] >> lane) & 1u) {
#pragma unroll
                for (int v = 0; v < W; ++v)
                    acc += __popcll(As[v * S + 32 * t + lane] & (((uint64_t)x[2 * v + 1] << 32) | x[2 * v]));
            }
        }
        const unsigned q = __reduce_add_sync(0xffffffffu, acc) & 3u;
        if (q & 1u) err = HLF_ERR_INTERNAL;  // q is even on Ker(A) for symmetric A
        if (lane == 0 && (q >> 1))
            atomicOr(reinterpret_cast<unsigned long long*>(&sm.z0[fw]), 1ull << fb);
    }
    if (err) atomicMax(&sm.err, err);

    write_basis(sm, rows, n, r, o, kTableRows);
    __syncthreads();
    const int e = sm.err;
    if (tid < W) {
        o.table[kTableZ0Row * W + tid] = sm.z0[tid];
        if (o.ptable) o.ptable[kTableZ0Row * W + tid] = sm.z0[tid];
    }
    if (tid == 0) write_info(o, e, e ? -1 : r);
    __syncthreads();  // shared memory may be reused by the caller
    return e ? -1 : r;
}

}  // namespace hlf
