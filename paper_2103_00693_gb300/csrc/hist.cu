// Histogram of a bit field of every solution in a window: the counts behind
// the paper's output distributions of Figs. 3, 6 and 7, where each square
// shows how often one bit pattern of the first or last bits occurs.
//
// The field of a solution, bits [lo, lo + nbits) of z, is a GF(2)-linear
// function of z. With f_k the field of B_k and f_z the field of z0, the field of
// z(i) is v(i) = f_z ^ XOR_{k in g(i)} f_k. Over an aligned block of 2^m
// indices the low m bits of g(i) take every value once and the others stay, so
// the fields of the block are the coset v(base) ^ span(f_0 .. f_{m-1}), each
// element of it 2^(m - rho_m) times, rho_m = rank(f_0 .. f_{m-1}). A window is
// at most 126 aligned blocks, hence the count of bin v is
//     sum over blocks of (v ^ v(base) in span(f_0 .. f_{m-1})) * 2^(m - rho_m),
// exactly what counting solution by solution gives, at a cost that depends on
// the bins and not on the solutions.
//
// Membership: the spans are nested, so one invertible map T of the field takes
// span(f_0 .. f_{m-1}) to the values below 2^rho_m for every m at once, and the
// test is (T(v) ^ T(v(base))) >> rho_m == 0. One warp finds T with a step per rank,
// all fields mapped as far as T is known: the first row whose image has a bit at or
// above the rank has its top bit swapped to the rank's position and cleared
// everywhere else, which leaves the earlier spans' images alone. Blocks whose span
// is the whole field add a constant to every bin.
//
// What bounds it: the launch and the prologue's serial steps up to 2^15 bins,
// the bins' stores above. 2^30 solutions into 2^14 bins take 5.7 us a call (8.2 with a
// step per row instead of per rank).
// Counting them one by one took 137-155 us, bound by one shared-memory atomic per
// solution.

#include "enum_impl.cuh"

namespace hlf {
namespace {

constexpr int kHistMaxBlocks = 128;
constexpr int kHistTables = (HLF_HIST_MAX_BITS + 3) / 4;

// The window's aligned blocks: [base, base + 2^m).
struct HistPlan {
    uint64_t base[kHistMaxBlocks];
    uint8_t m[kHistMaxBlocks];
    int n;
    int max_m;
    int W;  // the table's words per row
};

// A block that counts only some bins: 2^(m - rho) for each v with
// (T(v) ^ t) >> rho == 0.
struct __align__(16) HistPart {
    uint32_t t;
    uint32_t rho;
    uint64_t each;
};

__global__ void __launch_bounds__(kThreads) hist_kernel(const uint64_t* __restrict__ table,
                                                        const __grid_constant__ HistPlan pl, int lo, int nbits,
                                                        uint64_t* __restrict__ out)
{
    __shared__ uint32_t s_tf[kTableTotalRows];  // T of the fields of the rows and of z0
    __shared__ uint32_t s_col[32];              // T(e_l)
    __shared__ uint32_t s_T[kHistTables][16];   // T of four bits of the field
    __shared__ uint32_t s_G[16][16];            // T of four rows' fields, for the blocks' bases
    __shared__ uint64_t s_rows;                 // the rows k that raise the rank
    __shared__ HistPart s_part[kHistMaxBlocks];
    __shared__ unsigned long long s_all;  // what every bin gets
    __shared__ int s_nparts;
    const int tid = threadIdx.x;
    const int lane = tid & 31;
    if (warp_uniform(tid >> 5) == 0) {
        const int word = lo >> 6, sh = lo & 63;
        auto field = [&](int k) {
            const uint64_t* row = table + (size_t)k * pl.W;
            uint64_t v = row[word] >> sh;
            if (sh && word + 1 < pl.W) v |= row[word + 1] << (64 - sh);
            return (uint32_t)(v & ((1ull << nbits) - 1));
        };
        uint32_t u0 = field(lane), u1 = field(lane + 32), uz = field(kTableZ0Row);  // T of these, so far
        uint32_t col = lane < nbits ? 1u << lane : 0u;
        const bool in0 = lane < pl.max_m, in1 = lane + 32 < pl.max_m;
        uint64_t rows = 0;
        for (int rho = 0; rho < nbits; ++rho) {  // uniform
            const unsigned b0 = __ballot_sync(0xffffffffu, in0 && (u0 >> rho)), b1 = __ballot_sync(0xffffffffu, in1 && (u1 >> rho));
            if (!(b0 | b1)) break;
            const int k = b0 ? __ffs(b0) - 1 : 31 + __ffs(b1);  // the next row out of the span
            const uint32_t u = __shfl_sync(0xffffffffu, b0 ? u0 : u1, k & 31);
            const int p = 31 - __clz(u);  // at least rho
            // bits p and rho swap places; then the row's image keeps bit rho only
            auto swap = [&](uint32_t x) {
                const uint32_t d = ((x >> p) ^ (x >> rho)) & 1u;
                return p == rho ? x : x ^ (d << p) ^ (d << rho);
            };
            const uint32_t clear = swap(u) ^ (1u << rho);
            auto step = [&](uint32_t x) {
                x = swap(x);
                return (x >> rho) & 1u ? x ^ clear : x;
            };
            u0 = step(u0);
            u1 = step(u1);
            uz = step(uz);
            col = step(col);
            rows |= 1ull << k;
        }
        s_tf[lane] = u0;
        s_tf[lane + 32] = u1;
        s_col[lane] = col;
        if (lane == 0) {
            s_tf[kTableZ0Row] = uz;
            s_rows = rows;
            s_all = 0;
            s_nparts = 0;
        }
    }
    __syncthreads();
    {
        uint32_t v = 0, g = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            if ((tid >> b) & 1) {
                g ^= s_tf[(tid >> 4) * 4 + b];
                if (tid < kHistTables * 16) v ^= s_col[(tid >> 4) * 4 + b];
            }
        }
        s_G[tid >> 4][tid & 15] = g;
        if (tid < kHistTables * 16) s_T[tid >> 4][tid & 15] = v;
    }
    __syncthreads();
    auto map = [&](uint32_t v) {
        uint32_t u = s_T[0][v & 15];
#pragma unroll
        for (int q = 1; q < kHistTables; ++q) u ^= s_T[q][(v >> (4 * q)) & 15];
        return u;
    };
    for (int b = tid; b < pl.n; b += kThreads) {
        const int m = pl.m[b];
        const int rho = __popcll(s_rows & ((1ull << m) - 1));
        if (rho == nbits) {
            atomicAdd(&s_all, 1ull << (m - rho));
            continue;
        }
        const uint64_t g = pl.base[b] ^ (pl.base[b] >> 1);
        uint32_t t = s_tf[kTableZ0Row];
#pragma unroll
        for (int q = 0; q < 16; ++q) t ^= s_G[q][(g >> (4 * q)) & 15];
        s_part[atomicAdd(&s_nparts, 1)] = {t, (uint32_t)rho, 1ull << (m - rho)};
    }
    __syncthreads();
    const uint64_t all = s_all;
    const int np = s_nparts;
    const uint32_t nb = 1u << nbits;
    for (uint32_t v = blockIdx.x * kThreads + tid; v < nb; v += gridDim.x * kThreads) {
        const uint32_t u = map(v);
        uint64_t c = all;
        for (int j = 0; j < np; ++j) {
            const HistPart h = s_part[j];
            c += ((u ^ h.t) >> h.rho) == 0 ? h.each : 0ull;
        }
        if (HLF_IN_BOUNDS(v, nb, kSiteHistBin)) out[v] = c;
    }
}

}  // namespace

hlf_status launch_histogram(const uint64_t* table, int W, uint64_t offset, uint64_t count, int lo, int nbits,
                            uint64_t* out, cudaStream_t s)
{
    if (W < 1 || W > HLF_MAX_W || lo < 0 || nbits < 1 || nbits > HLF_HIST_MAX_BITS || lo + nbits > 64 * W)
        return HLF_ERR_ARG;
    HistPlan pl{};
    pl.W = W;
    // blocks as large as the position and what is left allow: sizes rise, then
    // fall, so at most 63 of each (the end may be 2^64, where `a` wraps to 0)
    for (uint64_t a = offset, left = count; left;) {
        int m = 63;
        while ((1ull << m) > left || (a & ((1ull << m) - 1))) --m;
        pl.base[pl.n] = a;
        pl.m[pl.n++] = (uint8_t)m;
        if (m > pl.max_m) pl.max_m = m;
        a += 1ull << m;
        left -= 1ull << m;
    }
    const uint32_t blocks = ((1u << nbits) + kThreads - 1) / kThreads;
    const uint32_t cap = (uint32_t)sm_count() * 4;
    hist_kernel<<<blocks < cap ? blocks : cap, kThreads, 0, s>>>(table, pl, lo, nbits, out);
    return cudaGetLastError() == cudaSuccess ? HLF_OK : HLF_ERR_CUDA;
}

HLF_DEBUG_TAKE(hist)

}  // namespace hlf
