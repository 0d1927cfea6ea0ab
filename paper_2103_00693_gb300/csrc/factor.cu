// Stage 1 for one matrix (the CLA module of Section 2, steps (1)-(4)).
//
// n <= 256 (W <= 4): one CTA runs factor_block (factor_impl.cuh): input
// checks, elimination, kernel vectors, q and z^a in one launch, which is what
// the latency of small and medium instances wants.
//
// n > 256 (W >= 5): the same results from two launches that spread the work
// that does not have to be sequential over many SMs:
//   factor_elim_kernel   CTA 0 runs the Gauss-Jordan elimination (step (1),
//                        eliminate_panels); CTAs 1.. check the input (padding
//                        bits, symmetry by 64 x 64 bit-block transposes) at the
//                        same time, each writing its own status slot.
//   factor_kvec_kernel   one CTA per free column f across the GPU: the
//                        kernel vector x_f, q(x_f) mod 4 and the bit z^a_f
//                        (steps (2)-(4)), the paper-order table, and, in
//                        the last CTA to finish, the status and rank.
//
// What bounds it is the serial chain of the pivots. Event averages over 20
// back-to-back launches, before (every warp holding live rows searched, with a CTA
// barrier per column; up to n = 256 every row took the pivot row's words each
// column) and now:
//   grid, p = 1/2        n = 100: 21.2 -> 14.4 us   256: 50.7 -> 28.7
//                        484: 81.8 -> 47.2          1024: 202 -> 99
//   random symmetric     n = 256: 47.4 -> 24.7      1024: 309 -> 200
// Per panel of 32 columns at n = 1024 (cycles): the search 4100 on a grid and 5200
// on a dense matrix (with a warp to itself and nothing else on the SM 1900 to 3500,
// by how many slices are live), the list and the first word's tables and updates
// 1000; the other words' tables and updates, 3000 on a grid, are hidden behind the
// next search; on a dense matrix their shared-memory reads (5900 cycles of bandwidth a
// panel at first) are what it waits for.
//
// Measured on the way: the search by ballot, find-first and shuffles instead of
// maxima 200 cycles a column against 60 to 110; the words dealt to their rows' owners
// instead of all row warps 131 us against 105 (grid 32 x 32), A loaded row by row
// instead of coalesced 17k cycles against 4k. A thread-block cluster sharing the
// rows: its barrier alone takes about 400 cycles a round trip on this GPU. 24 row warps
// instead of 11 to 16 above n = 512: grid 32 x 32 111 us against 105.

#include "factor_impl.cuh"

namespace hlf {
namespace {

template <int W>
constexpr int rows_per_thread() { return W <= 8 ? 1 : 2; }

// W = 1: one warp eliminates, three check.
template <int W>
constexpr int factor_threads(int n)
{
    constexpr int R = rows_per_thread<W>();
    return W == 1 ? 128 : elim_threads((n + R - 1) / R);
}

template <int W>
__global__ void __launch_bounds__(factor_threads<W>(64 * W), 1) factor_kernel(const uint64_t* __restrict__ A, int n, FactorOut o)
{
    extern __shared__ __align__(16) unsigned char smem[];
    factor_block<W, 1, 256>(A, n, o, smem);
}

template <int W>
hlf_status launch_factor_w(const uint64_t* A, int n, const FactorOut& o, cudaStream_t s)
{
    static_assert(factor_smem_bytes<W, 256>(64 * W, true) <= 48 * 1024, "fits the default dynamic shared-memory limit");
    factor_kernel<W><<<1, factor_threads<W>(n), factor_smem_bytes<W, 256>(n, true), s>>>(A, n, o);
    return cudaGetLastError() == cudaSuccess ? HLF_OK : HLF_ERR_CUDA;
}

// ------------------------------------------------------------ n > 256

constexpr int kChkCtas = 8;       // CTAs that check the input beside the elimination
constexpr int kWorkR = 16;        // work[16] = r
constexpr int kWorkInternal = 17; // work[17] = HLF_ERR_INTERNAL if some q(x_f) was odd
constexpr int kWorkDone = 18;     // work[18] = CTAs of factor_kvec_kernel done
constexpr int kWorkMask = 32;     // work[32..64) = the pivot columns, one bit each
constexpr int kKvecCtas = 256;    // CTAs of factor_kvec_kernel (one free column at a time each)
static_assert(kWorkMask + HLF_MAX_N / 32 <= kFactorWorkWords, "the pivot mask fits the scratch words");
static_assert(kWorkDone < kFactorDevInfo && kFactorDevInfo + 2 <= kWorkMask, "the scratch words do not overlap");
static_assert(kChkCtas <= kWorkR, "one status slot per checking CTA");

// Step (1) for the whole CTA: the reduced row echelon form, pivots and the
// enumeration table; the kernel-vector step and the input checks are left to the
// other CTAs and kernel. Also zeroes the z^a rows of both tables
// (factor_kvec_kernel ORs the bits in) and the scratch words the second kernel
// uses, and publishes r in work[kWorkR].
template <int W, int R>
__device__ void eliminate_only(const uint64_t* __restrict__ A, int n, const FactorOut& o, unsigned char* smem)
{
    FactorSmem<W, HLF_MAX_N>& sm = *reinterpret_cast<FactorSmem<W, HLF_MAX_N>*>(smem);
    const int tid = threadIdx.x;
    eliminate_panels<W, R, HLF_MAX_N>(A, n, smem, nullptr, [](int, int) {});
    const int r = order_pivots(sm, n);
    // Behind order_pivots' barriers: a CTA releases its dependents when the first of its
    // threads does, and the idle warps leave the elimination at its start.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int nb = r < HLF_MAX_VARYING ? r : HLF_MAX_VARYING;
    write_basis(sm, factor_rows<W, HLF_MAX_N>(smem), n, r, o, kTableTotalRows);
    if (o.ptable)
        for (int i = nb * W + tid; i < kTableTotalRows * W; i += blockDim.x) o.ptable[i] = 0ull;
    if (tid < HLF_MAX_N / 32) o.work[kWorkMask + tid] = (int32_t)sm.pivmask[tid];
    if (tid == 0) {
        o.work[kWorkR] = r;
        o.work[kWorkInternal] = 0;
        o.work[kWorkDone] = 0;
    }
}

// The input checks, spread over the checking CTAs. CTA k writes its verdict (0
// or the larger code) to work[k]; every slot is written, so nothing needs
// clearing beforehand.
template <int W>
__device__ void check_input(const uint64_t* __restrict__ A, int n, int cta, int nctas, int32_t* work)
{
    __shared__ int s_bad;
    const int nwarps = blockDim.x >> 5;
    if (threadIdx.x == 0) s_bad = 0;
    __syncthreads();
    const int bad = check_rows<W>(A, n, cta * nwarps + (threadIdx.x >> 5), nctas * nwarps);
    if (bad) atomicMax(&s_bad, bad);
    __syncthreads();
    if (threadIdx.x == 0) work[cta] = s_bad;
}

template <int W>
__global__ void __launch_bounds__(factor_threads<W>(64 * W), 1) factor_elim_kernel(const uint64_t* __restrict__ A, int n, FactorOut o)
{
    extern __shared__ __align__(16) unsigned char smem[];
    if (blockIdx.x > 0) {
        check_input<W>(A, n, (int)blockIdx.x - 1, (int)gridDim.x - 1, o.work);
        return;
    }
    eliminate_only<W, rows_per_thread<W>()>(A, n, o, smem);
}

// Steps (2)-(4), one CTA per free column f (the j-th free column, j =
// blockIdx.x, blockIdx.x + gridDim.x, ..., found from the pivot mask the
// elimination left in the scratch words): x_f = e_f + sum_k B_k[f] e_{p_k},
// q(x_f) = sum over i in supp(x_f) of popcount(A_i & x_f) mod 4, and
// z^a_f = q(x_f) / 2 (z^a vanishes on the pivots). Each thread takes every
// 256th k and every 256th row, so a free column costs a few rounds of
// memory latency, not one per row. Word v of the paper-order table is built by warp
// 1 of CTA v (all of it in one warp, rows in a chain, outlasted the free columns:
// 18 us against 11 at n = 1024, cold). The last CTA to finish folds the checking
// CTAs' verdicts and the q parity into the status word.
template <int W>
__global__ void __launch_bounds__(256) factor_kvec_kernel(const uint64_t* __restrict__ A, int n, FactorOut o,
                                                          int n_chk)
{
    __shared__ uint32_t s_mask[HLF_MAX_N / 32];  // free columns below n, by word
    __shared__ int s_before[HLF_MAX_N / 32];     // free columns in the words before
    __shared__ uint64_t s_x[W];
    __shared__ unsigned s_q;
    __shared__ bool s_last;
    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int warp = tid >> 5;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int r = __ldcg(o.work + kWorkR);
    if (warp == 0) {
        const int c0 = lane * 32;
        const uint32_t below_n = c0 >= n ? 0u : (n - c0 >= 32 ? ~0u : ((1u << (n - c0)) - 1u));
        const uint32_t fm = ~(uint32_t)__ldcg(o.work + kWorkMask + lane) & below_n;
        const int cnt = __popc(fm);
        int incl = cnt;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += t;
        }
        s_mask[lane] = fm;
        s_before[lane] = incl - cnt;
    }
    if (blockIdx.x < W && warp == 1 && o.ptable) {
        // the paper's order, word v of it by CTA v: row l = XOR of A's columns (= rows) at
        // p_{r-1}, .., p_{r-1-l}; lane l has rows l and l + 32, two scans
        const int v = blockIdx.x;
        const int nb = r < HLF_MAX_VARYING ? r : HLF_MAX_VARYING;
        uint64_t t0 = lane < nb ? A[(size_t)__ldcg(o.piv + r - 1 - lane) * W + v] : 0ull;
        uint64_t t1 = lane + 32 < nb ? A[(size_t)__ldcg(o.piv + r - 33 - lane) * W + v] : 0ull;
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
        if (lane < nb) o.ptable[lane * W + v] = t0;
        if (lane + 32 < nb) o.ptable[(lane + 32) * W + v] = t1;
    }
    __syncthreads();

    int err = 0;
    const int nfree = n - r;
    for (int j = blockIdx.x; j < nfree; j += gridDim.x) {
        // the j-th free column: the last mask word with at most j free
        // columns before it holds it
        const int l = 31 - __clz(__ballot_sync(0xffffffffu, s_before[lane] <= j));
        uint32_t m = s_mask[l];
        for (int t = j - s_before[l]; t > 0; --t) m &= m - 1u;
        if (!m) continue;  // not reached: the mask has n - r free columns (uniform)
        const int f = 32 * l + __ffs(m) - 1;
        const int fw = f >> 6;
        const int fb = f & 63;
        if (tid < W) s_x[tid] = tid == fw ? (1ull << fb) : 0ull;
        if (tid == 0) s_q = 0u;
        __syncthreads();
        // bit p_k of x_f is B_k[f]: thread t sets the bits of k = t, t + 256, ...
        for (int k0 = tid; k0 < r; k0 += 1024) {  // four loads in flight
            uint64_t bk[4];
            int pc[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = k0 + 256 * u;
                bk[u] = k < r ? __ldcg(o.basis + (size_t)k * W + fw) : 0ull;
                pc[u] = k < r ? __ldcg(o.piv + k) : 0;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (((bk[u] >> fb) & 1ull) && HLF_IN_BOUNDS(pc[u] >> 6, W, kSiteFactorKvec))
                    atomicOr(reinterpret_cast<unsigned long long*>(&s_x[pc[u] >> 6]), 1ull << (pc[u] & 63));
        }
        __syncthreads();
        uint64_t xr[W];
#pragma unroll
        for (int v = 0; v < W; ++v) xr[v] = s_x[v];
        unsigned acc = 0;
        for (int i0 = tid; i0 < n; i0 += 512) {  // two rows' loads in flight
            const int i1 = i0 + 256;
            const bool in0 = (s_x[i0 >> 6] >> (i0 & 63)) & 1ull;
            const bool in1 = i1 < n && ((s_x[i1 >> 6] >> (i1 & 63)) & 1ull);
#pragma unroll
            for (int v = 0; v < W; ++v) {
                const uint64_t a0 = in0 ? A[(size_t)i0 * W + v] : 0ull;
                const uint64_t a1 = in1 ? A[(size_t)i1 * W + v] : 0ull;
                acc += __popcll(a0 & xr[v]) + __popcll(a1 & xr[v]);
            }
        }
        acc = __reduce_add_sync(0xffffffffu, acc);
        if (lane == 0) atomicAdd(&s_q, acc);
        __syncthreads();
        if (tid == 0) {
            const unsigned q = s_q & 3u;
            if (q & 1u) err = HLF_ERR_INTERNAL;  // q is even on Ker(A) for symmetric A
            if ((q >> 1) && HLF_IN_BOUNDS(fw, W, kSiteFactorKvec)) {
                atomicOr(reinterpret_cast<unsigned long long*>(o.table + kTableZ0Row * W + fw), 1ull << fb);
                if (o.ptable)
                    atomicOr(reinterpret_cast<unsigned long long*>(o.ptable + kTableZ0Row * W + fw), 1ull << fb);
            }
        }
        __syncthreads();  // s_x and s_q serve the next free column
    }
    if (err) atomicMax(o.work + kWorkInternal, err);
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        s_last = atomicAdd(o.work + kWorkDone, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (s_last && tid == 0) {
        __threadfence();
        // an input fault first (as factor_block reports it), then an odd q
        int st = 0;
        for (int k = 0; k < n_chk; ++k) st = max(st, __ldcg(o.work + k));
        if (!st) st = __ldcg(o.work + kWorkInternal);
        write_info(o, st, st ? -1 : r);
    }
}

template <int W>
hlf_status launch_factor_large(const uint64_t* A, int n, const FactorOut& o, cudaStream_t s)
{
    if (!o.work) return HLF_ERR_INTERNAL;
    const size_t smem = factor_smem_bytes<W, HLF_MAX_N>(n, false);
    static bool attr_set[64] = {false};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 64 && !attr_set[dev]) {
        if (cudaFuncSetAttribute(factor_elim_kernel<W>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)factor_smem_bytes<W, HLF_MAX_N>(64 * W, false)) != cudaSuccess)
            return HLF_ERR_CUDA;
        attr_set[dev] = true;
    }
    factor_elim_kernel<W><<<1 + kChkCtas, factor_threads<W>(n), smem, s>>>(A, n, o);
    if (cudaGetLastError() != cudaSuccess) return HLF_ERR_CUDA;
    // Launched when the elimination has only its results to write: grid 32 x 32 102.5 us
    // (104.5 launched when it has ended), random symmetric n = 700 89.9 (92.4), n = 1024
    // 200.8 (202.9). Not sooner: its CTAs wait on every SM, and other streams' kernels of
    // large CTAs find no room beside them. Released at the elimination's start, 8
    // factorisations of n = 1024 on 8 streams took 391 us (now 221), and a reduce of 40 us
    // on another stream 208 (now 44).
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = kKvecCtas;
    cfg.blockDim = 256;
    cfg.stream = s;
    cudaLaunchAttribute beside{};
    beside.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    beside.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &beside;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, factor_kvec_kernel<W>, A, n, o, (int)kChkCtas) == cudaSuccess ? HLF_OK : HLF_ERR_CUDA;
}

}  // namespace

hlf_status launch_factor(const uint64_t* A, int n, int W, const FactorOut& o, cudaStream_t s)
{
    switch (W) {
    case 1: return launch_factor_w<1>(A, n, o, s);
    case 2: return launch_factor_w<2>(A, n, o, s);
    case 3: return launch_factor_w<3>(A, n, o, s);
    case 4: return launch_factor_w<4>(A, n, o, s);
    case 5: return launch_factor_large<5>(A, n, o, s);
    case 6: return launch_factor_large<6>(A, n, o, s);
    case 7: return launch_factor_large<7>(A, n, o, s);
    case 8: return launch_factor_large<8>(A, n, o, s);
    case 9: return launch_factor_large<9>(A, n, o, s);
    case 10: return launch_factor_large<10>(A, n, o, s);
    case 11: return launch_factor_large<11>(A, n, o, s);
    case 12: return launch_factor_large<12>(A, n, o, s);
    case 13: return launch_factor_large<13>(A, n, o, s);
    case 14: return launch_factor_large<14>(A, n, o, s);
    case 15: return launch_factor_large<15>(A, n, o, s);
    case 16: return launch_factor_large<16>(A, n, o, s);
    default: return HLF_ERR_SIZE;
    }
}

HLF_DEBUG_TAKE(factor)

}  // namespace hlf
