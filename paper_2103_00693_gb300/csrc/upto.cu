// Stage 2 for small instances without the rank on the host: the kernels read
// r from the words the factor kernel left in the handle's device memory.
//   store_upto_kernel   stores z(i) = z0 ^ XOR_{k in g(i)} B_k (Eq. 3 with
//                       the Gray-code basis order) for every i < min(2^r, cap),
//                       each by lookups in seed tables. Meant for
//                       instances of up to a few million solutions, where the
//                       time is the launch and the host round trip it saves;
//                       hlf_enumerate_store walks large windows.
//   reduce_upto_kernel  the reduce of [0, min(2^r, cap)) with the walk of the
//                       single-instance reduce; the run per thread is cut on
//                       the device from the actual count.

#include "enum_impl.cuh"
#include "upto.cuh"

namespace hlf {
namespace {

template <int W>
__global__ void __launch_bounds__(kThreads) store_upto_kernel(const uint64_t* __restrict__ table,
                                                              const int32_t* info, uint64_t cap,
                                                              uint64_t* __restrict__ out)
{
    __shared__ Table<W> t;
    __shared__ SeedTable<W> st;
    __shared__ uint64_t s_count;
    if (threadIdx.x == 0) {
        const int32_t r = *reinterpret_cast<const volatile int32_t*>(info + 1);  // -1 after a fault
        s_count = r < 0 ? 0ull : (r >= 64 ? cap : (cap < (1ull << r) ? cap : (1ull << r)));
    }
    load_table<W>(t, table);
    __syncthreads();
    const uint64_t count = s_count;
    const int ntab = seed_tables_for(cap - 1);
    build_seed_table<W>(st, t, ntab);
    __syncthreads();
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (uint64_t)gridDim.x * blockDim.x) {
        uint64_t z[W];
        seed_lookup<W>(st, ntab, i, z);
        if (HLF_IN_BOUNDS(i, cap, kSiteUptoStore)) {
#pragma unroll
            for (int w = 0; w < W; ++w) out[i * W + w] = z[w];
        }
    }
}

// CTAs an SM must hold (0: the compiler's choice). Left to itself it takes 48 registers
// at W = 5, too few to hash the four solutions of a block side by side: 2^20 solutions
// took 69.8 us, and take 53.6 with 70 registers; W = 8 92.7 -> 80.4, W = 3 37.4 -> 32.3.
// At W = 1 it lost 8% of 2^28, from W = 9 on it gave nothing.
constexpr int reduce_upto_ctas(int W) { return W > 1 && W <= 8 ? 2 : 0; }

template <int W, int U>
__global__ void __launch_bounds__(kThreads, reduce_upto_ctas(W)) reduce_upto_kernel(const uint64_t* __restrict__ table,
                                                               const int32_t* info, uint64_t cap,
                                                               hlf_reduce* __restrict__ out)
{
    __shared__ Table<W> t;
    __shared__ SeedTable<W> st;
    __shared__ uint64_t s_count;
    if (threadIdx.x == 0) {
        const int32_t r = *reinterpret_cast<const volatile int32_t*>(info + 1);  // -1 after a fault
        s_count = r < 0 ? 0ull : (r >= 64 ? cap : (cap < (1ull << r) ? cap : (1ull << r)));
    }
    const bool mixed = __syncthreads_or(load_table_hash_domain<W, U>(t, table));
    const uint64_t count = s_count;
    const int ntab = seed_tables_for(cap - 1);
    build_seed_table<W>(st, t, ntab);
    __syncthreads();
    const uint64_t threads = (uint64_t)gridDim.x * blockDim.x;
    uint64_t per = (count + threads - 1) / threads;
    per = (per + (1ull << U) - 1) & ~((1ull << U) - 1);  // runs stay aligned to the Gray blocks
    if (per == 0) per = 1ull << U;
    const uint64_t a = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) * per;
    Acc<W> acc;
    acc.zero();
    uint64_t cnt = 0;
    if (a < count) {
        cnt = min(per, count - a);
        uint64_t z[W];
        seed_lookup<W>(st, ntab, a, z);
        reduce_run_from<W, U>(t, mixed, a, cnt, z, acc);
    }
    block_reduce<W>(cnt, acc);
    if (threadIdx.x == 0 && cnt) {
        atomicAdd(reinterpret_cast<unsigned long long*>(&out->count), (unsigned long long)cnt);
        atomicAdd(reinterpret_cast<unsigned long long*>(&out->hsum), (unsigned long long)acc.hs);
#pragma unroll
        for (int w = 0; w < W; ++w) {
            const uint64_t f = acc.fold_word(w);
            if (f) atomicXor(reinterpret_cast<unsigned long long*>(&out->xor_fold[w]), (unsigned long long)f);
        }
    }
}

template <int W>
hlf_status launch_reduce_upto_w(const uint64_t* table, const int32_t* info, uint64_t cap, hlf_reduce* out,
                                cudaStream_t s)
{
    constexpr int U = reduce_unroll(W);
    // 8 CTAs of 256 threads per SM at most, and runs of at least 256 solutions
    // when the whole cap is enumerated, which makes 16 CTAs of 2^20
    const uint64_t most = (uint64_t)sm_count() * 8;
    uint64_t blocks = (cap + 256 * kThreads - 1) / (256 * kThreads);
    if (blocks > most) blocks = most;
    if (blocks == 0) blocks = 1;
    reduce_upto_kernel<W, U><<<(unsigned)blocks, kThreads, 0, s>>>(table, info, cap, out);
    return cudaGetLastError() == cudaSuccess ? HLF_OK : HLF_ERR_CUDA;
}

template <int W>
hlf_status launch_store_upto_w(const uint64_t* table, const int32_t* info, uint64_t cap, uint64_t* out,
                               cudaStream_t s)
{
    const uint64_t most = (uint64_t)sm_count() * 4;
    uint64_t blocks = (cap + kThreads - 1) / kThreads;
    if (blocks > most) blocks = most;
    if (blocks == 0) blocks = 1;
    store_upto_kernel<W><<<(unsigned)blocks, kThreads, 0, s>>>(table, info, cap, out);
    return cudaGetLastError() == cudaSuccess ? HLF_OK : HLF_ERR_CUDA;
}

}  // namespace

hlf_status launch_reduce_upto(const uint64_t* table, int W, const int32_t* info, uint64_t cap, hlf_reduce* out,
                              cudaStream_t s)
{
    switch (W) {
    case 1: return launch_reduce_upto_w<1>(table, info, cap, out, s);
    case 2: return launch_reduce_upto_w<2>(table, info, cap, out, s);
    case 3: return launch_reduce_upto_w<3>(table, info, cap, out, s);
    case 4: return launch_reduce_upto_w<4>(table, info, cap, out, s);
    case 5: return launch_reduce_upto_w<5>(table, info, cap, out, s);
    case 6: return launch_reduce_upto_w<6>(table, info, cap, out, s);
    case 7: return launch_reduce_upto_w<7>(table, info, cap, out, s);
    case 8: return launch_reduce_upto_w<8>(table, info, cap, out, s);
    case 9: return launch_reduce_upto_w<9>(table, info, cap, out, s);
    case 10: return launch_reduce_upto_w<10>(table, info, cap, out, s);
    case 11: return launch_reduce_upto_w<11>(table, info, cap, out, s);
    case 12: return launch_reduce_upto_w<12>(table, info, cap, out, s);
    case 13: return launch_reduce_upto_w<13>(table, info, cap, out, s);
    case 14: return launch_reduce_upto_w<14>(table, info, cap, out, s);
    case 15: return launch_reduce_upto_w<15>(table, info, cap, out, s);
    case 16: return launch_reduce_upto_w<16>(table, info, cap, out, s);
    default: return HLF_ERR_SIZE;
    }
}

hlf_status launch_store_upto(const uint64_t* table, int W, const int32_t* info, uint64_t cap, uint64_t* out,
                             cudaStream_t s)
{
    switch (W) {
    case 1: return launch_store_upto_w<1>(table, info, cap, out, s);
    case 2: return launch_store_upto_w<2>(table, info, cap, out, s);
    case 3: return launch_store_upto_w<3>(table, info, cap, out, s);
    case 4: return launch_store_upto_w<4>(table, info, cap, out, s);
    case 5: return launch_store_upto_w<5>(table, info, cap, out, s);
    case 6: return launch_store_upto_w<6>(table, info, cap, out, s);
    case 7: return launch_store_upto_w<7>(table, info, cap, out, s);
    case 8: return launch_store_upto_w<8>(table, info, cap, out, s);
    case 9: return launch_store_upto_w<9>(table, info, cap, out, s);
    case 10: return launch_store_upto_w<10>(table, info, cap, out, s);
    case 11: return launch_store_upto_w<11>(table, info, cap, out, s);
    case 12: return launch_store_upto_w<12>(table, info, cap, out, s);
    case 13: return launch_store_upto_w<13>(table, info, cap, out, s);
    case 14: return launch_store_upto_w<14>(table, info, cap, out, s);
    case 15: return launch_store_upto_w<15>(table, info, cap, out, s);
    case 16: return launch_store_upto_w<16>(table, info, cap, out, s);
    default: return HLF_ERR_SIZE;
    }
}

HLF_DEBUG_TAKE(upto)

}  // namespace hlf
