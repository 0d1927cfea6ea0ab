// Many enumeration windows, of different matrices and word counts, stored in
// ONE launch: the serving path's continuous batching. Each window is the
// stage-2 materialisation of hlf_enumerate_store (Section 2, Fig. 1(c)); the
// batching only schedules them together.
//
// The host cuts every window into tasks of about 4 KB of output: the first of a
// window write its ragged ends (the indices outside its groups), 32 indices each,
// the others cover task_groups(W) groups of consecutive indices each. A warp takes an equal run of tasks, finds its first window by binary
// search over the task prefix sums, and stores the groups of each window in the run
// in one walk (store_groups), so that it seeds itself once a window: a seed is one
// round of loads, every lane bringing two rows, and the window's first step rows are
// staged in shared memory.
// 48 windows of 106 MB: the kernel took 69 us with 64-group tasks taken one by one
// and seeded row by row from global memory, 52 with 16 KB tasks one by one, and takes
// about 33 now; calls in a row are bound by the host's 50 us a call.

#include <new>

#include "enum_impl.cuh"

namespace hlf {
namespace {

// A task is the unit that the warps' shares differ by.
__host__ __device__ constexpr uint64_t task_groups(uint32_t W) { return W == 1 ? 8 : (16 + W - 1) / W; }
constexpr int kTaskRows = 6;  // step rows C_0 .. C_5 staged per warp: ctz(h) of 63 in 64 steps

struct WinDesc {
    const uint64_t* table;  // [66][W]: B_0..B_64 (zero-padded), z0
    uint64_t* out;          // [count][W]
    uint64_t offset, count;
    GroupPlan g;
    uint64_t task_base;  // tasks of earlier windows
    uint32_t W, ntasks;
};

constexpr int kWarpWords = stage_words<HLF_MAX_W>() + kTaskRows * HLF_MAX_W;  // shared words per warp

// Tasks [u, u1) of window d by one warp.
template <int W>
__device__ void many_tasks(const WinDesc& d, uint64_t u, uint64_t u1, int lane, uint64_t* stage)
{
    constexpr int M = Groups<W>::kLog2;
    const uint64_t* tab = d.table;
    auto row = [&](int k) { return tab + k * W; };
    auto ok = [&](uint64_t i, uint64_t len) { return HLF_RANGE_IN_BOUNDS(i - d.offset, len, d.count, kSiteManyStore); };
    const uint64_t ragged = ragged_shares(d.g);  // the first tasks
    for (; u < min(ragged, u1); ++u) store_ragged<W>(row, d.g, d.offset, u, d.out, lane, ok);
    if (u >= u1) return;
    u -= ragged;
    u1 -= ragged;
    const uint64_t h0 = d.g.h_first + u * task_groups(W);
    const uint64_t h1 = min(d.g.h_first + u1 * task_groups(W), d.g.h_end);
    if (h0 >= h1) return;
    uint64_t* C = stage + stage_words<HLF_MAX_W>();  // [kTaskRows][W]
    for (int e = lane; e < kTaskRows * W; e += 32)
        C[e] = __ldg(tab + (M - 1) * W + e % W) ^ __ldg(tab + M * W + e);
    uint64_t z[W];
    seed_group<W>(row, h0, lane, z);
    __syncwarp();
    uint64_t rare[W];  // a step row that is not staged
    store_groups<W>(
        z, h0, h1, d.g.phase, __ldg(tab), d.out - d.offset * W, stage, lane,
        [&](int j) -> const uint64_t* {
            if (j < kTaskRows) return C + j * W;
#pragma unroll
            for (int w = 0; w < W; ++w) rare[w] = __ldg(tab + (M - 1) * W + w) ^ __ldg(tab + (M + j) * W + w);
            return rare;
        },
        ok);
    __syncwarp();  // the staged rows are rewritten for the next window
}

__global__ void __launch_bounds__(kThreads, 2) many_kernel(const WinDesc* __restrict__ d, int k, uint64_t total_tasks,
                                                           uint64_t per_warp)
{
    extern __shared__ __align__(16) uint64_t s_stage[];  // [warps][kWarpWords]
    uint64_t* stage = s_stage + (threadIdx.x >> 5) * kWarpWords;
    const int lane = threadIdx.x & 31;
    uint64_t t = (((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * per_warp;
    const uint64_t t1 = min(t + per_warp, total_tasks);
    if (t >= t1) return;
    int lo = 0, hi = k - 1;  // last window with task_base <= t
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (d[mid].task_base <= t) lo = mid;
        else hi = mid - 1;
    }
    for (; t < t1; ++lo) {
        const WinDesc& w = d[lo];
        const uint64_t u = t - w.task_base;
        const uint64_t u1 = min(t1 - w.task_base, (uint64_t)w.ntasks);
        t = w.task_base + u1;
        switch (w.W) {
        case 1: many_tasks<1>(w, u, u1, lane, stage); break;
        case 2: many_tasks<2>(w, u, u1, lane, stage); break;
        case 3: many_tasks<3>(w, u, u1, lane, stage); break;
        case 4: many_tasks<4>(w, u, u1, lane, stage); break;
        case 5: many_tasks<5>(w, u, u1, lane, stage); break;
        case 6: many_tasks<6>(w, u, u1, lane, stage); break;
        case 7: many_tasks<7>(w, u, u1, lane, stage); break;
        case 8: many_tasks<8>(w, u, u1, lane, stage); break;
        case 9: many_tasks<9>(w, u, u1, lane, stage); break;
        case 10: many_tasks<10>(w, u, u1, lane, stage); break;
        case 11: many_tasks<11>(w, u, u1, lane, stage); break;
        case 12: many_tasks<12>(w, u, u1, lane, stage); break;
        case 13: many_tasks<13>(w, u, u1, lane, stage); break;
        case 14: many_tasks<14>(w, u, u1, lane, stage); break;
        case 15: many_tasks<15>(w, u, u1, lane, stage); break;
        default: many_tasks<16>(w, u, u1, lane, stage); break;
        }
    }
}

// Host-side cut of one window into tasks (outputs are 16-byte aligned, checked by
// the caller).
void plan_window(WinDesc& d, uint32_t W)
{
    const uint64_t G = W == 1 ? Groups<1>::kSize : Groups<2>::kSize;
    d.g = plan_groups(d.offset, d.count, G, W == 1 ? store_phase(d.out, d.offset) : 0);
    d.W = W;
    const uint64_t tg = task_groups(W);
    d.ntasks = (uint32_t)(ragged_shares(d.g) + (d.g.h_end - d.g.h_first + tg - 1) / tg);
}

}  // namespace

// The handle's enumeration table, rank and word count, and the record of a
// use of the handle on a stream (defined in hlf_api.cu).
hlf_status handle_enum_view(hlf_handle* h, const uint64_t** table, int32_t* r, int32_t* W);
hlf_status handle_record_use(hlf_handle* h, cudaStream_t s);

HLF_DEBUG_TAKE(many)

}  // namespace hlf

struct hlf_many {
    int device = 0;
    int32_t max_windows = 0;
    hlf::WinDesc* dev[2] = {nullptr, nullptr};
    hlf::WinDesc* host[2] = {nullptr, nullptr};  // pinned staging
    cudaEvent_t done[2] = {nullptr, nullptr};
    int next = 0;
};

extern "C" {

hlf_status hlf_many_create(int32_t max_windows, hlf_many** out)
{
    if (!out) return HLF_ERR_ARG;
    *out = nullptr;
    if (max_windows < 1 || max_windows > (1 << 22)) return HLF_ERR_ARG;
    if (hlf::take_injected_alloc_failure()) return HLF_ERR_NOMEM;
    hlf_many* m = new (std::nothrow) hlf_many;
    if (!m) return HLF_ERR_NOMEM;
    m->max_windows = max_windows;
    if (cudaGetDevice(&m->device) != cudaSuccess) {
        delete m;
        return HLF_ERR_CUDA;
    }
    const size_t bytes = sizeof(hlf::WinDesc) * (size_t)max_windows;
    for (int b = 0; b < 2; ++b) {
        if (cudaMalloc(&m->dev[b], bytes) != cudaSuccess || cudaMallocHost(&m->host[b], bytes) != cudaSuccess ||
            cudaEventCreateWithFlags(&m->done[b], cudaEventDisableTiming) != cudaSuccess) {
            cudaGetLastError();
            hlf_many_destroy(m);
            return HLF_ERR_NOMEM;
        }
    }
    *out = m;
    return HLF_OK;
}

hlf_status hlf_enumerate_store_many(hlf_many* m, hlf_handle* const* hs, const uint64_t* offsets,
                                    const uint64_t* counts, uint64_t* const* outs_dev, int32_t k, void* stream)
{
    hlf::NvtxRange nvtx_range("hlf_enumerate_store_many");
    if (!m || k < 0 || k > m->max_windows) return HLF_ERR_ARG;
    if (k == 0) return HLF_OK;
    if (!hs || !offsets || !counts || !outs_dev) return HLF_ERR_ARG;
    int cur = -1;
    if (cudaGetDevice(&cur) != cudaSuccess || cur != m->device) return HLF_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int b = m->next;
    if (cudaEventSynchronize(m->done[b]) != cudaSuccess) return HLF_ERR_CUDA;  // staging b is free again
    hlf::WinDesc* d = m->host[b];
    uint64_t tasks = 0;
    int32_t used = 0;
    for (int32_t j = 0; j < k; ++j) {
        if (!hs[j] || (counts[j] && !outs_dev[j])) return HLF_ERR_ARG;
        if (reinterpret_cast<uintptr_t>(outs_dev[j]) % 16) return HLF_ERR_ARG;
        const uint64_t* table = nullptr;
        int32_t r = 0, W = 0;
        hlf_status st = hlf::handle_enum_view(hs[j], &table, &r, &W);
        if (st != HLF_OK) return st;
        const uint64_t off = offsets[j], cnt = counts[j];
        const bool ok = r < 64 ? (off <= (1ull << r) && cnt <= (1ull << r) - off)
                               : (cnt == 0 || cnt - 1 <= ~0ull - off);
        if (!ok) return HLF_ERR_RANGE;
        if (cnt == 0) continue;
        hlf::WinDesc& w = d[used++];
        w = hlf::WinDesc{};
        w.table = table;
        w.out = outs_dev[j];
        w.offset = off;
        w.count = cnt;
        hlf::plan_window(w, (uint32_t)W);
        w.task_base = tasks;
        tasks += w.ntasks;
    }
    if (used == 0) return HLF_OK;
    if (cudaMemcpyAsync(m->dev[b], d, sizeof(hlf::WinDesc) * (size_t)used, cudaMemcpyHostToDevice, s) !=
        cudaSuccess)
        return HLF_ERR_CUDA;
    // Two CTAs per SM keep HBM busy for stores and leave room on every SM for
    // the factorisations a serving loop runs alongside.
    const uint64_t warps_cap = (uint64_t)hlf::sm_count() * 2 * (hlf::kThreads / 32);
    const uint64_t per_warp = (tasks + warps_cap - 1) / warps_cap;
    const uint64_t warps = (tasks + per_warp - 1) / per_warp;
    const unsigned blocks = (unsigned)((warps * 32 + hlf::kThreads - 1) / hlf::kThreads);
    constexpr size_t smem = (size_t)(hlf::kThreads / 32) * hlf::kWarpWords * sizeof(uint64_t);
    hlf::many_kernel<<<blocks, hlf::kThreads, smem, s>>>(m->dev[b], used, tasks, per_warp);
    if (cudaGetLastError() != cudaSuccess) return HLF_ERR_CUDA;
    if (cudaEventRecord(m->done[b], s) != cudaSuccess) return HLF_ERR_CUDA;
    // every handle read by this launch must outlive it (hlf_destroy waits)
    for (int32_t j = 0; j < k; ++j) {
        if (j > 0 && hs[j] == hs[j - 1]) continue;
        hlf_status st = hlf::handle_record_use(hs[j], s);
        if (st != HLF_OK) return st;
    }
    m->next = 1 - b;
    return HLF_OK;
}

hlf_status hlf_many_destroy(hlf_many* m)
{
    if (!m) return HLF_OK;
    hlf_status st = HLF_OK;
    for (int b = 0; b < 2; ++b) {
        if (m->done[b] && cudaEventSynchronize(m->done[b]) != cudaSuccess) st = HLF_ERR_CUDA;
        if (m->dev[b] && cudaFree(m->dev[b]) != cudaSuccess) st = HLF_ERR_CUDA;
        if (m->host[b] && cudaFreeHost(m->host[b]) != cudaSuccess) st = HLF_ERR_CUDA;
        if (m->done[b]) cudaEventDestroy(m->done[b]);
    }
    delete m;
    return st;
}

}  // extern "C"
