// Shared host/device helpers of the janus kernels (status words, format decode, small scans).
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <stdint.h>

#include <atomic>
#include <mutex>

#include "../../include/janus.h"

namespace janus {

// ---- host-side error bookkeeping -------------------------------------------------------------
void set_last_cuda_error(cudaError_t e);

#define JANUS_CUDA_CHECK(expr)                         \
    do {                                               \
        cudaError_t _e = (expr);                       \
        if (_e != cudaSuccess) {                       \
            janus::set_last_cuda_error(_e);            \
            return JANUS_ERR_CUDA;                     \
        }                                              \
    } while (0)

// Id of the CUDA context that is current on this thread; 0 while there is none (the runtime makes one on its first call that needs it).
uint64_t current_context_id();

// Runs a function once in every context: kernel attributes belong to a context (a device may have several, one after the other or
// side by side) and setting them on each call costs a microsecond.  Callers on other threads wait until it has run.
class once_per_context {
  public:
    template <class F>
    cudaError_t run(F&& f) { return run_in(current_context_id(), f); }
    template <class F>
    cudaError_t run_in(uint64_t id, F&& f) {
        if (seen(id)) return cudaSuccess;
        std::lock_guard<std::mutex> lock(mu_);
        if (seen(id)) return cudaSuccess;
        const cudaError_t e = f();
        if (e != cudaSuccess || id == 0) return e;
        for (auto& d : done_) {
            if (d.load(std::memory_order_relaxed) != 0) continue;
            d.store(id, std::memory_order_release);
            break;
        }
        return e;      // (with more contexts than places the function runs on each call)
    }

  private:
    bool seen(uint64_t id) const {
        for (const auto& d : done_) {
            const uint64_t v = d.load(std::memory_order_acquire);
            if (v == 0) return false;
            if (v == id) return true;
        }
        return false;
    }
    std::atomic<uint64_t> done_[32] = {};
    std::mutex mu_;
};

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// ---- launches that overlap the end of the kernel before them -----------------------------------------------------------------
// Every kernel here is launched as a programmatic dependent of its predecessor in the stream: its CTAs may become resident, and
// run up to grid_wait(), while the predecessor still runs.  The order of memory accesses stays that of the stream, because every
// kernel waits, on every path, before its first access to global memory; grid_wait() returns when the predecessor has completed
// and its writes are visible, and the predecessor has itself waited for what came before.  Tensor memory is allocated after
// grid_wait(), so that no CTA holds it while it waits.  Inputs are read with ordinary loads (ld_input, __ldcg, __ldcs, asynchronous
// copies), never with read-only ones (__ldg, ld.global.nc, or const __restrict__ parameters, which the compiler may turn into them): those
// require memory that nobody writes while the kernel exists, and it exists while its predecessor still writes.  A short kernel lets its successor in at once with grid_launch_next(); the
// indexer and the attention of many tokens do not, because CTAs that wait beside them made them 1 % slower.  One-session decode step
// 51.2 -> 44.2 us, short message 59.9 -> 52.8, sharded prediction 1.70 -> 1.66 ms; the large passes are unchanged.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class T>
__device__ __forceinline__ T ld_input(const T* p) { return __ldca(p); }

template <class Kernel, class... Args>
inline cudaError_t launch_kernel(Kernel kernel, dim3 grid, int threads, size_t smem, cudaStream_t stream, int cluster, const Args&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// ---- device-side status word: first error wins ------------------------------------------------
__device__ __forceinline__ void report(int32_t* dev_status, int code) {
    if (dev_status != nullptr) atomicCAS(dev_status, 0, code);
}

// ---- storage formats ----------------------------------------------------------------------------
__device__ __forceinline__ float bf16_bits_to_float(uint16_t b) { return __uint_as_float(static_cast<uint32_t>(b) << 16); }

__device__ __forceinline__ float e4m3_to_float(uint8_t c) {
    __half_raw h = __nv_cvt_fp8_to_halfraw(static_cast<__nv_fp8_storage_t>(c), __NV_E4M3);
    return __half2float(__half(h));
}

// fp32 -> key whose unsigned order is the float order (larger float, larger key)
__device__ __forceinline__ uint32_t float_to_key(float x) {
    uint32_t u = __float_as_uint(x);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_to_float(uint32_t k) {
    uint32_t u = (k & 0x80000000u) ? (k & 0x7fffffffu) : ~k;
    return __uint_as_float(u);
}

// ---- block-wide exclusive scan of one int per thread (THREADS a multiple of 32, <= 1024) ---------
// `warp_sums` is shared scratch of at least 33 ints.  Returns the exclusive prefix; *total = block sum.
template <int THREADS>
__device__ __forceinline__ int block_exclusive_scan(int v, int* warp_sums, int* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
    }
    __syncthreads();  // protect warp_sums from a previous use
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int s = (lane < THREADS / 32) ? warp_sums[lane] : 0;
        int si = s;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, si, d);
            if (lane >= d) si += y;
        }
        if (lane < THREADS / 32) warp_sums[lane] = si - s;  // exclusive offset of each warp
        if (lane == 31) warp_sums[32] = si;                  // block total
    }
    __syncthreads();
    *total = warp_sums[32];
    return warp_sums[warp] + incl - v;
}

}  // namespace janus
