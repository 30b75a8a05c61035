// flame_launch.cuh -- what every launcher shares: device limits, occupancy,
// launches with an L2 window or programmatic dependence.
#pragma once

#include <cstdlib>
#include <cstring>
#include <mutex>
#include <set>
#include <utility>

#include "flame_internal.h"

namespace flame {

constexpr size_t kSmemBudget = 200 * 1024;  // what one CTA may take here
constexpr int kThreadsTarget = 256;
constexpr int kMaxThreads = 256;  // launch bound of every line-FFT kernel

static int sm_count() {
    static int n = 0;
    if (n == 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            n = 148;
    }
    return n;
}

// Raises a kernel's dynamic shared-memory limit to the device's opt-in
// maximum (less its static shared memory), once per kernel and device,
// before its first launch.
static cudaError_t opt_in(const void *kernel) {
    static std::mutex mu;
    static std::set<std::pair<const void *, int>> done;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(mu);
    if (done.count({kernel, dev})) return cudaSuccess;
    int optin = 0;
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa;
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kernel);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
    if (e == cudaSuccess) done.insert({kernel, dev});
    return e;
}

// CTAs of one kernel resident at once on the current device: a tile that
// starts now is followed, one wave later, by tile + resident_ctas.
static int resident_ctas(const void *kernel, const Geom &g) {
    if (opt_in(kernel) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    const int nsm = sm_count();
    int per = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, g.threads, g.smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return per * nsm;
}

// Launch with, when w.bytes > 0, an L2 persisting access window over [w.base, w.base + w.bytes) (a fraction w.hit of its
// accesses persisting, the rest streaming).
// With pdl, the launch is a programmatic dependent launch: its CTAs may be
// scheduled while the previous kernel on the stream drains, and wait in
// hardware (griddepcontrol.wait, the first statement of every step pass's
// body) until that kernel has completed and its memory is visible.  Only
// kernels whose bodies begin with that wait are launched so: the step's and the
// adjoint's passes in FP32, and in FP64 for columns of up to 96 points (N1 <=
// 128); in FP32 also a 2-D transform's second pass and passes A and B of a step
// with its area.  Per step (graph):
// FP32 256x512 9.5 -> 8.1 us, 1024x2048 18.1 -> 17.0, 4096x8192 level; FP64
// 128x256 23.5 -> 22.1, but 512x1024 77.4 -> 83.5: the early CTAs land where
// SMs drain first, and longer FP64 passes are bound by their fullest SM.
// Not for ensembles (96 flames: 7.2 against 7.7 ms with it): their launches fill
// the GPU many times over.  FLAME_PDL=0 or 1: none or all of the others.
static bool pdl_on(bool fp64, const StepArgs &a) {
    const char *v = getenv("FLAME_PDL");
    if (v && (strcmp(v, "0") == 0 || strcmp(v, "1") == 0)) return v[0] == '1';
    return !fp64 || a.la <= 5;
}
template <class... KArgs, class... Args>
static cudaError_t launch_x(const L2Window &w, bool pdl, void (*kernel)(KArgs...), dim3 grid, int threads,
                            size_t smem, cudaStream_t s, Args... args) {
    const cudaError_t oe = opt_in((const void *)kernel);
    if (oe != cudaSuccess) return oe;
    if (w.bytes == 0 && !pdl) {
        kernel<<<grid, threads, smem, s>>>(args...);
        return cudaGetLastError();
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    unsigned n = 0;
    if (pdl) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    if (w.bytes > 0) {
        attr[n].id = cudaLaunchAttributeAccessPolicyWindow;
        attr[n].val.accessPolicyWindow.base_ptr = const_cast<void *>(w.base);
        attr[n].val.accessPolicyWindow.num_bytes = w.bytes;
        attr[n].val.accessPolicyWindow.hitRatio = w.hit;
        attr[n].val.accessPolicyWindow.hitProp = cudaAccessPropertyPersisting;
        attr[n].val.accessPolicyWindow.missProp = cudaAccessPropertyStreaming;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}
template <class... KArgs, class... Args>
static cudaError_t launch_w(const L2Window &w, void (*kernel)(KArgs...), dim3 grid, int threads, size_t smem,
                            cudaStream_t s, Args... args) {
    return launch_x(w, false, kernel, grid, threads, smem, s, args...);
}
// a step pass: L2 window and programmatic dependent launch
template <class... KArgs, class... Args>
static cudaError_t launch_s(const L2Window &w, bool pdl, void (*kernel)(KArgs...), dim3 grid, int threads, size_t smem,
                            cudaStream_t s, Args... args) {
    return launch_x(w, pdl, kernel, grid, threads, smem, s, args...);
}
template <class... KArgs, class... Args>
static cudaError_t launch_k(void (*kernel)(KArgs...), dim3 grid, int threads, size_t smem, cudaStream_t s,
                             Args... args) {
    return launch_w(L2Window{nullptr, 0, 0.f}, kernel, grid, threads, smem, s, args...);
}
// Whether pass C needs its general epilogue (a two-stage scheme's stage,
// forcing or the per-step record) or the plain Euler one.
static bool general_epilogue(const FlameDesc &d) {
    return d.stage != kStageEuler || d.forcing != nullptr || d.forcing0 != 0.0 || d.rec != nullptr;
}

}  // namespace flame
