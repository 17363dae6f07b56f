// Shared host-side helpers of the library: error reporting, argument checks, and the small
// per-process caches (device properties, environment switches) that keep repeated calls cheap.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "powerattn.h"

namespace pa {

// Records a message for pa_last_error_message() and returns `s`.
pa_status fail(pa_status s, const char *fmt, ...);
void clear_error();

inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

constexpr int kMaxDevices = 64;

// Properties of the current device, looked up once per device and process.
struct DeviceInfo {
    int device, sms, cc_major;
};
// PA_OK with *out filled in if the current device is an sm_100 part, else PA_ERR_UNSUPPORTED /
// PA_ERR_CUDA.
pa_status current_sm100_device(DeviceInfo *out);

// One-time per-device set-up steps (kernel attributes) are keyed by these slots.
enum DeviceOnce : int {
    ONCE_PREFILL_ATTR = 0,  // (40: order of the units, head_dim, slots, output type)
    ONCE_DECODE_ATTR = ONCE_PREFILL_ATTR + 40,
    ONCE_BACKWARD_ATTR, ONCE_BACKWARD_ATTR_64, ONCE_BACKWARD_TC_ATTR, ONCE_BACKWARD_TC_ATTR_64,
    ONCE_COUNT
};
std::mutex &device_once_mutex();
bool &device_once_done(int device, DeviceOnce slot);
// Performs the step, a cudaError_t(), once per (device, slot); a step that fails is tried again by the next call.
// Another thread's call goes on only when the step is done.
template <typename Step>
pa_status device_once(int device, DeviceOnce slot, Step step)
{
    std::lock_guard<std::mutex> lock(device_once_mutex());
    bool &done = device_once_done(device, slot);
    if (done) return PA_OK;
    const cudaError_t e = step();
    if (e != cudaSuccess) return fail(PA_ERR_CUDA, "cudaFuncSetAttribute failed: %s", cudaGetErrorString(e));
    done = true;
    return PA_OK;
}
inline cudaError_t first_error(cudaError_t a, cudaError_t b) { return a != cudaSuccess ? a : b; }

// Environment switches (for tests and measurements).  They are read when the library first needs
// them and again on pa_reload_environment().
struct EnvSwitches {
    int decode_path;     // PA_DECODE_PATH: 0 unset, 1 splitk, 2 cluster, 3 persistent
    int decode_cluster;  // PA_DECODE_CLUSTER=1..8 chunks per row, 0 = chosen from the problem size
    int decode_stages;   // PA_DECODE_STAGES=1..8, 0 = chosen from the problem size
    int decode_ctas_per_sm;  // PA_DECODE_CTAS_PER_SM=n: size of the persistent grid (default 2 per SM)
    int validate;        // PA_VALIDATE=1
    int backward_mma;    // PA_BACKWARD_PATH=mma: the warp-level MMA kernels
};
EnvSwitches env_switches();

// Limit of the kernels' bounded barrier waits in clock cycles as set by pa_set_wait_limit_cycles
// (0: each kernel's default).
long long wait_limit_cycles();

// Launch attribute under which a kernel may start while the kernel before it in the stream still runs
// (programmatic dependent launch).  Such a kernel touches no global memory before pdl_wait(), which returns when
// everything ahead of it in the stream has completed; what it does before that (barriers, tensor memory, the
// launch itself) is hidden behind the other kernel's last microseconds.  One kernel breaks that rule: dq_kernel works beside
// dkv_kernel, the launch before it.  That one lets it start only behind its own pdl_wait() and a store that dq_kernel
// acquires (so that the preparation's results are there), neither writes what the other reads or writes, and
// dq_kernel ends behind pdl_wait() (so that whoever waits for it waits for both).
// Behind it, plain loads only: __ldg and ld.global.nc are for data that nobody writes while the kernel runs, which here
// includes the time before the wait, and the compiler may move them across it.
inline cudaLaunchAttribute pdl_attribute()
{
    cudaLaunchAttribute a;
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = 1;
    return a;
}
template <typename... Params, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(Params...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr = pdl_attribute();
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
// The next kernel of the stream may be scheduled as soon as every block of this one has said so or ended.
__device__ __forceinline__ void pdl_launch_next() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
#endif

#define PA_CUDA_OK(expr)                                                                    \
    do {                                                                                    \
        cudaError_t e_ = (expr);                                                            \
        if (e_ != cudaSuccess)                                                              \
            return ::pa::fail(PA_ERR_CUDA, "%s failed: %s", #expr, cudaGetErrorString(e_)); \
    } while (0)

}  // namespace pa
