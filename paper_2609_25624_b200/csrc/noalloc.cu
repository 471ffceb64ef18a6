// det_linear_run_noalloc: the linear layer for callers that must not allocate.
//
// Some hosts of this library cannot call cudaMalloc at the point where they need a linear layer:
// code running inside a memory pool or arena that owns all device memory, a plugin whose contract
// forbids allocation after initialisation, a latency-critical loop where an allocation (an implicit
// device synchronisation) is unacceptable.  The ordinary entry points allocate when a plan is
// created (status word, split-K partials).  This one allocates nothing, neither on the device nor
// on the host: the split-K partials live in a fixed array that is part of the library image.
//
// The paper has no counterpart for this entry point; it computes exactly the same thing (same
// order, same bits, same kernels) as det_linear_plan + det_linear_run.  M = 3, N = K = 4096 takes 8.4 us a call.
#include "internal.h"
#include "det_linear_test.h"
#include <mutex>

namespace detlin {

// Scratch for the split-K partials [S, M, N] (FP32).  Every GPU that loads the library holds these
// 4 MiB until the process exits.  All calls share the array.
constexpr size_t kNoallocScratchFloats = (size_t)1 << 20;
static __device__ __align__(256) float g_noalloc_scratch[kNoallocScratchFloats];

// Status word (first two words) and the schedule words that the prefill kernel expects beside it (all zero, not written
// here: they only matter to blocks that hand work over, which needs a workspace this entry point does not have).
static __device__ __align__(256) unsigned g_noalloc_words[64];

struct NoallocAddresses {
    float* scratch;
    unsigned* words;
};
static NoallocAddresses g_addr[kMaxDevices];    // device addresses of the arrays, per device
static std::mutex g_scratch_mutex;

// In host code the arrays are only handles for the runtime, not device addresses; the
// address a kernel can use has to be asked for, once per device, with that device current.
static cudaError_t static_addresses(int dev, NoallocAddresses* out)
{
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_scratch_mutex);
    if (!g_addr[dev].words) {
        void *p = nullptr, *q = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e == cudaSuccess) e = cudaGetSymbolAddress(&q, g_noalloc_words);
        if (e != cudaSuccess) return e;
        g_addr[dev].scratch = static_cast<float*>(p);
        g_addr[dev].words = static_cast<unsigned*>(q);
    }
    *out = g_addr[dev];
    return cudaSuccess;
}

// Bound of one device-side wait and test flag (det_test_noalloc_set_wait; never set outside the tests).
static unsigned long long g_wait_limit_ns = kDefaultWaitLimitNs;
static int g_test_flags = 0;

// The decode schedule depends on the shape and the device only: a loop that repeats its shapes searches once for each.  A search for a
// layout (any K, any alignment) takes 0.7 us of the host, one for a tiling more; sixteen entries hold the projections of a few
// kinds of layer at two batch sizes.
struct NoallocSchedule {
    int64_t M, N, K;                 // M = 0: empty
    int dev;
    bool tiled;                      // cfg is valid
    DecodeConfig cfg;
    AnyLayout layout;                // mt = 0: none yet
};
constexpr int kNoallocSchedules = 16;
static thread_local NoallocSchedule g_schedules[kNoallocSchedules];
static thread_local int g_next_schedule = 0;

static NoallocSchedule& schedule_of(int64_t M, int64_t N, int64_t K, int dev)
{
    for (NoallocSchedule& s : g_schedules)
        if (s.M == M && s.N == N && s.K == K && s.dev == dev) return s;
    NoallocSchedule& s = g_schedules[g_next_schedule];
    g_next_schedule = (g_next_schedule + 1) % kNoallocSchedules;
    s = NoallocSchedule{};
    s.M = M; s.N = N; s.K = K; s.dev = dev;
    return s;
}

}  // namespace detlin

using namespace detlin;

extern "C" det_status_t det_linear_run_noalloc(int64_t M, int64_t N, int64_t K, const float* x, const uint16_t* W,
                                               const float* b, float* y, void* stream)
{
    if (!x || !W || !y) { set_error("run_noalloc: x, W and y must not be NULL"); return DET_ERR_INVALID_ARG; }
    det_linear_params_t p;
    det_status_t st = fill_params(M, N, K, &p);
    if (st != DET_OK) return st;
    const uint64_t need = p.workspace_bytes / 4;            // split-K partials of the prefill bucket, in floats
    if (need > kNoallocScratchFloats) {
        set_error("run_noalloc: this shape splits K into %d segments and needs %llu bytes of partials; the built-in "
                  "scratch holds %llu bytes (use det_linear_plan + det_linear_run for larger problems)",
                  p.S, (unsigned long long)(need * 4), (unsigned long long)(kNoallocScratchFloats * 4));
        return DET_ERR_UNSUPPORTED_SHAPE;
    }
    int dev = 0, major = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) { set_error("run_noalloc: device query: %s", cudaGetErrorString(e)); return DET_ERR_CUDA; }
    if (major != 10) {
        set_error("run_noalloc: device %d is sm_%dx; this library is built for sm_100a only (no fallback)", dev, major);
        return DET_ERR_ARCH;
    }
    NoallocAddresses at{};
    e = static_addresses(dev, &at);
    if (e != cudaSuccess) {
        set_error("run_noalloc: cudaGetSymbolAddress failed: %s", cudaGetErrorString(e));
        return DET_ERR_CUDA;
    }
    // A plan on the stack, without memory of its own: the same kernels as det_linear_run.  No in-kernel fold of prefill
    // segments (its counters would be shared by calls of different shapes) and no stretches cut across blocks.
    det_linear_plan_t plan{};
    plan.prm = p;
    plan.device = dev;
    plan.sm_count = sms;
    plan.partials = need ? at.scratch : nullptr;            // every partial is written by the first pass before the
                                                            // second pass reads it: nothing has to start at zero
    plan.status = reinterpret_cast<DeviceStatus*>(at.words);
    plan.sync = at.words + 8;
    plan.n_count = N;
    plan.ldy = N;
    plan.forced_kernel = -1;
    plan.wait_limit_ns = g_wait_limit_ns;
    plan.test_flags = kFlagLateWeights | g_test_flags;                     // nothing was said here about W and b being older than the stream's last kernel
    plan.decode_cfg_variant = -1;
    plan.map_cfg_id = -1;
    if (p.bucket != 0) return run_device(&plan, x, W, b, y, static_cast<cudaStream_t>(stream));
    NoallocSchedule& s = schedule_of(M, N, K, dev);
    if (s.tiled) {
        plan.decode_cfg = s.cfg;
        plan.decode_cfg_variant = 0;
    }
    plan.any_layout = s.layout;
    st = run_device(&plan, x, W, b, y, static_cast<cudaStream_t>(stream));
    if (st == DET_OK) {
        s.tiled = plan.decode_cfg_variant == 0;
        s.cfg = plan.decode_cfg;
        s.layout = plan.any_layout;
    }
    return st;
}

extern "C" det_status_t det_linear_noalloc_check(void* stream)
{
    int dev = 0;
    NoallocAddresses at{};
    DeviceStatus h{};
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = static_addresses(dev, &at);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, at.words, sizeof h, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(at.words, 0, sizeof h, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) { set_error("noalloc_check: %s", cudaGetErrorString(e)); return DET_ERR_CUDA; }
    if (h.timeout_flag) {
        set_error("noalloc_check: a kernel gave up a bounded wait (site %u)", h.where);
        return DET_ERR_DEVICE_TIMEOUT;
    }
    return DET_OK;
}

extern "C" det_status_t det_test_noalloc_set_wait(uint64_t wait_limit_ns, int flags)
{
    if (wait_limit_ns == 0 || flags < 0 || flags > 1) { set_error("noalloc_set_wait: bad argument"); return DET_ERR_INVALID_ARG; }
    g_wait_limit_ns = wait_limit_ns;
    g_test_flags = flags;
    return DET_OK;
}
