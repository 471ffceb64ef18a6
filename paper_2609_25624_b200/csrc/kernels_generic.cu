// The dispatch for shapes and buffers that TMA cannot read (K % 8 != 0 or FP32 weights with K % 4 != 0, misaligned buffers),
// the split-K second pass, the copy of small activations and results across the bus and the row argmax.
#include "internal.h"
#include "device_utils.cuh"
#include <cooperative_groups.h>

namespace detlin {

cudaError_t launch_decode_any_wf0(const LaunchArgs& a);        // decode_any.cu
cudaError_t launch_decode_any_wf1(const LaunchArgs& a);
cudaError_t launch_decode_any_wf2(const LaunchArgs& a);

// Split-K second pass (rule R3): the S partials of every output are added in ascending segment
// order by one thread, then the bias; no atomics anywhere.
__global__ void __launch_bounds__(256)
combine_kernel(const float* __restrict__ partials, const float* __restrict__ b, float* __restrict__ y,
               int64_t MN, int64_t N, int S, int64_t ldy)
{
    // programmatic dependent launch: the next kernel may start its prologue; the partials are read
    // only after the kernel that wrote them has completed
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= MN) return;
    float t = partials[i];
    for (int s = 1; s < S; ++s) t = __fadd_rn(t, partials[(int64_t)s * MN + i]);
    const int64_t m = i / N, n = i % N;
    y[m * ldy + n] = b ? __fadd_rn(t, b[n]) : t;
}

// Any shape, any alignment: the same orders, the same bits.
cudaError_t launch_generic(const LaunchArgs& a, int bucket)
{
    if (bucket != 0) return launch_prefill_plain(a);
    return a.wfmt == 1 ? launch_decode_any_wf1(a) : a.wfmt == 2 ? launch_decode_any_wf2(a) : launch_decode_any_wf0(a);
}

cudaError_t launch_combine(const LaunchArgs& a)
{
    const int64_t MN = a.M * a.N;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)((MN + 255) / 256));
    cfg.blockDim = dim3(256);
    cfg.stream = a.stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, combine_kernel, (const float*)a.partials, a.b, a.y, MN, a.N, a.S, a.ldy);
}

// Activations from pinned host memory to device memory, or results the other way: whole lines across the bus, all of them on their
// way at once, and the kernel after this one may start its prologue and its weight stream meanwhile.  Not before this kernel's own
// wait: W and b may have been written by the kernel before it.
__global__ void __launch_bounds__(256) copy_across_bus_kernel(const float4* __restrict__ src, float4* __restrict__ dst, unsigned n)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (unsigned i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) dst[i] = __ldcv(src + i);
}

cudaError_t launch_copy_across_bus(const void* src, void* dst, size_t bytes, cudaStream_t stream)
{
    const unsigned n = (unsigned)(bytes / 16), blocks = (n + 255) / 256;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    cfg.gridDim = dim3(blocks < 256 ? blocks : 256);
    cfg.blockDim = dim3(256);
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, copy_across_bus_kernel, static_cast<const float4*>(src), static_cast<float4*>(dst), n);
}

// Row argmax, lowest index on ties (the paper's stated tie rule for greedy decoding).  Ordering
// key: NaN beats everything (first NaN wins), otherwise larger value, then smaller index.
// Comparisons only, so the result is exact and order-free.  A cluster of kArgmaxCluster blocks
// shares one row: each block scans a contiguous slice, the partial results meet in block 0 of the
// cluster through distributed shared memory (hardware cluster barrier, no spinning).
namespace cg = cooperative_groups;
constexpr int kArgmaxCluster = 8;

// A value as an unsigned key with the order above: NaN on top, -0 = +0.  A pair (key, index) is better if its key is
// larger, or equal with a smaller index; as one 64-bit number with the index complemented, the better pair is the larger.
__device__ __forceinline__ uint32_t argmax_key(float v)
{
    if (v != v) return 0xffffffffu;
    const uint32_t u = __float_as_uint(__fadd_rn(v, 0.0f));      // -0 + +0 = +0
    return u ^ ((u >> 31) ? 0xffffffffu : 0x80000000u);
}
__device__ __forceinline__ unsigned long long argmax_warp(unsigned long long p)
{
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, p, d);
        p = o > p ? o : p;
    }
    return p;
}

// Bound by latency for the few rows of a decode step: a thread's whole share of a row (16-byte loads where the row starts
// aligned) is in flight at once.  M = 8, N = 128256: 14 -> 4 us.
__global__ void __cluster_dims__(kArgmaxCluster, 1, 1) __launch_bounds__(1024)
argmax_rows_kernel(const float* __restrict__ y, int64_t N, int32_t* __restrict__ idx)
{
    __shared__ unsigned long long warp_best[32];
    __shared__ unsigned long long block_best;
    // programmatic dependent launch: let the next kernel of the stream start its prologue now, and
    // wait for the kernel that produced y before reading it
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const float* row = y + (int64_t)blockIdx.y * N;
    uint32_t key = 0, at = 0xffffffffu;              // 0 < any value's key: an empty share loses
    auto look = [&](float v, uint32_t n) {           // a thread's elements come in ascending order
        const uint32_t k = argmax_key(v);
        if (k > key) { key = k; at = n; }
    };
    if ((reinterpret_cast<uintptr_t>(row) & 15u) == 0) {
        const uint32_t quads = (uint32_t)(N / 4), per = (quads + kArgmaxCluster - 1) / kArgmaxCluster;
        const uint32_t lo = rank * per, hi = min(lo + per, quads);
        const float4* r4 = reinterpret_cast<const float4*>(row);
        uint32_t i = lo + threadIdx.x;
        for (; i + 3 * 1024 < hi; i += 4 * 1024) {
            float4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = r4[i + 1024 * u];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t n = 4 * (i + 1024 * u);
                look(v[u].x, n); look(v[u].y, n + 1); look(v[u].z, n + 2); look(v[u].w, n + 3);
            }
        }
        float4 v[3];
#pragma unroll
        for (int u = 0; u < 3; ++u)
            if (i + 1024 * u < hi) v[u] = r4[i + 1024 * u];
#pragma unroll
        for (int u = 0; u < 3; ++u)
            if (i + 1024 * u < hi) {
                const uint32_t n = 4 * (i + 1024 * u);
                look(v[u].x, n); look(v[u].y, n + 1); look(v[u].z, n + 2); look(v[u].w, n + 3);
            }
        if (rank == kArgmaxCluster - 1 && threadIdx.x < (N & 3)) look(row[4ll * quads + threadIdx.x], 4 * quads + threadIdx.x);
    } else {
        const uint32_t per = (uint32_t)((N + kArgmaxCluster - 1) / kArgmaxCluster);
        const int64_t lo = (int64_t)rank * per, hi = (lo + per < N) ? lo + per : N;
#pragma unroll 4
        for (int64_t n = lo + threadIdx.x; n < hi; n += 1024) look(row[n], (uint32_t)n);
    }
    unsigned long long best = argmax_warp(((unsigned long long)key << 32) | (uint32_t)~at);
    if ((threadIdx.x & 31) == 0) warp_best[threadIdx.x >> 5] = best;
    __syncthreads();
    if (threadIdx.x < 32) {
        best = argmax_warp(warp_best[threadIdx.x]);
        if (threadIdx.x == 0) block_best = best;
    }
    cluster.sync();
    if (rank == 0 && threadIdx.x < 32) {
        best = argmax_warp(threadIdx.x < kArgmaxCluster ? *cluster.map_shared_rank(&block_best, threadIdx.x) : 0ull);
        if (threadIdx.x == 0) idx[blockIdx.y] = (int32_t)~(uint32_t)best;
    }
    cluster.sync();     // keep every block's shared memory alive until block 0 has read it
}

cudaError_t launch_argmax(const float* y, int64_t M, int64_t N, int32_t* idx, cudaStream_t stream)
{
    const int64_t max_rows = 65535;
    for (int64_t m0 = 0; m0 < M; m0 += max_rows) {
        const int64_t mm = (M - m0 < max_rows) ? M - m0 : max_rows;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(kArgmaxCluster, (unsigned)mm);
        cfg.blockDim = dim3(1024);
        cfg.dynamicSmemBytes = 0;
        cfg.stream = stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        cudaError_t e = cudaLaunchKernelEx(&cfg, argmax_rows_kernel, y + m0 * N, N, idx + m0);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace detlin
