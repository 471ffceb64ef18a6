// Launchers of the prefill kernel for one weight format (DET_WF = 0 BF16, 1 FP16, 2 FP32), fed by TMA or (DET_PLAIN = 1) by plain
// loads for any K and alignment, and every tile: heights 80, 96, 112 and 128, widths 256, 128, 64 and 32.  Compiled once
// per format and feed.
#include "prefill_tma_kernel.cuh"

namespace detlin {

namespace {

using namespace prefill_detail;

template <int WF, int TR, int TC, int LX, int LY, bool PLAIN>
cudaError_t launch_t(const LaunchArgs& la, const CUtensorMap* map_w, const CUtensorMap* map_x)
{
    typedef Tile<WF, TR, TC, LX, LY, PLAIN> T;
    static bool configured[kMaxDevices];             // function attributes belong to a device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    auto kern = prefill_tma_kernel<WF, TR, TC, LX, LY, PLAIN>;
    if (!configured[dev]) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, T::kSmemBytes);
        if (e != cudaSuccess) return e;
        configured[dev] = true;
    }
    const long long tiles_m = (la.M + T::BM - 1) / T::BM, tiles_n = (la.N + T::BN - 1) / T::BN;
    const long long units = tiles_m * tiles_n * la.S;
    if (units > 0x7fffffffLL) return cudaErrorInvalidValue;
    Args a{};
    a.x = la.x; a.w = la.W;
    a.bias = la.b; a.y = la.y; a.partials = la.partials; a.handoff = la.handoff; a.sync = la.sync;
    a.tile_counters = (uint64_t)units * T::BM * T::BN <= la.partial_floats ? la.tile_counters : nullptr;
    a.status = la.status;
    a.ldy = la.ldy;
    a.M = (int)la.M; a.N = (int)la.N; a.K = (int)la.K;
    a.seg_slabs = (int)(la.seg_len / BK);
    a.tile_slabs = (int)((la.K + BK - 1) / BK);
    a.S = la.S; a.tiles_m = (int)tiles_m;
    a.total = tiles_m * tiles_n * a.tile_slabs;
    a.wait_limit_ns = la.wait_limit_ns;
    a.test_flags = la.test_flags;
    // Equal stretches as soon as the units need more than one wave.  A unit may be cut once only, so a stretch is at least
    // a segment long.
    long long grid = units;
    if (units > la.sm_count && la.handoff) {
        a.cut = 1;
        const long long most = a.total / (a.seg_slabs < a.tile_slabs ? a.seg_slabs : a.tile_slabs);
        grid = most < la.sm_count ? most : la.sm_count;
    }
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(T::kThreads);
    cfg.dynamicSmemBytes = T::kSmemBytes;
    cfg.stream = la.stream;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const CUtensorMap none{};
    e = cudaLaunchKernelEx(&cfg, kern, PLAIN ? none : *map_x, PLAIN ? none : *map_w, a);
    if (e != cudaSuccess) return e;
    if (la.S > 1 && !a.tile_counters) return launch_combine(la);
    return cudaSuccess;
}

// tile height 16 TM
template <int WF, int TM>
cudaError_t launch_h(const LaunchArgs& a, int width, const CUtensorMap* map_w, const CUtensorMap* map_x)
{
    switch (width) {
    case 256: return launch_t<WF, 2 * TM, 8, 32, 8, DET_PLAIN>(a, map_w, map_x);
    case 128: return launch_t<WF, 8, 8, 16, 2 * TM, DET_PLAIN>(a, map_w, map_x);
    case 64: return launch_t<WF, 4, 8, 8, 4 * TM, DET_PLAIN>(a, map_w, map_x);
    case 32:
        // 128 rows: one multiplying warp a scheduler with 8 x 4 outputs a thread (three loads per 16 packed FMAs) beats two with 4 x 4
        // (two per 8): 128 x 1000 x 1000 13.45 -> 12.35 us, 120 x 700 x 512 12.4 -> 11.5.  At 96 rows three such warps lose as often
        // (96 x 1000 x 1000 11.85 -> 11.80, 90 x 64 x 4096 13.0 -> 14.2).
        if constexpr (TM == 8) return launch_t<WF, 8, 4, 8, 2 * TM, DET_PLAIN>(a, map_w, map_x);
        else return launch_t<WF, 4, 4, 8, 4 * TM, DET_PLAIN>(a, map_w, map_x);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

#define DET_CAT3(a, b, c) a##b##_##c
#define DET_PREFILL_NAME(wf, plain) DET_CAT3(launch_prefill_wf, wf, plain)
cudaError_t DET_PREFILL_NAME(DET_WF, DET_PLAIN)(const LaunchArgs& a, int tm, int width, const CUtensorMap* map_w, const CUtensorMap* map_x)
{
    switch (tm) {
    case 5: return launch_h<DET_WF, 5>(a, width, map_w, map_x);
    case 6: return launch_h<DET_WF, 6>(a, width, map_w, map_x);
    case 7: return launch_h<DET_WF, 7>(a, width, map_w, map_x);
    case 8: return launch_h<DET_WF, 8>(a, width, map_w, map_x);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace detlin
