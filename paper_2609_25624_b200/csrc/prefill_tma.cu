// Dispatch of the TMA-fed prefill kernel (prefill_tma_kernel.cuh): tile width, workspace sizes, weight format.
#include "internal.h"

namespace detlin {

#define DET_DECLARE(wf) \
    cudaError_t launch_prefill_wf##wf##_0(const LaunchArgs& a, int tm, int width, const CUtensorMap* map_w, const CUtensorMap* map_x); \
    cudaError_t launch_prefill_wf##wf##_1(const LaunchArgs& a, int tm, int width, const CUtensorMap* map_w, const CUtensorMap* map_x);
DET_DECLARE(0)
DET_DECLARE(1)
DET_DECLARE(2)

// Tile width (schedule only: every width gives the same bits).  Wide tiles multiply fastest, narrow ones make more units:
// with more units than SMs the work is dealt out in equal stretches and the width's rate decides, with fewer the call
// takes as long as one unit.  A block of the three narrow widths has 16 tm / 16 = 5 .. 8 multiplying warps on four
// schedulers, so it takes as long as one of 128 rows whatever its height; the wide tile always has eight.  128 rows by 32 columns
// are the exception: four warps of 8 x 4 outputs a thread, 5 to 9 % faster than eight of 4 x 4.
// Rates = share of the FP32 peak, measured at M = 512, N = 28672, K = 4096: 86.6, 82.2, 63.4 and 50.0 % (128 rows by 32 columns 56.7 %).
// One or two cut units a block do not reach them: the hand-over costs 32 columns of 128 rows more than the rate gains, us at widths 64 /
// 32, K = 1024, M = 128: N = 1216 (152 units of 32 columns) 18.2 / 15.4, 1400 (176) 18.4 / 17.2, 1600 (200) 18.4 / 18.5, 1800 (228) 18.3 /
// 20.7; 0.42 puts the line at 198 units.  Either side of the
// line, us at widths 256 / 128 / 64 / 32: M = 128, N = 4096, K = 14336 (128 units of 256 columns on 148 SMs, or 256 of
// 128) 279 / 253 / 321 / 401; M = 96 likewise (tile height 96) 212 / 248 / 269 / 323; 100 x 1000 x 1000 with FP32 weights
// 44 / 27 / 18 / 13; M = 66, N = 300, K = 1000 31 / 26 / 16 / 11.
int prefill_tile_width(int64_t M, int64_t N, int64_t K, int S, int64_t seg_len, int tm, int sm_count)
{
    static const int widths[4] = {256, 128, 64, 32};
    static const double rates[4] = {0.88, 0.83, 0.63, 0.50};
    const int64_t bm = 16 * tm, tiles_m = (M + bm - 1) / bm;
    const int64_t seg = seg_len < K ? seg_len : K;
    int best = 256;
    double best_cost = 0.0;
    for (int i = 0; i < 4; ++i) {
        const int64_t tiles = tiles_m * ((N + widths[i] - 1) / widths[i]), units = tiles * S;
        const double k = units > sm_count ? (double)(tiles * K) / sm_count : (double)seg;       // k steps of the longest block
        const double rate = i == 3 && tm == 8 && units > sm_count ? 0.42 : rates[i];
        const double cost = k * (double)((i == 0 ? bm : 128) * widths[i]) / rate;
        if (i == 0 || cost < best_cost) { best = widths[i]; best_cost = cost; }
    }
    return best;
}

PrefillWorkspace prefill_workspace(int64_t M, int64_t N, int64_t K, int S, int64_t seg_len, int sm_count)
{
    PrefillWorkspace w{};
    const int tm = prefill_rows_per_thread(M);
    const int width = prefill_tile_width(M, N, K, S, seg_len, tm, sm_count);
    const uint64_t bm = 16 * (uint64_t)tm;
    const uint64_t units = ((uint64_t)M + bm - 1) / bm * (((uint64_t)N + width - 1) / width) * (uint64_t)S;
    w.sync_words = 8 + 8 * (uint64_t)sm_count;
    if (units > (uint64_t)sm_count) w.handoff_floats = (uint64_t)sm_count * 128 * 256;
    if (S > 1) {
        // any tile height and width (tests force them): tiles of at least 80 x 32, eight warps each
        w.counter_words = ((uint64_t)M + 79) / 80 * (((uint64_t)N + 31) / 32) * 8;
        // Segment sums by whole tiles, for the fold in place, where that is a matter of 16 MiB for any tile or of twice the sums
        // themselves for this one; layers of a few columns would pay many times over (64 000 x 1 x 2000: 131 MB for 0.5) and take a second pass.
        const uint64_t sums = (uint64_t)S * (uint64_t)M * (uint64_t)N, own = units * bm * (uint64_t)width;
        const uint64_t any = (uint64_t)S * ((uint64_t)M + 127) * (((uint64_t)N + 255) / 256 * 256);
        w.partial_floats = any <= (4u << 20) ? any : own <= 2 * sums ? own : sums;
    }
    return w;
}

cudaError_t launch_prefill_tma(const LaunchArgs& a, int tm, int width, const CUtensorMap* map_w, const CUtensorMap* map_x)
{
    if (!a.status || !a.sync) return cudaErrorInvalidValue;
    switch (a.wfmt) {
    case DET_WEIGHT_BF16: return launch_prefill_wf0_0(a, tm, width, map_w, map_x);
    case DET_WEIGHT_FP16: return launch_prefill_wf1_0(a, tm, width, map_w, map_x);
    case DET_WEIGHT_FP32: return launch_prefill_wf2_0(a, tm, width, map_w, map_x);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_prefill_plain(const LaunchArgs& a)
{
    if (!a.status) return cudaErrorInvalidValue;
    const int64_t most = (int64_t)1 << 30;           // rows are counted in 32 bits; no memory holds that many of several segments
    if (a.M > most) {
        if (a.S > 1) return cudaErrorInvalidValue;
        for (int64_t m = 0; m < a.M; m += most) {
            LaunchArgs part = a;
            part.x += m * a.K;
            part.y += m * a.ldy;
            part.M = a.M - m < most ? a.M - m : most;
            const cudaError_t e = launch_prefill_plain(part);
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    }
    const int tm = prefill_rows_per_thread(a.M);
    const int width = prefill_tile_width(a.M, a.N, a.K, a.S, a.seg_len, tm, a.sm_count);
    switch (a.wfmt) {
    case DET_WEIGHT_BF16: return launch_prefill_wf0_1(a, tm, width, nullptr, nullptr);
    case DET_WEIGHT_FP16: return launch_prefill_wf1_1(a, tm, width, nullptr, nullptr);
    case DET_WEIGHT_FP32: return launch_prefill_wf2_1(a, tm, width, nullptr, nullptr);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace detlin
