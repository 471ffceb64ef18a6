// Decode kernel dispatch: picks one of the compiled tilings for a shape.  The choice only changes
// the schedule (tile sizes, warp counts and ring depth are numerically inert: supplement C on
// rule R2), so it may read the SM count and the occupancy; the reduction order never does.
#include <cmath>

#include "decode_kernel.cuh"

namespace detlin {

namespace {

using decode_detail::DecodeEntry;

#define DET_TABLE_ROW(wf)                                                                                  \
    { &DET_TABLE_NAME(0, wf), &DET_TABLE_NAME(1, wf), &DET_TABLE_NAME(2, wf), &DET_TABLE_NAME(3, wf), \
      &DET_TABLE_NAME(4, wf), &DET_TABLE_NAME(5, wf) }

const DecodeClassTable* class_table(int wfmt, int cls)
{
    static const DecodeClassTable* const t[3][6] = {DET_TABLE_ROW(0), DET_TABLE_ROW(1), DET_TABLE_ROW(2)};
    return t[wfmt][cls];
}

int m_class(int64_t M) { return M <= 1 ? 0 : M <= 2 ? 1 : M <= 4 ? 2 : M <= 8 ? 3 : M <= 16 ? 4 : 5; }

// Predicted time of a tiling in SM clock cycles (schedule heuristic).  A work unit streams rb weight rows (at the SM's share of the
// HBM rate) and performs rb * mb * K multiply-adds at the FMA rate of an SM times an efficiency that depends on the warp tile;
// whichever is larger binds.  Units resident on one SM share it.  Fewer than eight consumer warps per SM hide latency badly; every
// unit pays for its lane trees (one per segment) and, with several segment groups, for the fold through shared memory.
// The rates were fitted to sweeps of every tiling on a 148-SM B200.
//   * 16-bit weights, up to 8 rows: the Llama-3-8B shapes, mean loss against the best tiling 0.5 %.
//   * 16-bit weights, more rows, K from 2560 on: 56 drawn and layer shapes, 9 to 64 rows, mean loss 2 % (3.5 % with the rates of few
//     rows: M = 16, N = 4096, K = 14336 44.5 -> 41.6 us, M = 16, N = 2083, K = 14096 49.8 -> 42.6).  Shorter rows are a matter of
//     latencies that these rates do not know (M = 16, N = 278, K = 2168 5.6 us, with the rates of few rows 4.8).
//   * FP32 weights, segments of more than two chunks: 52 shapes at batch 1 .. 64, 2 % (24 % with the rates of few rows).  Shorter ones
//     only in one wave of units of two chunks (M = 16, N = 1478, K = 440 3.8 us, by the rates of few rows 4.5) or in more than seven (M = 44, N =
//     22508, K = 264 38.7 and 44.6); between them the rates of few rows are better (M = 10, N = 3225, K = 368 4.6 us, otherwise 5.4).
// The last two only where the rates of few rows choose a tiling with more units than two thirds (16 bits) or half (FP32) of the SMs.
// With fewer, a block's rows and ring decide, not rates: M = 12, N = 99, K = 5832 (16 units) 8.1 us, by the rates of many rows 10.8; M = 35, N =
// 205, K = 5744 (75) 8.3 and 10.9; but M = 10, N = 871, K = 7248 (126) 14.4 and 13.3.  M = 4, N = 97, K = 8552 with FP32 weights (7) 11.4 and
// 14.9, but M = 7, N = 1081, K = 4112 (78) 13.2 and 11.3, M = 36, N = 388, K = 8976 (140) 26.4 and 21.1.
// Of 195 shapes of 16-bit weights none is then slower by more than 1.5 % than by the rates of many rows, of 144 of FP32 weights in long
// segments none by more than 2.5 %.
struct TilingRates {
    double eff8, eff4, eff2, eff1;       // share of the FMA rate by batch rows of a warp tile
    double wide, narrow;                 // ... times: 8-row tiles with half as many stage boundaries (KC 512); stages of 128
    double small8, small4;               // ... times: blocks of at most four consumer warps
    double hbm;                          // bytes per clock and SM (FP32 weights by the rates of 16 bits: twice as many)
    double other;                        // share of the term that does not bind
    double latency;                      // exponent of 8 / warps
    double tree, fold;                   // cycles per segment of a full tile; with several segment groups
    double part, part_exp;               // a last tile of the share p of a tile's rows takes part * p ^ part_exp of its time
};
constexpr TilingRates kRatesFewRows = {0.707, 0.70, 0.345, 0.2, 1.2, 0.9, 1.0, 1.0, 22.5, 0.0, 1.0, 1020.0, 1500.0, 1.08, 1.0};
constexpr TilingRates kRatesManyRows = {0.922, 0.844, 0.420, 0.141, 1.057, 0.9, 0.96, 0.973, 27.0, 0.0264, 1.703, 799.0, 1384.0, 0.7355, 0.567};
constexpr TilingRates kRatesFp32Short = {0.707, 0.70, 0.345, 0.2, 1.2, 0.9, 1.0, 1.0, 45.0, 0.0, 1.0, 1020.0, 1500.0, 1.08, 1.0};
constexpr TilingRates kRatesFp32 = {0.52, 0.43, 0.49, 0.075, 1.0, 1.0, 0.904, 0.558, 32.0, 0.0, 1.0, 1020.0, 1500.0, 1.08, 1.0};

int64_t tiling_units(const DecodeConfig& c, int64_t M, int64_t N)
{
    const int64_t rb = (int64_t)c.rt * c.wr, mb = (int64_t)c.mt * c.wm;
    return ((N + rb - 1) / rb) * ((M + mb - 1) / mb);
}

double tiling_cost(const DecodeEntry& e, const TilingRates& t, int wfmt, int64_t M, int64_t N, int64_t K, int S, int sm_count)
{
    const DecodeConfig& c = e.cfg;
    const int occ = e.occupancy(S);
    if (occ <= 0) return 1e300;
    const int64_t rb = (int64_t)c.rt * c.wr, mb = (int64_t)c.mt * c.wm;
    const int64_t mblocks = (M + mb - 1) / mb;
    const int64_t units = tiling_units(c, M, N);
    const int64_t rounds = (units + (int64_t)sm_count * occ - 1) / ((int64_t)sm_count * occ);
    const int64_t per_sm = (units + sm_count - 1) / sm_count;
    const double resident = (double)(per_sm < occ ? per_sm : occ);
    const double warps = resident * c.wm * c.wr * c.sk;
    const bool small = c.wm * c.wr * c.sk <= 4;
    double eff = c.mt >= 8 ? t.eff8 : c.mt == 4 ? t.eff4 : c.mt == 2 ? t.eff2 : t.eff1;
    if (c.kc >= 512 && c.mt >= 8) eff *= t.wide;
    if (c.kc <= 128) eff *= t.narrow;
    if (small && c.mt >= 8) eff *= t.small8;
    if (small && c.mt == 4) eff *= t.small4;
    const double latency = warps >= 8.0 ? 1.0 : pow(8.0 / warps, t.latency);
    const double fma = (double)rb * (double)mb * (double)K / 128.0 / eff * resident;
    // weights from HBM; the unit's activations come again from L2 for every unit
    const double row_bytes = (double)K * (wfmt == DET_WEIGHT_FP32 ? 4.0 : 2.0);
    const double hbm = ((double)rb * row_bytes / t.hbm + 0.06 * (double)mb * (double)K * 4.0 / 64.0) * resident;
    const double body = ((fma > hbm ? fma : hbm) + t.other * (fma > hbm ? hbm : fma)) * latency;
    const double overhead = (double)S * t.tree * ((double)(mb * rb) / 896.0) + (c.sk > 1 ? t.fold : 0.0);
    if ((rb >= 56 && mb >= 16) || rb >= 112) {
        // what is left after whole rounds is dealt out by row groups (Cfg::kDealRest); part of a tile takes longer than its
        // share of the time (one warp per scheduler)
        int64_t shares = (int64_t)sm_count * occ / mblocks;
        const int64_t groups = (N + c.rt - 1) / c.rt;
        shares = shares < 1 ? 1 : shares > groups ? groups : shares;
        const int64_t whole = groups / (shares * c.wr), rest = groups - whole * shares * c.wr;
        const double part = (double)((rest + shares - 1) / shares) / c.wr;
        // Tiles of 112 rows only from five rounds of a batch block's shares on (8 rows share all SMs, 24 a third of them).  us, by 112 rows
        // and by the better one of 28 and 56: M = 8, N = 28672, K = 4096 (1.7 rounds) 50.5 and 50.1; M = 8, N = 33152, K = 2048 (2) 27.9 and
        // 27.5; M = 7, N = 50000 (3.02) 45.9 and 44.1; M = 8, N = 58016, K = 4096 (3.5) 93.0 and 83.6; M = 8, N = 66304 FP16 (4) 53.4 and
        // 57.9; M = 8, N = 74592, K = 4096 (4.5) 110 and 106; M = 8, N = 82884 FP16 (5) 70.8 and 75.8; M = 5, N = 132608 (8) 99.5 and
        // 98.8; N = 128256, K = 4096 (7.7) 181.4 and 184.8.  More rows: M = 24, N = 28672, K = 4096 (5.2) 127 and 122, M = 20 with FP16 134
        // and 135; M = 40 (8.8) 200 and 202, with FP16 213 and 223; M = 24, N = 50000, K = 2560 (9.1) 138 and 135; M = 36, N = 40000 (12)
        // 181 and 179.
        if (rb >= 112 && whole < 5) return 1e300;
        if (whole > 0) return (double)whole * (body + overhead) + (part < 1.0 ? t.part * pow(part, t.part_exp) : 1.0) * body + (rest ? overhead : 0.0);
    }
    return (double)rounds * (body + overhead);
}

// Tilings that can serve batch size M: those of M's own class and, for M > 8, the 8-row tilings
// (the batch is then walked in blocks of 8 rows that run side by side).
int candidate_classes(int64_t M, int* out)
{
    const int cls = m_class(M);
    int n = 0;
    out[n++] = cls;
    if (cls > 3) out[n++] = 3;
    return n;
}

}  // namespace

int decode_num_variants()
{
    int n = 0;
    for (int c = 0; c < 6; ++c) n = class_table(0, c)->count > n ? class_table(0, c)->count : n;
    return n;
}

// variant 0 = automatic; variant v >= 1 = the v-th tiling, among those that can run the shape, for this
// batch size (own class first, then the 8-row tilings when M > 8).  A tiling whose segment groups do
// not divide S, or that does not fit the device, cannot run the shape and is not counted.
bool decode_config_for(int64_t M, int64_t N, int64_t K, int S, int wfmt, int variant, DecodeConfig* out)
{
    int classes[2];
    const int n_classes = candidate_classes(M, classes);
    if (variant < 0 || S < 1 || S > kDecodeMaxSegments) return false;
    int sms = 148;
    if (variant == 0) {
        count_schedule_search();
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
            sms = 148;
    }
    int pick_cls = classes[0], pick = -1;
    auto choose = [&](const TilingRates& t) {
        double best = 1e299;
        for (int ci = 0; ci < n_classes; ++ci) {
            const DecodeClassTable* tab = class_table(wfmt, classes[ci]);
            for (int i = 0; i < tab->count; ++i) {
                const double c = tiling_cost(tab->entries[i], t, wfmt, M, N, K, S, sms);
                if (c < best) { best = c; pick_cls = classes[ci]; pick = i; }
            }
        }
    };
    if (variant == 0) {
        const bool fp32 = wfmt == DET_WEIGHT_FP32;
        choose(fp32 ? kRatesFp32Short : kRatesFewRows);
        if (pick >= 0) {
            const int64_t units = tiling_units(class_table(wfmt, pick_cls)->entries[pick].cfg, M, N), seg = decode_segment(K, S);
            if (!fp32) {
                if (M > 8 && K >= 2560 && 3 * units > 2 * sms) choose(kRatesManyRows);
            } else if ((seg > 256 && units > sms / 2) || (seg == 256 && units > sms / 2 && units <= sms) || units > 7 * sms) {
                choose(kRatesFp32);
            }
        }
    } else {
        int seen = 0;
        for (int ci = 0; ci < n_classes && pick < 0; ++ci) {
            const DecodeClassTable* tab = class_table(wfmt, classes[ci]);
            for (int i = 0; i < tab->count && pick < 0; ++i)
                if (tab->entries[i].occupancy(S) > 0 && ++seen == variant) { pick_cls = classes[ci]; pick = i; }
        }
    }
    if (pick < 0) return false;
    *out = class_table(wfmt, pick_cls)->entries[pick].cfg;
    out->id = pick_cls * 64 + pick;
    return true;
}

int decode_config_occupancy(int wfmt, const DecodeConfig& cfg, int S)
{
    return class_table(wfmt, cfg.id / 64)->entries[cfg.id % 64].occupancy(S);
}

cudaError_t launch_decode(const LaunchArgs& a, const DecodeConfig& cfg, const CUtensorMap* map_w, const CUtensorMap* map_g, const CUtensorMap* map_x)
{
    return class_table(a.wfmt, cfg.id / 64)->entries[cfg.id % 64].fn(a, map_w, map_g, map_x);
}

}  // namespace detlin
