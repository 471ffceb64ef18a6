// How a decode call for any K is laid out over the SMs (schedule only: every layout gives the same bits).  Host arithmetic.
#include "internal.h"

namespace detlin {

AnyGrid any_grid(const AnyLayout& l, int64_t M, int64_t N, int64_t K, int sms)
{
    // Two blocks of 8 warps per SM, or one of 16 where only that keeps all activations of a batch block in shared memory; the
    // window holds whole chunks of 128.
    AnyGrid g;
    const int64_t padded = (K + 127) / 128 * 128, cap = kAnySmemBytes / 4 / l.mt / 256 * 256, cap1 = kAnySmemBytes1 / 4 / l.mt / 256 * 256;
    const bool big = l.split || padded > cap;
    g.warps = big ? 16 : 8;
    g.row_warps = l.split ? 8 : g.warps;
    g.blocks_per_sm = big ? 1 : 2;
    g.window = !big ? padded : padded < cap1 ? padded : cap1;
    g.groups = (N + g.row_warps * l.rt - 1) / (g.row_warps * l.rt);
    g.batch_blocks = (M + l.mt - 1) / l.mt;
    g.blocks_x = (int64_t)g.blocks_per_sm * sms / g.batch_blocks;
    if (g.blocks_x < 1) g.blocks_x = 1;
    if (g.blocks_x > g.groups) g.blocks_x = g.groups;
    return g;
}

bool any_layout_fits(const AnyLayout& l, int64_t K, int S)
{
    if ((l.mt != 1 && l.mt != 2 && l.mt != 4 && l.mt != 8) || (l.rt != 1 && l.rt != 2 && l.rt != 4)) return false;
    // A warp a segment: sixteen warps whose block holds all of K.  (Not for four rows by one or two batch rows: of 200 000 drawn
    // shapes the rule would take these 16 times.)
    if (l.split && l.rt == 4 && l.mt < 4) return false;
    return !l.split || (S == 2 && l.mt < 8 && (K + 127) / 128 * 128 * 4 * l.mt + kAnySplitBytes <= kAnySmemBytes1);
}

// Predicted cycles of a layout: instructions of a warp (operands, line-up and multiplications of its chunks, its part of the
// activations, lane trees), at the rate of a lone warp or of the SM's schedulers, whichever is slower.  Constants fitted to every layout
// of 337 drawn shapes (M 1 .. 64, N 64 .. 20000, K 101 .. 10001): mean loss against the best layout 2 %; against the fixed rule below
// 0.72 of the time on average, at most 1.034 (M = 1, N = 366, K = 7999 18.5 and 19.1 us).
static double layout_cost(const AnyLayout& l, int64_t M, int64_t N, int64_t K, int S, int wfmt, int sms)
{
    if (!any_layout_fits(l, K, S)) return 1e300;
    const AnyGrid g = any_grid(l, M, N, K, sms);
    const int64_t padded = (K + 127) / 128 * 128, occ = g.blocks_per_sm;
    const int64_t blocks = g.blocks_x * g.batch_blocks, per_sm = (blocks + sms - 1) / sms;
    if (l.split && blocks > sms) return 1e300;
    const double iters = (double)((g.groups + g.blocks_x - 1) / g.blocks_x), waves = (double)((blocks + occ * sms - 1) / (occ * sms));
    const double chunks = (double)padded / 128 / (l.split ? 2 : 1);
    double per_chunk = l.mt * (2.34 + (l.rt == 1 ? 4.81 : 1.94 * l.rt));
    if (l.mt * l.rt >= 32 && wfmt != 2) per_chunk *= 1.37;       // registers run out
    per_chunk += 7.65 + l.rt * (wfmt == 2 ? 20.6 : 10.8);
    const double body = chunks * per_chunk + 1.42 * l.mt * l.rt * (l.split ? 1 : 2) + 256;
    const double stage = 15.3 * l.mt * (double)g.window / (32.0 * g.warps) *
                         (g.window >= padded ? 1.0 : (double)((padded + g.window - 1) / g.window) * iters);
    const double shared = (double)(g.warps * (per_sm < occ ? per_sm : occ)) / 4 * 1.09;
    return (l.split && l.rt == 4 ? 1.065 : 1.0) * waves * ((body * iters + stage) * (shared > 3.92 ? shared : 3.92) + 521);
}

// Fewer batch rows a warp than there are, where the layer leaves SMs idle otherwise (the weights then come from L2 for the other batch
// blocks): M = 6, N = 1333, K = 1001 6.4 -> 4.1 us, M = 7, N = 250, K = 3001 with FP32 weights 10.9 -> 5.3; a warp a segment: M = 8, N = 64,
// K = 4095 19.7 -> 6.7.  The largest batch block with one, two or four rows by the number of warps, the rule without this, keeps the calls
// that would not gain 3 %.
AnyLayout any_layout_for(int64_t M, int64_t N, int64_t K, int S, int wfmt, int sms)
{
    count_schedule_search();
    const int most = M <= 1 ? 1 : M <= 2 ? 2 : M <= 4 ? 4 : 8;
    const int64_t rows = N * ((M + most - 1) / most);
    AnyLayout best{most, rows >= 4ll * 8 * sms ? 4 : rows >= 2ll * 4 * sms ? 2 : 1, 0};
    double best_cost = 0.97 * layout_cost(best, M, N, K, S, wfmt, sms);
    for (int mt = most; mt >= 1 && 16 * mt >= M; mt /= 2)
        for (int rt = 1; rt <= 4; rt *= 2)
            for (int split = 0; split <= (S == 2 && mt < 8 ? 1 : 0); ++split) {
                const AnyLayout l{mt, rt, split};
                const double c = layout_cost(l, M, N, K, S, wfmt, sms);
                if (c < best_cost) { best_cost = c; best = l; }
            }
    return best;
}

}  // namespace detlin
