// Prefill kernel (bucket M > 64): register-tiled FP32 GEMM on the CUDA cores (rule R1:
// IEEE FMA only, never tensor cores) in the frozen prefill order (V=1, L=1, P=1): every output is one
// accumulation chain per K segment, strictly ascending in k; segments are summed in ascending order and
// the bias comes last (rule R3).
//
// One packed fma.rn.f32x2 advances the chains of two output columns of the same row by one element; each half is
// an ordinary fma.rn.f32, so the pairing is invisible in the bits.
//
// What bounds this loop on B200 (measured on resident shared memory): a packed FMA takes two issue slots, every other
// instruction comes on top (a 16-byte shared load costs about 1.8 slots, an integer operation one; nothing issues
// beside a packed FMA), so the fraction of the FP32 peak is the packed FMAs' share of the slots, less what the warps
// wait for.  The schedule keeps everything else out of the multiply loop, and nothing in it waits for a latency:
//   * a thread owns 16 rows x 8 columns (14, 12 or 10 rows where that pads the batch less): six 16-byte shared loads
//     per 64 packed FMAs.  On resident tiles that loop reaches 94 % of the peak (8 x 8: 91 %, 8 x 4: 82 %, 4 x 8: 77 %,
//     4 x 4: 64 %); the smaller thread tiles serve problems that would otherwise leave SMs without work;
//   * the multiplying warps do nothing else.  Four more warps prepare their operands: both tiles arrive by TMA as they
//     are stored ([rows][32 k]), the loop wants them k-major in FP32 (Eq. 2: the upcast is exact).  A thread
//     converts blocks of 4 rows x 4 k: four shared loads, the widenings, four 16-byte stores.  TMA fills what lies outside
//     the matrices with zeros, so there are no bounds checks.  The two groups of warps meet in mbarriers only.  With the
//     multiplying warps converting for themselves between block-wide barriers the same 16 x 8 tile reached 76 % (two
//     warps per scheduler stand still together);
//   * the first operands of the next slab are loaded under the last FMAs of this one (79 -> 86 % together with
//     conflict-free preparation and no block-wide stops at the ends of units).
// Schedule (numerically inert): K in slabs of 32, block tile BM rows (128, 112, 96 or 80) by 256, 128, 64 or 32 columns.
//
// Split of the work: a unit is one K segment of one output tile (one chain per output).  Where there are more units than
// SMs, the slabs of all units form one line, tile by tile, segment by segment, and every block takes an equal
// stretch of it, so no SM idles in a last wave.  Where a stretch ends inside a unit, the block that owns the unit's
// beginning hands its accumulators over through memory and the next block carries the same chains on: the sequence of
// roundings is that of one block.  A block works on the unit it has to hand over FIRST and on the unit it takes over
// LAST, so the hand-over is long done when it is needed.  Blocks number themselves in the order in which they start (a
// ticket), so a block only ever waits for one that is already running; the wait is bounded like every other.
//
// Measured on B200, whole call: M = 512, N = 28672, K = 4096 1862 us (86.7 % of 74.45 TFLOP/s); M = 2048, N = 4096, K = 14336 3616 us
// (89.3 %); M = 72, N = 28672, K = 4096 311 us; M = 128, N = 4096, K = 14336 255 us; 100 x 1000 x 1000 with FP32 weights 12.6 us.  (8 x 8
// outputs a thread, every warp converting for itself, activations transposed by a first launch: 2005, 3916, 391, 299 and 41 us.)
//
// Any K, any alignment (PLAIN): rows that start anywhere are out of TMA's reach, so the preparing warps load them themselves,
// a slab ahead (a block of 4 rows x 4 k ahead for the 256 columns wide tile, whose register split leaves no more: 56 registers
// spilled, so they get 88 here and the multiplying warps 208); a 16-bit row's weights are two or three aligned words, lined up
// by byte permutations (element by element where such a word would reach outside of W).  Beyond K they store -0.0 for
// activations and +0 for weights: the product is -0.0, and adding -0.0 changes no accumulator (not even a -0.0 one), so the
// multiply loop may run on to a whole octet.  Everything else is the same kernel.  M = 300, N = 8192, K = 4097 379 us (71 % of 74.45
// TFLOP/s; the scalar loads hold it up; one thread per output 13362); 100 x 1001 x 1001 18 us, with FP32 weights 17 (156, 157);
// 130 x 500 x 333 13 us (48).
//
// Every wait is bounded: one that expires records the fact in the device status word and the block returns without
// storing.
#pragma once
#include "internal.h"
#include "device_utils.cuh"
#include "pipeline_utils.cuh"
#include <type_traits>

namespace detlin {

namespace prefill_detail {

using namespace pipe;

constexpr int BK = 32;
constexpr int kPrepWarps = 4, kPrepThreads = 32 * kPrepWarps;
constexpr int kMaxMulWarps = 8;
constexpr int kPrepBarrier = 1;                      // named barrier of the preparing warps

// Thread tile TR x TC on LX x LY multiplying threads (columns x rows).
template <int WF, int TR, int TC, int LX, int LY, bool PLAIN = false> struct Tile {
    static constexpr int BM = TR * LY, BN = TC * LX;
    static constexpr int kMulThreads = LX * LY, kMulWarps = kMulThreads / 32, kThreads = kMulThreads + kPrepThreads;
    static constexpr int kXGroups = BM / 4, kWGroups = BN / 4;            // 16-byte groups of a k row
    static constexpr int kXPitch = kXGroups * 16;                         // bytes of a prepared k row of activations
    static constexpr int kWPitch = BN * 4 + 16;                           // and of weights: 4 pitches are 64 bytes off the bank period
    static constexpr int kXBytes = BK * kXPitch, kWBytes = BK * kWPitch;  // one prepared stage
    static constexpr int kRawXBytes = BM * BK * 4, kRawWBytes = BN * BK * WeightElem<WF>::bytes;
    static constexpr int kRawBytes = kRawXBytes + kRawWBytes;
    static constexpr bool kWide = TR * TC > 64;
    // Raw stages cover the latency of memory: a slab of the wide tile takes 4 us, of the narrow ones down to 0.3 us.
    static constexpr int kRawStages = PLAIN ? 0 : kWide ? 2 : (BN > 64 ? 3 : 4);
    static constexpr int kBudget = 227 * 1024 - 1024 - 256;
    static constexpr int kStages = 3 * (kXBytes + kWBytes) + kRawStages * kRawBytes <= kBudget ? 3 : 2;
    static constexpr int kSmemBytes = kStages * (kXBytes + kWBytes) + kRawStages * kRawBytes + 256 + 1024;   // + barriers, + alignment
    static_assert(kSmemBytes <= 227 * 1024, "shared memory");
    // A block of twelve warps is launched with 168 registers a thread; a 16 x 8 tile wants more, the preparing warps less:
    // 256 x 224 + 128 x 56 = 384 x 168 = 256 x 208 + 128 x 88.
    static constexpr int kMulRegs = PLAIN ? 208 : 224, kPrepRegs = PLAIN ? 88 : 56;
    static_assert(!kWide || kMulThreads * kMulRegs + kPrepThreads * kPrepRegs <= kThreads * 168, "the block's own registers");
    static_assert(!kWide || kMulWarps % 4 == 0, "registers move between whole warpgroups");
    static_assert(kMulWarps <= kMaxMulWarps && kMulThreads % 32 == 0, "warps");
};

struct Args {
    const float* x;              // PLAIN: the operands themselves
    const void* w;
    const float* bias;
    float* y;
    float* partials;             // S > 1: segment sums, [tile][segment][piece][thread] in 8-byte pieces with counters, else [segment][M][N]
    float* handoff;              // [block][piece][thread] in 8-byte pieces: accumulators of a unit carried on by the next block
    unsigned* sync;              // [0] ticket, [8 + 8 block + warp] hand-over flags; all zero between launches
    unsigned* tile_counters;     // S > 1: one per tile and multiplying warp, zero between launches; nullptr: a second launch combines
    DeviceStatus* status;
    long long ldy, total;        // total = slabs of all units
    int M, N, K;
    int seg_slabs, tile_slabs;   // slabs of a (full) segment and of a tile
    int S, tiles_m;
    int cut;                     // 1: blocks take equal stretches of slabs; 0: block b is unit b
    unsigned long long wait_limit_ns;
    int test_flags;
};

template <int REGS>
__device__ __forceinline__ void reg_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS)); }
template <int REGS>
__device__ __forceinline__ void reg_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS)); }

// Barrier of the preparing warps that carries a vote (every warp takes part, whatever its vote).
__device__ __forceinline__ bool prep_vote(bool ok)
{
    int r;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %1, 0;\n\tbar.red.and.pred q, %2, %3, p;\n\tselp.s32 %0, 1, 0, q;\n\t}"
                 : "=r"(r) : "r"((int)ok), "n"(kPrepBarrier), "n"(kPrepThreads) : "memory");
    return r != 0;
}
__device__ __forceinline__ void sts128(uint32_t addr, float a, float b, float c, float d)
{
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}
__device__ __forceinline__ float2 lds_f2(uint32_t addr)
{
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr));
    return v;
}

// A block's stretch of the line of slabs and the order in which it visits its units: the last one first (the next block
// may be waiting for it), then the others ascending, the first one last.
struct Walk {
    long long lo, hi;
    int u_first, u_last;
    __device__ __forceinline__ int count() const { return u_last - u_first + 1; }
    __device__ __forceinline__ int unit(int j) const { return j == 0 ? u_last : (j == count() - 1 ? u_first : u_first + j); }
};

// one unit's stretch inside a block: tile, segment, first k and number of slabs
struct Piece {
    int tile, s, k0, n_slabs;
    bool takes_over, hands_over;
};

__device__ __forceinline__ int unit_at(const Args& a, long long pos)
{
    const int tile = (int)(pos / a.tile_slabs);
    return tile * a.S + (int)(pos - (long long)tile * a.tile_slabs) / a.seg_slabs;
}

__device__ __forceinline__ Piece piece_of(const Args& a, const Walk& w, int j)
{
    Piece p;
    // (in the order of visits the middle units are u_first + 1 .. u_last - 1)
    const int u = w.unit(j);
    p.tile = u / a.S;
    p.s = u - p.tile * a.S;
    const int s_lo = p.s * a.seg_slabs, s_hi = min(a.tile_slabs, s_lo + a.seg_slabs);
    const long long base = (long long)p.tile * a.tile_slabs;
    const int lo = (int)max((long long)s_lo, w.lo - base), hi = (int)min((long long)s_hi, w.hi - base);
    p.k0 = lo * BK;
    p.n_slabs = hi - lo;
    p.takes_over = lo > s_lo;
    p.hands_over = hi < s_hi;
    return p;
}

// The requesting thread's position in the block's sequence of slabs.
struct Cursor {
    int j, left, k, m0, n0;
};

template <int WF, int TR, int TC, int LX, int LY, bool PLAIN>
__global__ void __launch_bounds__((Tile<WF, TR, TC, LX, LY, PLAIN>::kThreads), 1)
prefill_tma_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w, const __grid_constant__ Args a)
{
    typedef Tile<WF, TR, TC, LX, LY, PLAIN> T;
    constexpr int BM = T::BM, BN = T::BN, ST = T::kStages, RS = T::kRawStages;
    constexpr int kMulThreads = T::kMulThreads, kMulWarps = T::kMulWarps;
    constexpr int XG = TR / 4, XR = TR % 4;          // a thread's rows: XG groups of four, then XR (0 or 2)
    static_assert(XR == 0 || XR == 2, "rows per thread: even");
    constexpr int NGX = T::kXGroups, NGW = T::kWGroups;
    constexpr int kStageBytes = T::kXBytes + T::kWBytes;
    __shared__ int shared_ticket;
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw0 = (smem_u32(smem_raw) + 1023u) & ~1023u;          // raw stages: weights, then activations
    const uint32_t ring = raw0 + RS * T::kRawBytes;                       // prepared stages: weights, then activations
    const uint32_t full0 = ring + ST * kStageBytes;                       // prepared stage is complete
    const uint32_t empty0 = full0 + 8 * ST;                               // prepared stage has been read
    const uint32_t rawfull0 = empty0 + 8 * ST;                            // raw stage has landed
    const uint32_t abort_flag = rawfull0 + 8 * RS;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < ST; ++i) { mbar_init(full0 + 8 * i, kPrepWarps); mbar_init(empty0 + 8 * i, kMulWarps); }
        for (int i = 0; i < RS; ++i) mbar_init(rawfull0 + 8 * i, 1);
        sts_volatile_i32(abort_flag, 0);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        shared_ticket = a.cut ? (int)atomicInc(a.sync, gridDim.x - 1) : (int)blockIdx.x;     // the ticket wraps to zero
    }
    __syncthreads();
    const int blk = shared_ticket;

    Walk w;
    if (a.cut) {
        w.lo = a.total * blk / (int)gridDim.x;
        w.hi = a.total * (blk + 1) / (int)gridDim.x;
    } else {
        const int tile = blk / a.S, s = blk - tile * a.S;
        w.lo = (long long)tile * a.tile_slabs + s * a.seg_slabs;
        w.hi = min(w.lo + a.seg_slabs, (long long)(tile + 1) * a.tile_slabs);
    }
    w.u_first = unit_at(a, w.lo);
    w.u_last = unit_at(a, w.hi - 1);
    const int n_it = (int)(w.hi - w.lo);             // slabs of this block
    const int n_pieces = w.count();

    if (warp >= kMulWarps) {
        // ---------------- preparing warps ----------------
        if constexpr (T::kWide) reg_dec<T::kPrepRegs>();
        const int t = threadIdx.x - kMulThreads;
        if constexpr (PLAIN) {
            typedef typename WeightElem<WF>::type WT;
            constexpr int NHW = (NGW + 15) / 16, NHX = (NGX + 15) / 16, NB = NHW + NHX;      // blocks of a slab per thread
            const int g0 = (t & 7) + 8 * (t >> 6), q = (t >> 3) & 7;
            const WT* wg = static_cast<const WT*>(a.w);
            asm volatile("griddepcontrol.wait;" ::: "memory");
            struct Block { uint32_t v[4][4]; unsigned odd; };
            int j = 0, k = 0, left = 0, m0 = 0, n0 = 0;
            auto open = [&]() {
                if (j >= n_pieces) return;
                const Piece p = piece_of(a, w, j);
                left = p.n_slabs;
                k = p.k0;
                m0 = (p.tile % a.tiles_m) * BM;
                n0 = (p.tile / a.tiles_m) * BN;
            };
            open();
            // block b of the slab at the cursor: weights first, then activations.  Rows beyond the matrices repeat the last one.
            auto load = [&](Block& r, int b) {
                const int kq = k + 4 * q;
                r.odd = 0u;
                if (b < NHW) {
                    if (NGW % 16 != 0 && g0 + 16 * b >= NGW) return;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int n = min(n0 + g0 + 16 * b + NGW * i, a.N - 1);
                        const WT* src = wg + (long long)n * a.K + kq;
                        const bool odd = WF != 2 && (reinterpret_cast<uintptr_t>(src) & 2u) != 0;
                        if (kq + 4 <= a.K && !(odd && ((n == 0 && kq == 0) || (n == a.N - 1 && kq + 4 == a.K)))) {
                            if constexpr (WF == 2) {
#pragma unroll
                                for (int e = 0; e < 4; ++e) r.v[i][e] = __float_as_uint(__ldg(src + e));
                            } else {
                                const uint32_t* p = reinterpret_cast<const uint32_t*>(reinterpret_cast<uintptr_t>(src) & ~(uintptr_t)3);
                                r.v[i][0] = __ldg(p);
                                r.v[i][1] = __ldg(p + 1);
                                r.v[i][2] = odd ? __ldg(p + 2) : 0u;
                                r.odd |= (odd ? 1u : 0u) << i;
                            }
                        } else {
                            uint32_t e[4];
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                if constexpr (WF == 2) e[u] = kq + u < a.K ? __float_as_uint(__ldg(src + u)) : 0u;
                                else e[u] = kq + u < a.K ? (uint32_t)__ldg(src + u) : 0u;
                            }
                            if constexpr (WF == 2) {
#pragma unroll
                                for (int u = 0; u < 4; ++u) r.v[i][u] = e[u];
                            } else {
                                r.v[i][0] = e[0] | (e[1] << 16);
                                r.v[i][1] = e[2] | (e[3] << 16);
                                r.v[i][2] = 0u;
                            }
                        }
                    }
                } else {
                    const int h = b - NHW;
                    if (NGX % 16 != 0 && g0 + 16 * h >= NGX) return;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int m = min(m0 + g0 + 16 * h + NGX * i, a.M - 1);
                        const float* src = a.x + (long long)m * a.K + kq;
#pragma unroll
                        for (int e = 0; e < 4; ++e) r.v[i][e] = kq + e < a.K ? __float_as_uint(__ldg(src + e)) : 0x80000000u;
                    }
                }
            };
            auto store = [&](const Block& r, int b, uint32_t stage) {
                float f[4][4];                       // [row][k]
                uint32_t dst;
                uint32_t pitch;
                if (b < NHW) {
                    if (NGW % 16 != 0 && g0 + 16 * b >= NGW) return;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if constexpr (WF == 2) {
#pragma unroll
                            for (int e = 0; e < 4; ++e) f[i][e] = __uint_as_float(r.v[i][e]);
                        } else {
                            const uint32_t sel = ((r.odd >> i) & 1u) ? 0x5432u : 0x3210u;
                            const uint32_t lo = __byte_perm(r.v[i][0], r.v[i][1], sel), hi = __byte_perm(r.v[i][1], r.v[i][2], sel);
                            f[i][0] = up16_lo<WF>(lo); f[i][1] = up16_hi<WF>(lo);
                            f[i][2] = up16_lo<WF>(hi); f[i][3] = up16_hi<WF>(hi);
                        }
                    }
                    pitch = T::kWPitch;
                    dst = stage + (uint32_t)(4 * q * T::kWPitch + ((g0 + 16 * b) << 4));
                } else {
                    const int h = b - NHW;
                    if (NGX % 16 != 0 && g0 + 16 * h >= NGX) return;
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int e = 0; e < 4; ++e) f[i][e] = __uint_as_float(r.v[i][e]);
                    pitch = T::kXPitch;
                    dst = stage + T::kWBytes + (uint32_t)(4 * q * T::kXPitch + ((g0 + 16 * h) << 4));
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) sts128(dst + (uint32_t)e * pitch, f[0][e], f[1][e], f[2][e], f[3][e]);
            };
            auto advance = [&]() {
                k += BK;
                if (--left == 0) { ++j; open(); }
            };
            // narrow tiles leave the registers to have a whole slab on its way, wide ones a block
            constexpr bool kSlabAhead = !T::kWide;
            Block r[kSlabAhead ? NB : 2];
#pragma unroll
            for (int b = 0; b < (kSlabAhead ? NB : 1); ++b) load(r[b], b);
            int st = 0;
            unsigned phase = 0;
#pragma unroll 1
            for (int it = 0; it < n_it; ++it) {
                if (it >= ST) {
                    const bool ok = mbar_wait(empty0 + 8 * st, phase ^ 1u, abort_flag, a.status, a.wait_limit_ns, 3);
                    if (!__all_sync(0xffffffffu, ok)) return;
                }
                const uint32_t stage = ring + (uint32_t)(st * kStageBytes);
                if constexpr (kSlabAhead) {
                    advance();
#pragma unroll
                    for (int b = 0; b < NB; ++b) {
                        store(r[b], b, stage);
                        if (it + 1 < n_it) load(r[b], b);
                    }
                } else {
#pragma unroll
                    for (int b = 0; b < NB; ++b) {
                        if (b + 1 < NB) {
                            load(r[(b + 1) & 1], b + 1);
                        } else {
                            advance();
                            if (it + 1 < n_it) load(r[NB & 1], 0);
                        }
                        store(r[b & 1], b, stage);
                    }
                    if constexpr (NB & 1) r[0] = r[1];
                }
                __syncwarp();
                // (test hook: the first block's first slab is never announced, so the multiplying warps' wait for it expires)
                if (lane == 0 && !((a.test_flags & 1) && blk == 0 && it == 0)) mbar_arrive(full0 + 8 * st);
                if (++st == ST) { st = 0; phase ^= 1u; }
            }
            return;
        }
        constexpr int RSN = RS > 0 ? RS : 1;         // (nothing below is reached without raw stages)
        Cursor c{};
        auto cursor_at = [&](int j) {
            c.j = j;
            if (j >= n_pieces) return;
            const Piece p = piece_of(a, w, j);
            c.left = p.n_slabs;
            c.k = p.k0;
            c.m0 = (p.tile % a.tiles_m) * BM;
            c.n0 = (p.tile / a.tiles_m) * BN;
        };
        // (test hook: the first block never requests its first activation tile, so its first wait expires)
        const bool withhold = (a.test_flags & 1) && blk == 0;
        auto request = [&](int it, int slot) {       // one thread: the raw stage at the cursor, which moves on
            const uint32_t bar = rawfull0 + 8 * slot, dst = raw0 + (uint32_t)slot * T::kRawBytes;
            mbar_arrive_expect_tx(bar, T::kRawBytes);
            tma_load_2d_plain(dst, &map_w, c.k, c.n0, bar);
            if (!(withhold && it == 0)) tma_load_2d_plain(dst + T::kRawWBytes, &map_x, c.k, c.m0, bar);
            c.k += BK;
            if (--c.left == 0) cursor_at(c.j + 1);
        };
        int requested = min(RS, n_it);
        if (t == 0) {
            cursor_at(0);
            asm volatile("griddepcontrol.wait;" ::: "memory");
            for (int i = 0; i < requested; ++i) request(i, i);
        }
        // Blocks of 4 rows {g, g + NG, g + 2 NG, g + 3 NG} x 4 k (quad q): element (row g + NG i, k) goes to element i of the
        // 16-byte group g of k row k.  The raw tiles are swizzled by TMA in 16-byte chunks (128-byte rows: chunk ^ row & 7;
        // 64-byte rows: chunk ^ row / 2 & 3), so that eight lanes with consecutive g and one q (or a pair of q, 64-byte
        // rows) load from distinct banks; with the same lanes the stores fill whole k rows, or half rows that the pitch
        // places on different banks.
        const int g0 = (WF == 2 ? t & 7 : (t >> 1) & 7) + 8 * (t >> 6), q = WF == 2 ? (t >> 3) & 7 : (t & 1) + 2 * ((t >> 4) & 3);
        const uint32_t src_w0 = WF == 2 ? (uint32_t)(g0 * 128 + ((q ^ (g0 & 7)) << 4))
                                        : (uint32_t)(g0 * 64 + (((q >> 1) ^ ((g0 >> 1) & 3)) << 4) + ((q & 1) << 3));
        const uint32_t dst_w0 = (uint32_t)(4 * q * T::kWPitch + (g0 << 4));
        const int gx = (t & 7) + 8 * (t >> 6), qx = (t >> 3) & 7;
        const uint32_t src_x0 = (uint32_t)(gx * 128 + ((qx ^ (gx & 7)) << 4)), dst_x0 = (uint32_t)(4 * qx * T::kXPitch + (gx << 4));
        constexpr int kWRow = BK * WeightElem<WF>::bytes;
        static_assert(NGW % 8 == 0 && NGX % 4 == 0, "swizzle phase of rows NG apart");
        int st = 0, rs = 0;
        unsigned phase = 0, rphase = 0;
        bool ok = true;
#pragma unroll 1
        for (int it = 0; it < n_it; ++it) {
            ok = mbar_wait(rawfull0 + 8 * rs, rphase, abort_flag, a.status, a.wait_limit_ns, 3);
            if (ok && it >= ST) ok = mbar_wait(empty0 + 8 * st, phase ^ 1u, abort_flag, a.status, a.wait_limit_ns, 3);
            ok = __all_sync(0xffffffffu, ok);
            if (ok) {
                const uint32_t raw = raw0 + (uint32_t)rs * T::kRawBytes;
                const uint32_t stage = ring + (uint32_t)(st * kStageBytes);
                const uint32_t src_w = raw + src_w0, dst_w = stage + dst_w0;
#pragma unroll
                for (int h = 0; h < (NGW + 15) / 16; ++h) {
                    if (NGW % 16 == 0 || g0 + 16 * h < NGW) {
                        float v[4][4];               // [row][k]
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const uint32_t src = src_w + (uint32_t)((16 * h + NGW * i) * kWRow);
                            if constexpr (WF == 2) {
                                const float4 f = lds128(src);
                                v[i][0] = f.x; v[i][1] = f.y; v[i][2] = f.z; v[i][3] = f.w;
                            } else {
                                const uint2 f = lds64(src);
                                v[i][0] = up16_lo<WF>(f.x); v[i][1] = up16_hi<WF>(f.x);
                                v[i][2] = up16_lo<WF>(f.y); v[i][3] = up16_hi<WF>(f.y);
                            }
                        }
#pragma unroll
                        for (int e = 0; e < 4; ++e) sts128(dst_w + (uint32_t)(e * T::kWPitch + h * 256), v[0][e], v[1][e], v[2][e], v[3][e]);
                    }
                }
                const uint32_t src_x = raw + T::kRawWBytes + src_x0, dst_x = stage + T::kWBytes + dst_x0;
#pragma unroll
                for (int h = 0; h < (NGX + 15) / 16; ++h) {
                    if (NGX % 16 == 0 || gx + 16 * h < NGX) {
                        float4 v[4];
                        // rows an odd multiple of 4 apart (NGX % 8 = 4) sit in the other half of the swizzle period
#pragma unroll
                        for (int i = 0; i < 4; ++i) v[i] = lds128((src_x ^ (uint32_t)((NGX % 8) * (i & 1) << 4)) + (uint32_t)((16 * h + NGX * i) * BK) * 4u);
                        const uint32_t d = dst_x + (uint32_t)(h * 256);
                        sts128(d, v[0].x, v[1].x, v[2].x, v[3].x);
                        sts128(d + T::kXPitch, v[0].y, v[1].y, v[2].y, v[3].y);
                        sts128(d + 2 * T::kXPitch, v[0].z, v[1].z, v[2].z, v[3].z);
                        sts128(d + 3 * T::kXPitch, v[0].w, v[1].w, v[2].w, v[3].w);
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(full0 + 8 * st);
            }
            if (++st == ST) { st = 0; phase ^= 1u; }
            // the raw stage has been read by all four warps: it may be overwritten
            ok = prep_vote(ok);
            if (!ok) break;
            if (requested < n_it) {
                if (t == 0) request(requested, rs);
                ++requested;
            }
            if (++rs == RS) { rs = 0; rphase ^= 1u; }
        }
        if (!ok && t == 0) {
            // aborting: wait (bounded) for the requests still in flight
            const unsigned long long t0 = global_timer_ns();
            for (int i = requested > RS ? requested - RS : 0; i < requested; ++i)
                while (!(withhold && i == 0) && !mbar_try_wait(rawfull0 + 8 * (i % RSN), (uint32_t)(i / RSN) & 1u))
                    if (global_timer_ns() - t0 > a.wait_limit_ns) return;
        }
        return;
    }

    // ---------------- multiplying warps ----------------
    if constexpr (T::kWide) reg_inc<T::kMulRegs>();
    const int tid = threadIdx.x;
    // a warp = 16 column groups x 2 row groups, or 8 x 4 where a tile is only eight groups wide
    constexpr int LNX = LX >= 16 ? 16 : 8, WX = LX / LNX, LNY = 32 / LNX;
    const int tx = (lane & (LNX - 1)) + LNX * (warp % WX), ty = lane / LNX + LNY * (warp / WX);

    // acc[r][2 h + p]: row r of the thread, column group tx + LX h, columns of elements 2 p and 2 p + 1 of the group.
    // Column group g holds the columns g, g + NGW, g + 2 NGW, g + 3 NGW; row group g likewise.  The thread's row groups are
    // ty + LY h and, with a remainder, half of group LY XG + ty / 2.
    float2 acc[TR][TC / 2];
    const uint32_t w_thr = ring + (uint32_t)(tx << 4);
    const uint32_t x_thr = ring + T::kWBytes + (uint32_t)(ty << 4);
    const uint32_t x_rem = ring + T::kWBytes + (uint32_t)((LY * XG + (ty >> 1)) << 4) + (uint32_t)((ty & 1) << 3);

    // Operands of the current k: the thread's activations and the first half of its weights (TC = 4: all of them); what the
    // next k needs is loaded into the same registers as soon as their last use has been issued.
    float4 xv[XG] = {}, wa = {};
    float2 xw = make_float2(0.0f, 0.0f);
    auto fma_group = [&](int g, int j, const float2& wv) {    // rows 4 g .. 4 g + 3, column pair j
        fma2(acc[4 * g][j], xv[g].x, wv);
        fma2(acc[4 * g + 1][j], xv[g].y, wv);
        fma2(acc[4 * g + 2][j], xv[g].z, wv);
        fma2(acc[4 * g + 3][j], xv[g].w, wv);
    };
    auto fma_rest = [&](int j, const float2& wv) {
        if constexpr (XR == 2) {
            fma2(acc[4 * XG][j], xw.x, wv);
            fma2(acc[4 * XG + 1][j], xw.y, wv);
        }
    };
    auto load_first = [&](uint32_t off) {            // operands of the first k at offset `off` of the ring
#pragma unroll
        for (int g = 0; g < XG; ++g) xv[g] = lds128(x_thr + off + (uint32_t)(16 * LY * g));
        if constexpr (XR == 2) xw = lds_f2(x_rem + off);
        wa = lds128(w_thr + off);
    };
    // N k of a slab at the addresses w, x, r; the operands of the k after them are loaded from wn, xn, rn.  The order of
    // the instructions is pinned (volatile): consecutive packed FMAs share the weight pair, and a load sits where its
    // registers have just become free.  Left to itself the compiler loads ahead into further registers, runs out of the
    // 168 that twelve warps leave a thread and spills (82 % of the peak on resident tiles instead of 94 %).
    auto steps = [&](uint32_t w, uint32_t x, [[maybe_unused]] uint32_t r, uint32_t wn, uint32_t xn, [[maybe_unused]] uint32_t rn, auto n_c) {
        constexpr int NK = decltype(n_c)::value;
#pragma unroll
        for (int e = 0; e < NK; ++e) {
            const uint32_t w_next = e < NK - 1 ? w + (uint32_t)((e + 1) * T::kWPitch) : wn;
            const uint32_t x_next = e < NK - 1 ? x + (uint32_t)((e + 1) * T::kXPitch) : xn;
            float4 wd;                               // TC = 8: second half of the weights; TC = 4: the next k's weights
            if constexpr (TC == 8) wd = lds128(w + (uint32_t)(e * T::kWPitch + 16 * LX));
            else wd = lds128(w_next);
            const float2 p0 = make_float2(wa.x, wa.y), p1 = make_float2(wa.z, wa.w);
            if constexpr (TC == 8) {
#pragma unroll
                for (int g = 0; g < XG; ++g) fma_group(g, 0, p0);
                fma_rest(0, p0);
#pragma unroll
                for (int g = 0; g < XG; ++g) fma_group(g, 1, p1);
                fma_rest(1, p1);
                wa = lds128(w_next);
                const float2 p2 = make_float2(wd.x, wd.y), p3 = make_float2(wd.z, wd.w);
#pragma unroll
                for (int g = 0; g < XG; ++g) fma_group(g, 2, p2);
                fma_rest(2, p2);
#pragma unroll
                for (int g = 0; g < XG; ++g) {
                    fma_group(g, 3, p3);
                    xv[g] = lds128(x_next + (uint32_t)(16 * LY * g));
                }
                fma_rest(3, p3);
            } else {
#pragma unroll
                for (int g = 0; g < XG; ++g) fma_group(g, 0, p0);
                fma_rest(0, p0);
#pragma unroll
                for (int g = 0; g < XG; ++g) {
                    fma_group(g, 1, p1);
                    xv[g] = lds128(x_next + (uint32_t)(16 * LY * g));
                }
                fma_rest(1, p1);
                wa = wd;
            }
            if constexpr (XR == 2) xw = lds_f2(e < NK - 1 ? r + (uint32_t)((e + 1) * T::kXPitch) : rn);
        }
    };

    auto row_of = [&](int i) {
        return i < 4 * XG ? ty + LY * (i >> 2) + NGX * (i & 3) : LY * XG + (ty >> 1) + NGX * (2 * (ty & 1) + i - 4 * XG);
    };
    auto col_of = [&](int h, int e) { return tx + LX * h + NGW * e; };
    auto store_y = [&](int m0, int n0) {
        float bv[TC / 4][4];
#pragma unroll
        for (int h = 0; h < TC / 4; ++h)
#pragma unroll
            for (int e = 0; e < 4; ++e) bv[h][e] = (a.bias && n0 + col_of(h, e) < a.N) ? __ldg(a.bias + n0 + col_of(h, e)) : 0.0f;
#pragma unroll
        for (int i = 0; i < TR; ++i) {
            const int m = m0 + row_of(i);
            if (m >= a.M) continue;
            float* row = a.y + (long long)m * a.ldy + n0;
#pragma unroll
            for (int h = 0; h < TC / 4; ++h) {
                const float v[4] = {acc[i][2 * h].x, acc[i][2 * h].y, acc[i][2 * h + 1].x, acc[i][2 * h + 1].y};
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (n0 + col_of(h, e) < a.N) row[col_of(h, e)] = a.bias ? __fadd_rn(v[e], bv[h][e]) : v[e];
            }
        }
    };
    // a thread's accumulators as 8-byte pieces, one every kMulThreads pieces (coalesced).  Not as 16-byte pieces: those would
    // tie four accumulators to four consecutive registers
    auto acc_store = [&](float* dst) {
        float2* p = reinterpret_cast<float2*>(dst) + tid;
#pragma unroll
        for (int i = 0; i < TR; ++i)
#pragma unroll
            for (int c = 0; c < TC / 2; ++c) __stcg(p + (i * (TC / 2) + c) * kMulThreads, acc[i][c]);
    };
    auto acc_load = [&](const float* src) {
        const float2* p = reinterpret_cast<const float2*>(src) + tid;
#pragma unroll
        for (int i = 0; i < TR; ++i)
#pragma unroll
            for (int c = 0; c < TC / 2; ++c) acc[i][c] = __ldcg(p + (i * (TC / 2) + c) * kMulThreads);
    };
    auto acc_add = [&](const float* src) {           // acc = acc + src
        const float2* p = reinterpret_cast<const float2*>(src) + tid;
#pragma unroll
        for (int i = 0; i < TR; ++i)
#pragma unroll
            for (int c = 0; c < TC / 2; ++c) {
                const float2 f = __ldcg(p + (i * (TC / 2) + c) * kMulThreads);
                acc[i][c] = make_float2(__fadd_rn(acc[i][c].x, f.x), __fadd_rn(acc[i][c].y, f.y));
            }
    };

    constexpr size_t kTileFloats = (size_t)BM * BN;
    // Workspaces and y belong to the kernels before this one until they end.  Then the next kernel may start: not before, since it
    // may request its weights at once, and not ahead of this block's ticket, since it may draw tickets of the same plan.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    int st = 0;
    unsigned phase = 0;
    bool loaded = false;                             // the first operands of the next slab are in registers already
#pragma unroll 1
    for (int j = 0; j < n_pieces; ++j) {
        const Piece p = piece_of(a, w, j);
        if (p.takes_over) {
            // carry on the chains that the same warp of the block before this one has begun
            unsigned v = 0u;
            if (lane == 0) {
                unsigned* flag = a.sync + 8 * blk + warp;        // flags of block blk - 1
                const unsigned long long t0 = global_timer_ns();
                for (;;) {
                    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
                    if (v != 0u) break;
                    if (lds_volatile_i32(abort_flag)) break;
                    if (global_timer_ns() - t0 > a.wait_limit_ns) {
                        sts_volatile_i32(abort_flag, 1);
                        atomicMax(&a.status->where, 5u);
                        atomicExch(&a.status->timeout_flag, 1u);
                        break;
                    }
                }
                *flag = 0u;                          // for the next launch
            }
            if (!__any_sync(0xffffffffu, v != 0u)) return;
            acc_load(a.handoff + (size_t)(blk - 1) * kTileFloats);
        } else {
#pragma unroll
            for (int i = 0; i < TR; ++i)
#pragma unroll
                for (int c = 0; c < TC / 2; ++c) acc[i][c] = make_float2(0.0f, 0.0f);
        }
        // k beyond the end of the segment is skipped, not zero-filled; segments end on multiples of 8 (16-bit weights)
        // or 4 (FP32 weights)
        int k_left = min(a.K, (p.s + 1) * a.seg_slabs * BK) - p.k0;
#pragma unroll 1
        for (int sl = 0; sl < p.n_slabs; ++sl) {
            const uint32_t off = (uint32_t)(st * kStageBytes);
            if (!loaded) {
                if (!__all_sync(0xffffffffu, mbar_wait(full0 + 8 * st, phase, abort_flag, a.status, a.wait_limit_ns, 4))) return;
                load_first(off);
            }
            const int st_cur = st;
            if (++st == ST) { st = 0; phase ^= 1u; }
            uint32_t wp = w_thr + off, xp = x_thr + off, rp = x_rem + off;
            using Eight = std::integral_constant<int, 8>;
            using Four = std::integral_constant<int, 4>;
            int n = min(BK, k_left);
            if constexpr (PLAIN) n = (n + 7) & ~7;   // the operands beyond K change nothing
            k_left -= BK;
#pragma unroll 1
            for (; n > 8; n -= 8) {
                steps(wp, xp, rp, wp + 8 * T::kWPitch, xp + 8 * T::kXPitch, rp + 8 * T::kXPitch, Eight());
                wp += 8 * T::kWPitch;
                xp += 8 * T::kXPitch;
                rp += 8 * T::kXPitch;
            }
            // the last k of the slab are followed by the first ones of the next slab, if that has been prepared already
            loaded = __all_sync(0xffffffffu, mbar_test_wait(full0 + 8 * st, phase));
            const uint32_t off_n = loaded ? (uint32_t)(st * kStageBytes) : off;
            if (WF != 2 || PLAIN || n == 8) steps(wp, xp, rp, w_thr + off_n, x_thr + off_n, x_rem + off_n, Eight());
            else steps(wp, xp, rp, w_thr + off_n, x_thr + off_n, x_rem + off_n, Four());
            __syncwarp();
            if (lane == 0) mbar_arrive(empty0 + 8 * st_cur);
        }

        const int m0 = (p.tile % a.tiles_m) * BM, n0 = (p.tile / a.tiles_m) * BN;
        if (p.hands_over) {
            acc_store(a.handoff + (size_t)blk * kTileFloats);
            __threadfence();
            __syncwarp();
            if (lane == 0) asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(a.sync + 8 + 8 * blk + warp), "r"(1u) : "memory");
        } else if (a.S == 1) {
            store_y(m0, n0);
        } else if (a.tile_counters) {
            // ---- split-K fold without a second launch (rule R3): the warp that completes the count of S segment sums of
            // its part of a tile adds them in ascending segment order, then the bias, and stores.  In which block that is
            // depends on timing; what it computes does not.  Nobody waits for anybody, no warp for the others of its
            // block.  The counter returns to zero for the next run. ----
            float* tile_sums = a.partials + (size_t)p.tile * a.S * kTileFloats;
            acc_store(tile_sums + (size_t)p.s * kTileFloats);
            __threadfence();                         // this warp's partials are visible before its count
            __syncwarp();
            int last = 0;
            if (lane == 0) {
                unsigned* cnt = a.tile_counters + (size_t)p.tile * kMulWarps + warp;
                last = atomicAdd(cnt, 1u) == (unsigned)(a.S - 1);
                if (last) *cnt = 0u;
            }
            if (__any_sync(0xffffffffu, last)) {
                __threadfence();                     // the other blocks' partials, counted before ours, are visible
                acc_load(tile_sums);
                for (int s2 = 1; s2 < a.S; ++s2) acc_add(tile_sums + (size_t)s2 * kTileFloats);
                store_y(m0, n0);
            }
        } else {
#pragma unroll
            for (int i = 0; i < TR; ++i) {
                const int m = m0 + row_of(i);
                if (m >= a.M) continue;
                float* row = a.partials + ((long long)p.s * a.M + m) * a.N + n0;
#pragma unroll
                for (int h = 0; h < TC / 4; ++h) {
                    const float v[4] = {acc[i][2 * h].x, acc[i][2 * h].y, acc[i][2 * h + 1].x, acc[i][2 * h + 1].y};
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (n0 + col_of(h, e) < a.N) row[col_of(h, e)] = v[e];
                }
            }
        }
    }
}

}  // namespace prefill_detail

}  // namespace detlin
