// Fixed-order decode attention: one query row per (batch, head) against T cached keys and values.
// Not one of the paper's kernels: the paper keeps vendor attention and names fixed-order attention as the
// outstanding source of residual divergence between GPU architectures.  Here every reduction of the
// attention runs in an order fixed by (T, D) alone, every step one IEEE-754 binary32 operation, so the
// bits do not depend on the batch size, the grid, the SM count or the stream:
//
//   1. s_j = dot(q, k_j) * scale; the dot product in the decode lane order over D (chunks of 128 ascending,
//      lane l owns the 4 consecutive elements c + 4 l + jj, one fma.rn per element from +0, elements
//      beyond D skipped, the 32 lane sums added adjacent-first: xor 1, 2, 4, 8, 16), then one multiply;
//   2. m = max_j s_j (comparisons only);
//   3. e_j = exp_det(s_j - m): one subtraction and the fixed-sequence exponential below;
//   4. l = sum_j e_j in the lane order over j (chunks of 128 keys ascending, lane l owns keys c + 4 l + jj,
//      one add.rn per key from +0, keys beyond T skipped, adjacent-first lane tree);
//   5. for every d: keys in segments of 256; inside a segment a = fma.rn(e_j, v_j[d], a) from +0 with j
//      ascending; segment sums added left to right in ascending order; o[d] = sum / l (one div.rn).
//
// Schedule (numerically inert): a cluster of C thread blocks (C = 1, 2, 4, 8 or 16) per (batch, KV head) serves
// the G = Hq / Hkv query heads that share the head's keys and values, so K and V cross the memory bus once
// per group.  Block r of the cluster owns the keys [r Tc, (r + 1) Tc), Tc a whole number of 256-key
// segments; everything that crosses the blocks goes through distributed shared memory behind hardware
// cluster barriers (no spinning): the exact row maxima (comparisons, order-free), the weights that block 0
// reads to form the denominators in the lane order over ALL keys, and the segment sums that every block
// reads to fold its slice of the outputs in ascending segment order.  C only depends on how many blocks
// fill the GPU and on the shared memory a block may use; every C gives the same bits.
// Inside a block, eight warps: in step 1 a warp takes several keys at a time and folds their lane trees into
// one butterfly reduce-scatter (one shuffle per (key, head) instead of five); scores and weights live in
// shared memory; in step 5 a warp owns (segment, slice of d) items, as wide as keeps every warp busy.  A ninth warp forms
// the denominators meanwhile.
// What bounds it is the stream of K and V, and the stream must not stop while a block computes or waits for its cluster:
// every lane copies the elements that it will itself consume, K first, then V, through a ring of its own in shared
// memory (cp.async: no registers held, no barrier, nobody else reads them), several groups ahead; while the cluster agrees on
// maxima and weights, the ring fills with V.  (Asking for more of V in L2 ahead of use, by bulk prefetch, gained nothing.)
// A block whose scores leave no room for the ring (three groups), or with too little to do for it, loads through registers instead
// (ring_or_registers below).  Next come the instructions: the lane trees (their operands are
// permuted so that no step selects between registers), P.V in packed FMAs.  Small shapes are bound by latency, of reads
// from other blocks' shared memory among others: what crosses blocks is read many values at a time.
// Measured on B200, 32 query / 8 KV heads, D = 128, us a call (in brackets with loads through registers only): B = 8, T = 4096 55.9
// (61.6); B = 8, T = 8192 86.9 (105.6); B = 32, T = 2048 86.3 (97.9); B = 2, T = 4096 31.4 (40.6); B = 1, T = 32768 85.9 (131.8); 8 / 8
// heads, B = 8, T = 2000 28.5 (40.7).
#include "internal.h"
#include "device_utils.cuh"
#include <cooperative_groups.h>

namespace detlin {

namespace {

namespace cg = cooperative_groups;

constexpr int kAttnWarps = 8;            // warps that score keys and multiply values
constexpr int kWorkThreads = 32 * kAttnWarps;
// NS slots of the ring (see below); 0 and 1 stand for loads through registers, by eight warps or with a ninth one that forms the
// denominators meanwhile (as it does with the ring).
template <int NS> constexpr int kAttnThreads = kWorkThreads + (NS > 0 ? 32 : 0);
// Blocks to an SM, which cap a thread's registers: with eight warps, as many as leave eight keys in flight their registers.
template <int G, int DC, int NS> constexpr int kAttnBlocks = NS != 0 ? 2 : G * DC <= 2 ? 4 : G * DC <= 8 ? 2 : 1;
// keys a warp scores together when they come through registers
template <int G, int DC, int NS> constexpr int kPassKeys = NS == 1 && G * DC >= 16 ? 2 : 8;
constexpr int kGroupBytes = 2048;        // ring: bytes a warp copies as one group
constexpr int kSegKeys = 256;            // P.V segment length (part of the order)
constexpr int kMaxCluster = 16;          // blocks per row at most (8 is the portable cluster size, 16 needs the opt-in below)

// The attention's exponential for x <= 0: range reduction by ln 2 in two pieces, degree-7 Taylor polynomial
// by Horner's rule with fused multiply-adds, scaling by 2^n (through 2^(n+64) and 2^-64 below the normal
// range).  Every step is one explicitly rounded binary32 operation; the constants are given by bit pattern.
__device__ __forceinline__ float exp_det(float x)
{
    if (x < -104.0f) return 0.0f;
    const float t = __fmul_rn(x, __uint_as_float(0x3FB8AA3Bu));               // log2(e)
    const float n = rintf(t);                                                // nearest, ties to even
    float f = __fmaf_rn(n, -__uint_as_float(0x3F317200u), x);                // ln 2, high part
    f = __fmaf_rn(n, -__uint_as_float(0x35BFBE8Eu), f);                      // ln 2, low part
    float p = __uint_as_float(0x39500D01u);                                  // 1/5040
    p = __fmaf_rn(p, f, __uint_as_float(0x3AB60B61u));                       // 1/720
    p = __fmaf_rn(p, f, __uint_as_float(0x3C088889u));                       // 1/120
    p = __fmaf_rn(p, f, __uint_as_float(0x3D2AAAABu));                       // 1/24
    p = __fmaf_rn(p, f, __uint_as_float(0x3E2AAAABu));                       // 1/6
    p = __fmaf_rn(p, f, 0.5f);
    p = __fmaf_rn(p, f, 1.0f);
    p = __fmaf_rn(p, f, 1.0f);
    const int ni = (int)n;
    if (ni >= -126) return __fmul_rn(p, __uint_as_float((uint32_t)(ni + 127) << 23));
    const float u = __fmul_rn(p, __uint_as_float((uint32_t)(ni + 64 + 127) << 23));
    return __fmul_rn(u, __uint_as_float((uint32_t)(-64 + 127) << 23));
}

// P.V work items of one block (see step 5 of the kernel).  VW = consecutive d per lane (1, 2 or 4; D % 4 == 0, so a
// lane's VW elements are all inside or all outside D).
template <int G, int VW>
__device__ __forceinline__ void pv_items(const float* e_s, float* part, const float* __restrict__ vb, int Tc, int Tl, int D,
                                         int n_seg_l, int warp, int lane)
{
    constexpr int kKeys = (VW == 4) ? 8 : 16;                  // keys loaded together
    const int n_slices = (D + 32 * VW - 1) / (32 * VW);
    for (int item = warp; item < n_seg_l * n_slices; item += kAttnWarps) {
        const int sgm = item / n_slices, d = 32 * VW * (item % n_slices) + VW * lane;
        const bool ok = d < D;
        float acc[G][VW];
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
            for (int e = 0; e < VW; ++e) acc[g][e] = 0.0f;
        const int j_lo = sgm * kSegKeys, j_hi = min(Tl, j_lo + kSegKeys);
        const float* vp = vb + (ok ? d : 0);
        for (int j0 = j_lo; j0 < j_hi; j0 += kKeys) {
            float vv[kKeys][VW];
#pragma unroll
            for (int p = 0; p < kKeys; ++p) {
                const float* src = vp + (size_t)(j0 + p) * D;
                const bool in = j0 + p < j_hi && ok;
                if constexpr (VW == 4) {
                    const float4 t = in ? __ldg(reinterpret_cast<const float4*>(src)) : make_float4(0.f, 0.f, 0.f, 0.f);
                    vv[p][0] = t.x; vv[p][1] = t.y; vv[p][2] = t.z; vv[p][3] = t.w;
                } else if constexpr (VW == 2) {
                    const float2 t = in ? __ldg(reinterpret_cast<const float2*>(src)) : make_float2(0.f, 0.f);
                    vv[p][0] = t.x; vv[p][1] = t.y;
                } else {
                    vv[p][0] = in ? __ldg(src) : 0.0f;
                }
            }
#pragma unroll
            for (int p4 = 0; p4 < kKeys; p4 += 4) {
                float4 ew[G];                                    // the weights of four keys (j0 is a multiple of 8)
#pragma unroll
                for (int g = 0; g < G; ++g) ew[g] = *reinterpret_cast<const float4*>(e_s + g * Tc + j0 + p4);
#pragma unroll
                for (int pp = 0; pp < 4; ++pp) {
                    if (j0 + p4 + pp < j_hi) {                   // keys beyond the segment are skipped
#pragma unroll
                        for (int g = 0; g < G; ++g) {
                            const float w = pp == 0 ? ew[g].x : pp == 1 ? ew[g].y : pp == 2 ? ew[g].z : ew[g].w;
#pragma unroll
                            for (int e = 0; e < VW; ++e) acc[g][e] = __fmaf_rn(w, vv[p4 + pp][e], acc[g][e]);
                        }
                    }
                }
            }
        }
        if (ok) {
#pragma unroll
            for (int g = 0; g < G; ++g)
#pragma unroll
                for (int e = 0; e < VW; ++e) part[((size_t)sgm * G + g) * D + d + e] = acc[g][e];
        }
    }
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const float* src)
{
    asm volatile("cp.async.cg.shared.global.L2::256B [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
template <int BYTES>
__device__ __forceinline__ void cp_async_ca(uint32_t dst, const float* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// The P.V items of one warp as a sequence of groups of 16 / VW keys (VW consecutive d per lane): position of the next group.
template <int VW>
struct VCursor {
    static constexpr int kKeys = 16 / VW;
    int item, j0, j_hi;
    __device__ __forceinline__ void open(int it, int n_items, int n_slices, int Tl)
    {
        item = it;
        if (it < n_items) {
            j0 = it / n_slices * kSegKeys;
            j_hi = min(Tl, j0 + kSegKeys);
        }
    }
    __device__ __forceinline__ void next(int n_items, int n_slices, int Tl)
    {
        j0 += kKeys;
        if (j0 >= j_hi) open(item + kAttnWarps, n_items, n_slices, Tl);
    }
};

// One lane's ring: groups of its warp's K, then of its V.  NS slots, NS - 1 groups on their way; a group is issued when the one
// before the current has been used up by this very lane.
template <int DC, int NS>
struct Ring {
    [[maybe_unused]] static constexpr int KP = 4 / DC;                         // keys of a K group
    uint32_t base;                                            // the lane's address in slot 0 (16-byte elements)
    int issue_slot, use_slot;
    __device__ __forceinline__ void init(uint32_t warp_base, int lane) { base = warp_base + lane * 16; issue_slot = use_slot = 0; }
    __device__ __forceinline__ void issued() { cp_async_commit(); if (++issue_slot == NS) issue_slot = 0; }
    __device__ __forceinline__ uint32_t used()                // slot of the oldest group, which has landed afterwards
    {
        cp_async_wait<NS - 2>();
        const uint32_t at = base + use_slot * kGroupBytes;
        if (++use_slot == NS) use_slot = 0;
        return at;
    }
    __device__ __forceinline__ void copy_k(const float* kb, int j0, int Tl, int D, int lane, const bool (&d_ok)[DC])
    {
        const float* src = kb + (size_t)j0 * D + 4 * lane;
        const uint32_t dst = base + issue_slot * kGroupBytes;
#pragma unroll
        for (int p = 0; p < KP; ++p, src += D)
            if (j0 + p < Tl) {
#pragma unroll
                for (int c = 0; c < DC; ++c)
                    if (d_ok[c]) cp_async16(dst + (p * DC + c) * 512, src + 128 * c);
            }
    }
    template <int VW>
    __device__ __forceinline__ void copy_v(const float* vb, const VCursor<VW>& cur, int n_slices, int D, int lane)
    {
        const int d = 32 * VW * (cur.item % n_slices) + VW * lane;
        if (d >= D) return;
        const uint32_t dst = base - lane * 16 + issue_slot * kGroupBytes + lane * (4 * VW);
        const float* src = vb + (size_t)cur.j0 * D + d;
        auto copy = [&](int p) {
            if constexpr (VW == 4) cp_async16(dst + p * 512, src);
            else cp_async_ca<4 * VW>(dst + p * (128 * VW), src);
            src += D;
        };
        if (cur.j0 + VCursor<VW>::kKeys <= cur.j_hi) {
#pragma unroll
            for (int p = 0; p < VCursor<VW>::kKeys; ++p) copy(p);
        } else {
#pragma unroll
            for (int p = 0; p < VCursor<VW>::kKeys; ++p)
                if (cur.j0 + p < cur.j_hi) copy(p);
        }
    }
};

// lane_tree_scatter for values that every lane holds in its own order: value t of lane l is value t ^ perm(l), perm having the
// lane's bit 0 at the top of the index, bit 1 below it and so on.  Partners then always keep the lower half and send the
// upper one, and lane l ends with the sum of value perm(l).
template <int NV>
__device__ __forceinline__ float lane_tree_scatter_permuted(float (&v)[NV])
{
    constexpr int H = Scatter<NV>::kSteps;
    static_assert(Scatter<NV>::kKeep == 1, "a power of two, at most 32");
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        if (i < H) {
            const int half = NV >> (i + 1);
#pragma unroll
            for (int t = 0; t < NV / 2; ++t)
                if (t < half) v[t] = __fadd_rn(v[t], __shfl_xor_sync(0xffffffffu, v[t + half], 1 << i));
        } else {
            v[0] = __fadd_rn(v[0], __shfl_xor_sync(0xffffffffu, v[0], 1 << i));
        }
    }
    return v[0];
}
// The lower H bits of the lane in reverse order: its perm for 2^H values.
template <int H>
__device__ __forceinline__ int lane_perm(int lane)
{
    return H == 0 ? 0 : (int)(__brev((unsigned)lane) >> (32 - (H == 0 ? 1 : H)));
}

// Step 1 from the ring: scores of the block's keys; leaves the first groups of V on their way.  Returns the lane's part of the
// row maxima: a lane that holds scores holds those of one head only.
template <int G, int DC, int NS, int VW>
__device__ __forceinline__ float ring_scores(Ring<DC, NS>& ring, VCursor<VW>& ahead, const float4 (&qv)[G][DC], const bool (&d_ok)[DC], float scale,
                                             const float* kb, const float* vb, float* e_s, int Tc, int Tl, int D, int n_items, int n_slices, int warp, int lane)
{
    constexpr int KP = Ring<DC, NS>::KP, NV = KP * G;
    const int n_k = (Tl + kAttnWarps * KP - 1) / (kAttnWarps * KP);
    int issued = 0;
    auto issue = [&]() {
        if (issued < n_k) ring.copy_k(kb, (issued * kAttnWarps + warp) * KP, Tl, D, lane, d_ok);
        else if (ahead.item < n_items) {
            ring.template copy_v<VW>(vb, ahead, n_slices, D, lane);
            ahead.next(n_items, n_slices, Tl);
        }
        ring.issued();
        ++issued;
    };
    for (int i = 0; i < NS - 1; ++i) issue();
    constexpr int kSteps = Scatter<NV>::kSteps;
    static_assert(Scatter<NV>::kKeep == 1, "one score per lane and group");
    const int perm = lane_perm<kSteps>(lane);                 // the lane's own order of the values p * G + g, and its score in the end
    const int p_mine = perm / G, g_mine = perm % G;           // (the heads' order is that of qv)
    float top = -INFINITY;
#pragma unroll 1
    for (int it = 0; it < n_k; ++it) {
        const uint32_t at = ring.used() ^ (uint32_t)(p_mine * DC * 512);      // slots start at multiples of 2048
        issue();
        const int j0 = (it * kAttnWarps + warp) * KP;
        float a[NV];                                        // value index p * G + g
#pragma unroll
        for (int p = 0; p < KP; ++p) {
            float4 kv[DC];
#pragma unroll
            for (int c = 0; c < DC; ++c)
                asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(kv[c].x), "=f"(kv[c].y), "=f"(kv[c].z), "=f"(kv[c].w) : "r"(at ^ (uint32_t)((p * DC + c) * 512)));
#pragma unroll
            for (int g = 0; g < G; ++g) {
                float acc = 0.0f;
#pragma unroll
                for (int c = 0; c < DC; ++c) {
                    if (d_ok[c]) {                           // elements beyond D are skipped, not zero-filled
                        acc = __fmaf_rn(qv[g][c].x, kv[c].x, acc);
                        acc = __fmaf_rn(qv[g][c].y, kv[c].y, acc);
                        acc = __fmaf_rn(qv[g][c].z, kv[c].z, acc);
                        acc = __fmaf_rn(qv[g][c].w, kv[c].w, acc);
                    }
                }
                a[p * G + g] = acc;
            }
        }
        const float sc = __fmul_rn(lane_tree_scatter_permuted<NV>(a), scale);
        if ((lane >> kSteps) == 0 && j0 + p_mine < Tl) {
            e_s[g_mine * Tc + j0 + p_mine] = sc;
            top = fmaxf(top, sc);
        }
    }
    return top;
}

// Step 5 from the ring.
template <int G, int DC, int NS, int VW>
__device__ __forceinline__ void ring_pv(Ring<DC, NS>& ring, VCursor<VW>& ahead, const float* e_s, float* part, const float* vb, int Tc, int Tl, int D,
                                        int n_items, int n_slices, int warp, int lane)
{
    constexpr int kKeys = VCursor<VW>::kKeys;
    for (int item = warp; item < n_items; item += kAttnWarps) {
        const int sgm = item / n_slices, d = 32 * VW * (item % n_slices) + VW * lane;
        const bool ok = d < D;
        constexpr int kPairs = VW > 1 ? VW / 2 : G > 1 ? G / 2 : 1;      // packed FMAs: two d of a head, or (VW = 1) two heads of a d
        float2 acc[VW > 1 ? G : 1][kPairs];
#pragma unroll
        for (int g = 0; g < (VW > 1 ? G : 1); ++g)
#pragma unroll
            for (int e = 0; e < kPairs; ++e) acc[g][e] = make_float2(0.0f, 0.0f);
        const int j_lo = sgm * kSegKeys, j_hi = min(Tl, j_lo + kSegKeys);
#pragma unroll 1
        for (int j0 = j_lo; j0 < j_hi; j0 += kKeys) {
            const uint32_t at = ring.used() - lane * 16 + lane * (4 * VW);
            if (ahead.item < n_items) {
                ring.template copy_v<VW>(vb, ahead, n_slices, D, lane);
                ahead.next(n_items, n_slices, Tl);
            }
            ring.issued();
#pragma unroll
            for (int p4 = 0; p4 < kKeys; p4 += 4) {
                if (j0 + p4 < j_hi) {
                    float vv[4][VW];
#pragma unroll
                    for (int pp = 0; pp < 4; ++pp) {
                        const uint32_t src = at + (p4 + pp) * (128 * VW);
                        if constexpr (VW == 4)
                            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(vv[pp][0]), "=f"(vv[pp][1]), "=f"(vv[pp][2]), "=f"(vv[pp][3]) : "r"(src));
                        else if constexpr (VW == 2)
                            asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(vv[pp][0]), "=f"(vv[pp][1]) : "r"(src));
                        else
                            asm volatile("ld.shared.f32 %0, [%1];" : "=f"(vv[pp][0]) : "r"(src));
                    }
                    float4 ew[G];                                // the weights of four keys (j0 is a multiple of 4)
#pragma unroll
                    for (int g = 0; g < G; ++g) ew[g] = *reinterpret_cast<const float4*>(e_s + g * Tc + j0 + p4);
                    auto add_key = [&](int pp) {
                        auto wt = [&](int g) { return pp == 0 ? ew[g].x : pp == 1 ? ew[g].y : pp == 2 ? ew[g].z : ew[g].w; };
                        if constexpr (VW > 1) {
#pragma unroll
                            for (int g = 0; g < G; ++g)
#pragma unroll
                                for (int e = 0; e < kPairs; ++e)
                                    acc[g][e] = __ffma2_rn(make_float2(wt(g), wt(g)), make_float2(vv[pp][2 * e], vv[pp][2 * e + 1]), acc[g][e]);
                        } else if constexpr (G > 1) {
#pragma unroll
                            for (int e = 0; e < kPairs; ++e)
                                acc[0][e] = __ffma2_rn(make_float2(wt(2 * e), wt(2 * e + 1)), make_float2(vv[pp][0], vv[pp][0]), acc[0][e]);
                        } else {
                            acc[0][0].x = __fmaf_rn(wt(0), vv[pp][0], acc[0][0].x);
                        }
                    };
                    if (j0 + p4 + 4 <= j_hi) {
#pragma unroll
                        for (int pp = 0; pp < 4; ++pp) add_key(pp);
                    } else {
#pragma unroll
                        for (int pp = 0; pp < 4; ++pp)
                            if (j0 + p4 + pp < j_hi) add_key(pp);        // keys beyond the segment are skipped
                    }
                }
            }
        }
        if (ok) {
#pragma unroll
            for (int g = 0; g < G; ++g) {
                float* dst = part + ((size_t)sgm * G + g) * D + d;
                if constexpr (VW > 1) {
#pragma unroll
                    for (int e = 0; e < kPairs; ++e) *reinterpret_cast<float2*>(dst + 2 * e) = acc[g][e];
                } else {
                    *dst = (g & 1) ? acc[0][g / 2].y : acc[0][g / 2].x;
                }
            }
        }
    }
}

// G: query heads per KV head (1, 2, 4 or 8); DC: 128-element chunks of the head dimension (1 or 2); NS: slots of the
// ring (0: loads through registers); VW: consecutive d per lane in P.V.
// Grid (C, B Hkv) in clusters of (C, 1, 1); Tc = keys per block (a multiple of 256), t_pitch = Tc.
template <int G, int DC, int NS, int VW>
__global__ void __launch_bounds__(kAttnThreads<NS>, kAttnBlocks<G, DC, NS>)
attention_decode_kernel(const float* __restrict__ q, const float* __restrict__ k, const float* __restrict__ v, float scale,
                        int Hq, int Hkv, int T, int D, int Tc, float* __restrict__ o)
{
    extern __shared__ __align__(16) float smem_f[];
    cg::cluster_group cluster = cg::this_cluster();
    const int C = (int)cluster.num_blocks();
    const int rank = (int)cluster.block_rank();
    // the same layout in every block of the cluster (remote addresses are computed from it)
    const int segs_per_block = Tc / kSegKeys;
    float* e_s = smem_f;                                       // [G][Tc]: scores, then weights, of the block's keys
    float* part = e_s + (size_t)G * Tc;                        // [segs_per_block][G][D]
    float* l_s = part + (size_t)segs_per_block * G * D;        // [16] denominators of the heads of this block
    float* red = l_s + 16;                                     // [8][kAttnWarps] the warps' row maxima, by head
    const uint32_t ring0 = ((uint32_t)__cvta_generic_to_shared(red + 8 * kAttnWarps) + kGroupBytes - 1) & ~(uint32_t)(kGroupBytes - 1);   // [kAttnWarps][NS] groups
    // The next kernel may start, and request its weights, only once what precedes this kernel is complete.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b = blockIdx.y / Hkv, hk = blockIdx.y % Hkv;
    const int j_begin = rank * Tc;                             // first key of this block
    const int Tl = max(0, min(T - j_begin, Tc));               // keys of this block
    const int n_seg = (T + kSegKeys - 1) / kSegKeys;           // segments of the row
    const int n_seg_l = (Tl + kSegKeys - 1) / kSegKeys;        // segments of this block
    const float* qb = q + ((size_t)b * Hq + (size_t)hk * G) * D;
    const float* kb = k + (((size_t)b * Hkv + hk) * (size_t)T + j_begin) * D;
    const float* vb = v + (((size_t)b * Hkv + hk) * (size_t)T + j_begin) * D;
    float* ob = o + ((size_t)b * Hq + (size_t)hk * G) * D;

    const int n_slices = (D + 32 * VW - 1) / (32 * VW);
    [[maybe_unused]] const int n_items = n_seg_l * n_slices;
    [[maybe_unused]] Ring<DC, NS < 2 ? 3 : NS> ring;
    [[maybe_unused]] VCursor<VW> ahead;

    // the lane's elements of a row of D floats: d = 128 c + 4 lane + jj (all four inside or outside D: D % 4 == 0)
    bool d_ok[DC];
#pragma unroll
    for (int c = 0; c < DC; ++c) d_ok[c] = 128 * c + 4 * lane < D;

    // ---- step 1: scores of the block's keys ----
    if (warp < kAttnWarps) {
        // (with the ring, the lane's own order of the heads: see ring_scores)
        const int head_perm = NS > 1 ? lane_perm<Scatter<(4 / DC) * G>::kSteps>(lane) % G : 0;
        float4 qv[G][DC];
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
            for (int c = 0; c < DC; ++c)
                qv[g][c] = d_ok[c] ? __ldg(reinterpret_cast<const float4*>(qb + (size_t)(g ^ head_perm) * D + 128 * c + 4 * lane)) : make_float4(0.f, 0.f, 0.f, 0.f);
        if constexpr (NS > 1) {
            ring.init(ring0 + warp * NS * kGroupBytes, lane);
            ahead.open(warp, n_items, n_slices, Tl);
            float m = ring_scores<G, DC, NS, VW>(ring, ahead, qv, d_ok, scale, kb, vb, e_s, Tc, Tl, D, n_items, n_slices, warp, lane);
            // the lanes that differ in their lowest bits only (those of the key) hold the same head
            constexpr int kKeyBits = DC == 1 ? 2 : 1;
#pragma unroll
            for (int i = 0; i < kKeyBits; ++i) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1 << i));
            if ((lane >> kKeyBits) < G && (lane & ((1 << kKeyBits) - 1)) == 0) red[head_perm * kAttnWarps + warp] = m;
        } else {
        constexpr int kKeysPerPass = kPassKeys<G, DC, NS>;
        float top[G];                                          // the lane's row maxima
#pragma unroll
        for (int g = 0; g < G; ++g) top[g] = -INFINITY;
        for (int j0 = warp * kKeysPerPass; j0 < Tl; j0 += kAttnWarps * kKeysPerPass) {
            float4 kv[kKeysPerPass][DC];
#pragma unroll
            for (int p = 0; p < kKeysPerPass; ++p)
#pragma unroll
                for (int c = 0; c < DC; ++c)
                    kv[p][c] = (j0 + p < Tl && d_ok[c]) ? __ldg(reinterpret_cast<const float4*>(kb + (size_t)(j0 + p) * D + 128 * c + 4 * lane))
                                                        : make_float4(0.f, 0.f, 0.f, 0.f);
            float a[kKeysPerPass * G];                          // value index p * G + g
#pragma unroll
            for (int p = 0; p < kKeysPerPass; ++p)
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    float acc = 0.0f;
#pragma unroll
                    for (int c = 0; c < DC; ++c) {
                        if (d_ok[c]) {                           // elements beyond D are skipped, not zero-filled
                            acc = __fmaf_rn(qv[g][c].x, kv[p][c].x, acc);
                            acc = __fmaf_rn(qv[g][c].y, kv[p][c].y, acc);
                            acc = __fmaf_rn(qv[g][c].z, kv[p][c].z, acc);
                            acc = __fmaf_rn(qv[g][c].w, kv[p][c].w, acc);
                        }
                    }
                    a[p * G + g] = acc;
                }
            lane_tree_scatter<kKeysPerPass * G>(a, lane);
            constexpr int NV = kKeysPerPass * G;
            constexpr int kSteps = Scatter<NV>::kSteps, kKeep = Scatter<NV>::kKeep;
            int base = 0;
            {
                int n = NV;
#pragma unroll
                for (int i = 0; i < kSteps; ++i) { n >>= 1; base += ((lane >> i) & 1) * n; }
            }
            if ((lane >> kSteps) == 0) {
#pragma unroll
                for (int t = 0; t < kKeep; ++t) {
                    const int idx = base + t, p = idx / G, g = idx % G;
                    if (j0 + p < Tl) e_s[g * Tc + j0 + p] = __fmul_rn(a[t], scale);
                }
            }
        }
        // every lane looks at scores of its warp's keys (written by this warp)
        __syncwarp();
        for (int j0 = warp * kKeysPerPass; j0 < Tl; j0 += kAttnWarps * kKeysPerPass)
            if (lane < kKeysPerPass && j0 + lane < Tl) {
#pragma unroll
                for (int g = 0; g < G; ++g) top[g] = fmaxf(top[g], e_s[g * Tc + j0 + lane]);
            }
#pragma unroll
        for (int g = 0; g < G; ++g) {
#pragma unroll
            for (int dlt = 4; dlt > 0; dlt >>= 1) top[g] = fmaxf(top[g], __shfl_xor_sync(0xffffffffu, top[g], dlt));
            if (lane == 0) red[g * kAttnWarps + warp] = top[g];
        }
        }
    }
    cluster.sync();                                            // every block's scores and its warps' maxima are in place

    // ---- step 2: row maxima (exact), from those of all warps of the cluster; step 3: weights of the block's keys.  (Reads
    // from the other blocks take some hundred cycles each: a lane per warp of the cluster, all heads at once.  Four
    // keys at a time: four exponentials side by side.) ----
    if (warp < kAttnWarps) {
        float m[G];
#pragma unroll
        for (int g = 0; g < G; ++g) m[g] = -INFINITY;
        for (int i = lane; i < C * kAttnWarps; i += 32) {
            const float* src = cluster.map_shared_rank(red, i / kAttnWarps) + i % kAttnWarps;
#pragma unroll
            for (int g = 0; g < G; ++g) m[g] = fmaxf(m[g], src[g * kAttnWarps]);
        }
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
            for (int dlt = 16; dlt > 0; dlt >>= 1) m[g] = fmaxf(m[g], __shfl_xor_sync(0xffffffffu, m[g], dlt));
#pragma unroll
        for (int g = 0; g < G; ++g)
            for (int j = 4 * (int)threadIdx.x; j < Tl; j += 4 * kWorkThreads) {      // (keys beyond Tl in the last quad: nobody reads them)
                float4* p = reinterpret_cast<float4*>(e_s + g * Tc + j);
                const float4 sc = *p;
                *p = make_float4(exp_det(__fsub_rn(sc.x, m[g])), exp_det(__fsub_rn(sc.y, m[g])), exp_det(__fsub_rn(sc.z, m[g])),
                                 exp_det(__fsub_rn(sc.w, m[g])));
            }
    }
    cluster.sync();                                            // every block's weights are in place

    // ---- step 4: denominators (head g in block g mod C), with the ring by a warp of their own while the others go on; the 32
    // chains of a sum are a warp's lanes and run over ALL keys in ascending chunks of 128, reading the other blocks' weights in
    // place, eight chunks at a time (a read from another block takes as long as some hundred instructions) ----
    if (NS == 0 || warp == kAttnWarps) {
        for (int g = rank + (NS == 0 ? C * warp : 0); g < G; g += NS == 0 ? C * kAttnWarps : C) {
            float a = 0.0f;
            int owner = 0, c = 0;                              // next chunk: block and first key in the block
            for (int k0 = 0; k0 < T; k0 += 1024) {
                float4 ev[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    if (k0 + 128 * u < T) {
                        ev[u] = *reinterpret_cast<const float4*>(cluster.map_shared_rank(e_s, owner) + g * Tc + c + 4 * lane);
                        c += 128;
                        if (c == Tc) { c = 0; ++owner; }
                    }
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int j = k0 + 128 * u + 4 * lane;     // keys beyond T are skipped
                    if (j < T) a = __fadd_rn(a, ev[u].x);
                    if (j + 1 < T) a = __fadd_rn(a, ev[u].y);
                    if (j + 2 < T) a = __fadd_rn(a, ev[u].z);
                    if (j + 3 < T) a = __fadd_rn(a, ev[u].w);
                }
            }
            a = lane_tree_sum(a);
            if (lane == 0) l_s[g] = a;
        }
    }

    // ---- step 5: P.V.  A work item is (256-key segment of the block, slice of 32 VW consecutive d): a lane owns VW
    // consecutive d and runs their G chains a = fma(e_j, v_j[d], a) over the segment's keys in ascending order.
    // Items are dealt to the warps round robin; the slices are as wide as still leaves every warp an item, so a
    // block with two segments keeps all eight warps loading and a block with many uses 16-byte loads ----
    if (warp < kAttnWarps) {
        if constexpr (NS > 1) ring_pv<G, DC, NS, VW>(ring, ahead, e_s, part, vb, Tc, Tl, D, n_items, n_slices, warp, lane);
        else pv_items<G, VW>(e_s, part, vb, Tc, Tl, D, n_seg_l, warp, lane);
    }
    cluster.sync();                                            // segment sums and denominators are in place

    // ---- fold the segment sums in ascending order, divide: block r takes the r-th slice of the G D outputs ----
    {
        const int per = (G * D + C - 1) / C;
        const int i_lo = rank * per, i_hi = min(G * D, i_lo + per);
        for (int i = i_lo + (int)threadIdx.x; i < i_hi; i += kAttnThreads<NS>) {
            const int g = i / D;
            const float l = cluster.map_shared_rank(l_s, g % C)[g];
            float t = 0.0f;
            int owner = 0, sl = 0;                             // next segment: block and number in the block
            for (int s0 = 0; s0 < n_seg; s0 += 8) {
                float pv[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    if (s0 + u < n_seg) {
                        pv[u] = cluster.map_shared_rank(part, owner)[(size_t)sl * G * D + i];
                        if (++sl == segs_per_block) { sl = 0; ++owner; }
                    }
                }
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (s0 + u < n_seg) t = (s0 + u == 0) ? pv[u] : __fadd_rn(t, pv[u]);
            }
            ob[i] = __fdiv_rn(t, l);
        }
    }
    cluster.sync();                                            // nobody leaves while its shared memory may still be read
}

int g_attention_force_split = 0;        // test hook: 0 = automatic, else the cluster size to use (1, 2, 4, 8)

// shared memory of one block that owns Tc keys
size_t block_smem_bytes(int G, int Tc, int D)
{
    return 4 * ((size_t)G * Tc + (size_t)(Tc / kSegKeys) * G * D + 16 + (size_t)kAttnWarps * 8);
}

// keys per block for a cluster of C blocks: the row's 256-key segments dealt out in equal whole numbers
int keys_per_block(int T, int C)
{
    const int n_seg = (T + kSegKeys - 1) / kSegKeys;
    return (n_seg + C - 1) / C * kSegKeys;
}

// Slots of the ring beside a block's other shared memory: as many as fit with two blocks on an SM.  (Never more, even for few
// blocks: with one block to an SM a cluster of 8 wants 8 whole SMs of a GPC, and not all of 16 clusters fit at once: B = 2,
// T = 4096 40 -> 62 us with 8 slots.)
int ring_slots(size_t base)
{
    const size_t limit = 111u * 1024u - kGroupBytes, slot = (size_t)kAttnWarps * kGroupBytes;
    return base + 5 * slot <= limit ? 5 : base + 3 * slot <= limit ? 3 : 0;
}

// The ring's slots, or 0 or 1 for loads through registers (see kAttnThreads).  Times in us on 148 SMs.
int ring_or_registers(int G, int DC, int D, int Tc, long long blocks, int sm_count, int slots)
{
    const int work = G * DC;                         // float4s of q a lane holds
    // Few blocks of a single segment each: half of the warps have no P.V item and the others' 256 keys are one chain of loads and
    // additions, which starts sooner through registers (32 / 8 heads, D = 128: B = 1, T = 512 14.6, with the ring 17.1; but B = 4,
    // T = 1024, 128 blocks, 24.2 and 21.2).  A ninth warp takes 0.3 off where it leaves eight keys their registers.
    if (Tc <= kSegKeys && blocks <= sm_count / 2) return work < 8 ? 1 : 0;
    // Many blocks with little to do, or rows of half a chunk, which fill half of a ring: four blocks to an SM without the ring's
    // shared memory (16 / 8 heads, D = 128, B = 64: T = 64 13.6 and 17.8 with the ring, T = 512 53.0 and 58.5; 32 / 32, D = 64, B = 16,
    // T = 8192 333 and 435; but 32 / 32, D = 128, B = 16, T = 4096 3.5 % slower)
    if (work <= 2 && blocks > 2 * sm_count && (Tc <= 1024 || D <= 64)) return 0;
    if (work >= 16) {
        // Eight heads of more than 128 elements take 168 registers for eight keys in flight: one block to an SM, the better form where
        // one is enough (64 / 8, D = 256: B = 4, T = 1024 34.1, with the ring 44.2; B = 1, T = 8192 83.5, with two keys in flight
        // and two blocks to an SM 182) ...
        if (blocks <= sm_count) return 0;
        // ... and where not even two make it a single wave (B = 16, T = 4096 325 and 420); in between 248 and 213 (B = 4, T = 8192)
        if (slots == 0) return blocks <= 2 * sm_count ? 1 : 0;
    }
    // no room for a ring (eight heads, D = 128, B = 16, T = 4096 138 by eight warps, 193 by nine with four keys in flight; four
    // heads, B = 8, T = 32768 393 and 384 with eight keys in flight either way)
    if (slots == 0) return work < 8 ? 1 : 0;
    return slots;
}

template <int G, int DC, int NS, int VW>
cudaError_t launch_variant(const cudaLaunchConfig_t* cfg, bool query, const float* q, const float* k, const float* v, float scale, int Hq, int Hkv, int T, int D,
                           int Tc, float* o)
{
    static bool configured[kMaxDevices];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    auto kern = attention_decode_kernel<G, DC, NS, VW>;
    if (!configured[dev]) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);   // clusters of 16
        if (e != cudaSuccess) return e;
        configured[dev] = true;
    }
    if (query) {
        int n_clusters = 0;
        e = cudaOccupancyMaxActiveClusters(&n_clusters, kern, cfg);
        return e != cudaSuccess ? e : n_clusters >= 1 ? cudaSuccess : cudaErrorLaunchOutOfResources;
    }
    return cudaLaunchKernelEx(cfg, kern, q, k, v, scale, Hq, Hkv, T, D, Tc, o);
}

template <int G, int DC>
cudaError_t launch_attention_t(const float* q, const float* k, const float* v, float scale, int B, int Hq, int Hkv, int T, int D,
                               float* o, int C, int sm_count, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[2];
    for (;;) {
        const int Tc = keys_per_block(T, C);
        const size_t base = block_smem_bytes(G, Tc, D);
        if (base > 227u * 1024u) return cudaErrorLaunchOutOfResources;
        const int ns = ring_or_registers(G, DC, D, Tc, (long long)C * B * Hkv, sm_count, ring_slots(base));
        // P.V items: (segment, slice of 32 VW consecutive d), the widest slices that still give every warp of a block an item
        const int segs = Tc / kSegKeys;
        const int vw = segs * ((D + 127) / 128) >= kAttnWarps ? 4 : segs * ((D + 63) / 64) >= kAttnWarps ? 2 : 1;
        cfg.gridDim = dim3((unsigned)C, (unsigned)(B * Hkv));
        cfg.blockDim = dim3(ns ? kAttnThreads<1> : kAttnThreads<0>);
        cfg.dynamicSmemBytes = base + (ns > 1 ? (size_t)ns * kAttnWarps * kGroupBytes + kGroupBytes : 0);     // + alignment
        cfg.stream = stream;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)C;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        auto go = [&](bool query) -> cudaError_t {
            cfg.numAttrs = query ? 1 : 2;
#define DET_ATTN_V(NS_, VW_) return launch_variant<G, DC, NS_, VW_>(&cfg, query, q, k, v, scale, Hq, Hkv, T, D, Tc, o)
#define DET_ATTN_N(NS_) { if (vw == 4) DET_ATTN_V(NS_, 4); if (vw == 2) DET_ATTN_V(NS_, 2); DET_ATTN_V(NS_, 1); }
            if (ns == 5) DET_ATTN_N(5)
            if (ns == 3) DET_ATTN_N(3)
            if constexpr (G * DC != 8) { if (ns == 1) DET_ATTN_N(1) }
            if constexpr (G * DC != 4) DET_ATTN_N(0)      // (never without the ninth warp)
            return cudaErrorInvalidValue;
#undef DET_ATTN_N
#undef DET_ATTN_V
        };
        // a cluster this large may not fit where the stream runs (few SMs, a partition): halve it while the scores
        // of a block still fit (schedule only: same bits)
        const cudaError_t e = go(true);
        if (e == cudaSuccess) return go(false);
        cudaGetLastError();
        if (C == 1) return e;
        C /= 2;
    }
}

}  // namespace

// Cluster size for a shape: the largest power of two that still lets all blocks be resident at once (two blocks of
// 256 threads per SM: one wave, measured best at about 256 blocks on 148 SMs), never more blocks than the row has
// segments, and at least as many as it takes for a block's scores and segment sums to fit in the shared memory
// that lets two blocks share an SM (or in a block's maximum, if that is all that fits).  Schedule only.
int attention_split(int B, int Hkv, int G, int T, int D, int sm_count)
{
    const int n_seg = (T + kSegKeys - 1) / kSegKeys;
    int c_max = 1;
    while (c_max < kMaxCluster && 2 * c_max <= n_seg) c_max *= 2;
    if (g_attention_force_split) return g_attention_force_split <= c_max ? g_attention_force_split : c_max;
    // clusters of 16 (not portable, one GPC each) only pay for very few, very long rows (measured: 8 rows of 16384 keys
    // or more; 16 rows, or 4096 keys, are faster in clusters of 8)
    const bool few_long_rows = (long long)B * Hkv * 16 <= sm_count && n_seg >= 64;
    const int c_auto = (c_max > 8 && !few_long_rows) ? 8 : c_max;
    int c = 1;
    while (c < c_auto && (long long)B * Hkv * (2 * c) <= 2ll * sm_count) c *= 2;
    while (c < c_max && block_smem_bytes(G, keys_per_block(T, c), D) > 110u * 1024u) c *= 2;
    return c;
}

// Dynamic shared memory of a block for the most finely split schedule the shape allows (the least the shape needs).
size_t attention_smem_bytes(int G, int T, int D)
{
    const int n_seg = (T + kSegKeys - 1) / kSegKeys;
    int c_max = 1;
    while (c_max < kMaxCluster && 2 * c_max <= n_seg) c_max *= 2;
    return block_smem_bytes(G, keys_per_block(T, c_max), D);
}

size_t attention_block_smem_bytes(int G, int T, int D, int C) { return block_smem_bytes(G, keys_per_block(T, C), D); }

void attention_test_force_split(int c) { g_attention_force_split = (c == 1 || c == 2 || c == 4 || c == 8 || c == 16) ? c : 0; }

cudaError_t launch_attention_decode(const float* q, const float* k, const float* v, float scale, int B, int Hq, int Hkv, int T, int D,
                                    float* o, cudaStream_t stream)
{
    const int G = Hq / Hkv;
    const int dc = (D + 127) / 128;
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
        sms = 148;
    int C = attention_split(B, Hkv, G, T, D, sms);
    while (C < kMaxCluster && block_smem_bytes(G, keys_per_block(T, C), D) > 227u * 1024u) C *= 2;   // must fit at all
    if (block_smem_bytes(G, keys_per_block(T, C), D) > 227u * 1024u) return cudaErrorInvalidValue;
#define DET_ATTN(GG, DD) return launch_attention_t<GG, DD>(q, k, v, scale, B, Hq, Hkv, T, D, o, C, sms, stream)
    if (dc == 1) {
        switch (G) { case 1: DET_ATTN(1, 1); case 2: DET_ATTN(2, 1); case 4: DET_ATTN(4, 1); case 8: DET_ATTN(8, 1); default: break; }
    } else if (dc == 2) {
        switch (G) { case 1: DET_ATTN(1, 2); case 2: DET_ATTN(2, 2); case 4: DET_ATTN(4, 2); case 8: DET_ATTN(8, 2); default: break; }
    }
#undef DET_ATTN
    return cudaErrorInvalidValue;
}

}  // namespace detlin
