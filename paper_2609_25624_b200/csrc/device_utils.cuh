// Device helpers shared by the kernels: the register upcast of Eq. 2 for each weight format and the
// adjacent-first lane tree.  (Rule R1: every multiply-accumulate in the kernels is an explicit fma
// intrinsic -- __fmaf_rn, __ffma2_rn -- never the compiler's contraction.)
#pragma once
#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cstdint>

namespace detlin {

// Weight formats: WF = 0 BF16, 1 FP16, 2 FP32 (det_weight_format_t).  A 32-bit word of a 16-bit
// format holds elements (k, k+1) in its (low, high) half; both widenings are exact.
template <int WF>
__device__ __forceinline__ float up16_lo(uint32_t w)
{
    if (WF == 0) return __uint_as_float(__byte_perm(w, 0u, 0x1044));       // (faster than the shift: 82.5 against 80 % in the decode loop)
    return __half2float(__ushort_as_half((unsigned short)(w & 0xffffu)));
}
template <int WF>
__device__ __forceinline__ float up16_hi(uint32_t w)
{
    if (WF == 0) return __uint_as_float(w & 0xffff0000u);
    return __half2float(__ushort_as_half((unsigned short)(w >> 16)));
}
template <int WF> struct WeightElem { typedef uint16_t type; static constexpr int bytes = 2; };
template <> struct WeightElem<2> { typedef float type; static constexpr int bytes = 4; };
template <int WF>
__device__ __forceinline__ float up_elem(typename WeightElem<WF>::type v)
{
    if constexpr (WF == 2) return v;
    else if constexpr (WF == 1) return __half2float(__ushort_as_half(v));
    else return __uint_as_float(((uint32_t)v) << 16);
}

// d = x * w + d in both halves, each an IEEE fma.rn.f32; volatile: keeps its place in the instruction order
__device__ __forceinline__ void fma2(float2& d, float x, const float2& w)
{
    asm volatile("{\n\t.reg .b64 a, b, c;\n\tmov.b64 a, {%2, %2};\n\tmov.b64 b, {%3, %4};\n\tmov.b64 c, {%0, %1};\n\t"
                 "fma.rn.f32x2 c, a, b, c;\n\tmov.b64 {%0, %1}, c;\n\t}"
                 : "+f"(d.x), "+f"(d.y) : "f"(x), "f"(w.x), "f"(w.y));
}

// Balanced tree over the 32 lanes of a warp, adjacent lanes first (xor 1, 2, 4, 8, 16 in that
// order).  fadd is commutative, so both partners compute identical bits and every lane ends with
// the tree's root.
__device__ __forceinline__ float lane_tree_sum(float a)
{
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) a = __fadd_rn(a, __shfl_xor_sync(0xffffffffu, a, d));
    return a;
}

// Butterfly reduce-scatter that realises the adjacent-first lane tree for NV values per lane at once.  At
// step i (i = 0..4) lanes l and l ^ (1 << i) are partners.  While the number of values a lane holds is
// even, the partners exchange halves and add (the lane with bit i set keeps the upper half), so the work
// per step halves; afterwards the remaining steps add whole arrays.  kSteps = number of halving steps,
// kKeep = values a lane holds at the end (v[0 .. kKeep)); they are the sums of the values with index
// base + t, base = sum over halving steps i of bit_i(lane) * (NV >> (i + 1)); lanes whose bits
// kSteps .. 4 are zero hold distinct results.
template <int NV>
struct Scatter {
    static constexpr int steps()
    {
        int n = NV, h = 0;
        while (h < 5 && n % 2 == 0) { n /= 2; ++h; }
        return h;
    }
    static constexpr int kSteps = steps();
    static constexpr int kKeep = NV >> kSteps;
};

template <int NV>
__device__ __forceinline__ void lane_tree_scatter(float (&v)[NV], int lane)
{
    constexpr int H = Scatter<NV>::kSteps;
    int n = NV;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const int d = 1 << i;
        if (i < H) {
            const int half = n >> 1;
            const bool hi = (lane >> i) & 1;
#pragma unroll
            for (int t = 0; t < NV / 2; ++t) {
                if (t < half) {
                    const float send = hi ? v[t] : v[t + half];
                    const float keep = hi ? v[t + half] : v[t];
                    v[t] = __fadd_rn(keep, __shfl_xor_sync(0xffffffffu, send, d));
                }
            }
            n = half;
        } else {
#pragma unroll
            for (int t = 0; t < Scatter<NV>::kKeep; ++t) v[t] = __fadd_rn(v[t], __shfl_xor_sync(0xffffffffu, v[t], d));
        }
    }
}

}  // namespace detlin
