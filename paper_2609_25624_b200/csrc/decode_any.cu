// Decode order (V=4, L=32, P=1, S segments) for any K and any alignment (K % 8 != 0, misaligned buffers); compiled once per
// weight format (DET_WF = 0 BF16, 1 FP16, 2 FP32).
//
// A warp owns RT weight rows and MT batch rows: lane l owns k = c + 4l + j in every 128-element chunk of a segment and
// accumulates them in ascending order into one chain per output; the 32 lane sums of an output are added adjacent-first;
// segment sums are added in ascending order as the warp goes (rule R3).
//
// What bounds it: with rows that start anywhere, TMA and vector loads are out, and a warp that walks its row chunk by
// chunk waits for memory every time.
//   * weights go from memory to registers, a group of UC chunks of every row loaded ahead of the group that is
//     being multiplied.  16-bit rows start on any 2-byte boundary: a lane loads the two or three aligned words that hold
//     its four weights, two byte permutations line them up (rows at the very ends of W, where such a word would reach
//     outside of W, and the last partial chunk of a row are loaded element by element);
//   * activations sit in shared memory, rows padded to whole chunks; the warps of a block share them.  The padding is
//     -0.0 and weights beyond K count as +0: the product is -0.0, and adding -0.0 changes no accumulator (not even a
//     -0.0 one), so elements beyond K are skipped in effect without a test in the loop;
//   * two rows' chains advance in one packed FMA (RT > 1), the lane sums of all outputs fold in one butterfly.
//   * a small layer is one wave of warps that wait for their own instructions: batch blocks of fewer rows and a warp per segment
//     spread them over the SMs (decode_any_layout.cpp).
// Measured on B200, us a call in a chain (in brackets a warp per row that walks it chunk by chunk, for every batch row again): M = 6, N =
// 1333, K = 1001 4.1 (15.8); M = 3, N = K = 4097 13.1 (49.6); M = 64, N = 8192, K = 4097 214 (1705; 27 % of the FP32 peak: line-up and
// widening of every weight in every batch block, one-word loads); M = 64, N = 300, K = 333 4.1 (68).
#include "internal.h"
#include "device_utils.cuh"

namespace detlin {

namespace {

// SPLIT: the two segments of a row belong to two warps, the second half of the block's warps to the second ones.
// WINDOWS: shared memory does not hold the activations' whole K.  A kernel of its own: where all of K is there, the window's bookkeeping
// in the loop costs registers that spill (M = 26, N = 4857, K = 2669 with FP32 weights 70.6 -> 58.4 us, M = 58, N = 9341, K = 4893 367 ->
// 323; over 180 shapes in one layout each 0.88 of the time).
template <int WF, int MT, int RT, bool SPLIT, bool WINDOWS>
__global__ void __launch_bounds__(512, 1)
decode_any_kernel(const float* __restrict__ x, const typename WeightElem<WF>::type* __restrict__ W, const float* __restrict__ b,
                  float* __restrict__ y, int M, int N, unsigned K, unsigned seg_len, long long ldy, unsigned win, int groups)
{
    typedef typename WeightElem<WF>::type WT;
    constexpr int UC = 8 / RT;                       // chunks of a row loaded together
    constexpr int NW = WF == 2 ? 4 : 3;              // words a lane loads of a chunk
    extern __shared__ __align__(16) float xs[];      // [MT][win]
    const int lane = threadIdx.x & 31, threads = blockDim.x;
    const int rows_of_warps = threads >> (SPLIT ? 6 : 5);     // warps that have rows of their own
    const int warp = SPLIT ? (int)(threadIdx.x >> 5) % rows_of_warps : (int)(threadIdx.x >> 5);
    const bool second = SPLIT && (int)(threadIdx.x >> 5) >= rows_of_warps;
    const int m0 = blockIdx.y * MT;
    // The next kernel may start, and request its weights, only once what precedes this kernel is complete.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // Activations of the window [w_lo, w_lo + win) into shared memory.  All of K, once, for few rows of weights as a rule: column by
    // column, the batch rows' copies of a column one after the other, under the first weights' way from memory.  Window by window: row
    // by row (M = 16, N = 12155, K = 7337 with FP32 weights 213 us, by columns 229; M = 31, N = 2057, K = 7807 69 and 74).
    auto stage = [&](unsigned w_lo) {
        const unsigned len = min(win, K - w_lo);
        const uint32_t base = (uint32_t)__cvta_generic_to_shared(xs);
        if constexpr (WINDOWS) {
#pragma unroll 1
            for (int m = 0; m < MT; ++m) {
                const float* src = x + (size_t)min(m0 + m, M - 1) * K + w_lo;     // rows beyond M repeat the last one
#pragma unroll 4
                for (unsigned i = threadIdx.x; i < len; i += threads)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(base + (m * win + i) * 4u), "l"(src + i) : "memory");
                for (unsigned i = len + threadIdx.x; i < win; i += threads) xs[m * win + i] = -0.0f;
            }
        } else {
            for (unsigned i = threadIdx.x; i < win; i += threads) {
                const float* src = x + (size_t)m0 * K + i;
                if (i < len) {
#pragma unroll
                    for (int m = 0; m < MT; ++m) {
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(base + (m * win + i) * 4u), "l"(src) : "memory");
                        if (m0 + m + 1 < M) src += K;    // (likewise)
                    }
                } else {
#pragma unroll
                    for (int m = 0; m < MT; ++m) xs[m * win + i] = -0.0f;
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto staged = [&]() {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
    };

    // (With WINDOWS never so, which the launcher knows.  Asked all the same: without it the compiler keeps other registers, M = 16, N =
    // 3796, K = 8841 with FP16 weights 94 -> 121 us, M = 32, N = 4096, K = 14335 256 -> 288.)
    [[maybe_unused]] const bool one_window = K <= win;
    if constexpr (!WINDOWS) stage(0);
    for (int grp = (int)blockIdx.x; grp < groups; grp += (int)gridDim.x) {
        const int n0 = (grp * rows_of_warps + warp) * RT;

        // The warp's rows, as the word that holds the lane's first weight, and how the lane's words are lined up: bytes
        // 0 .. 3 of two words for rows that start on a word, bytes 2 .. 5 for the others.  A warp with a row at
        // which such a word could reach outside of W loads by elements.
        const uint32_t* pw[RT];
        uint32_t sel[RT];
        bool by_word = true;
#pragma unroll
        for (int r = 0; r < RT; ++r) {
            const int n = min(n0 + r, N - 1);        // rows beyond N repeat the last one; their sums are not stored
            const uintptr_t at = reinterpret_cast<uintptr_t>(W + (size_t)n * K + 4 * lane);
            const bool odd = WF != 2 && (at & 2u) != 0;
            pw[r] = reinterpret_cast<const uint32_t*>(at & ~(uintptr_t)3);
            sel[r] = odd ? 0x5432u : 0x3210u;
            if (odd && (n == 0 || n == N - 1)) by_word = false;
        }
        uint32_t raw[2][UC][RT][NW];
        // one chunk of every row, `u` chunks behind the words' position, by words
        auto load_words = [&](uint32_t (&v)[RT][NW], int u) {
#pragma unroll
            for (int r = 0; r < RT; ++r) {
                if constexpr (WF == 2) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) v[r][j] = __ldg(pw[r] + 128 * u + j);
                } else {
                    v[r][0] = __ldg(pw[r] + 64 * u);
                    v[r][1] = __ldg(pw[r] + 64 * u + 1);
                    if (sel[r] == 0x5432u) v[r][2] = __ldg(pw[r] + 64 * u + 2);
                }
            }
        };
        // the chunks of [c, end): whole ones by words, a partial one by elements; the words advance
        auto load = [&](uint32_t (&v)[UC][RT][NW], unsigned c, unsigned end) {
            if (by_word && end - c == 128 * UC) {
#pragma unroll
                for (int u = 0; u < UC; ++u) load_words(v[u], u);
            } else {
#pragma unroll
                for (int u = 0; u < UC; ++u) {
                    if (by_word && c + 128 * u + 128 <= end) load_words(v[u], u);
                    else if (c + 128 * u < end) {
                        const unsigned k = c + 128 * u + 4 * lane;
#pragma unroll
                        for (int r = 0; r < RT; ++r) {
                            const WT* p = W + (size_t)min(n0 + r, N - 1) * K + k;
                            uint32_t e[4];
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                if constexpr (WF == 2) e[j] = k + j < end ? __float_as_uint(__ldg(p + j)) : 0u;
                                else e[j] = k + j < end ? (uint32_t)__ldg(p + j) : 0u;
                            }
                            if constexpr (WF == 2) {
#pragma unroll
                                for (int j = 0; j < 4; ++j) v[u][r][j] = e[j];
                            } else {
                                v[u][r][0] = e[0] | (e[1] << 16);
                                v[u][r][1] = e[2] | (e[3] << 16);
                            }
                        }
                    }
                }
            }
            const unsigned step = (end - c) * sizeof(WT) / 4;        // (a partial chunk is the row's last: not used after it)
#pragma unroll
            for (int r = 0; r < RT; ++r) pw[r] += step;
        };
        float acc[MT][RT];
        float tot[Scatter<MT * RT>::kKeep];
        auto multiply = [&](const uint32_t (&v)[RT][NW], const float* xl, bool words) {
            float w[RT][4];
#pragma unroll
            for (int r = 0; r < RT; ++r) {
                if constexpr (WF == 2) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) w[r][j] = __uint_as_float(v[r][j]);
                } else {
                    const uint32_t sl = words ? sel[r] : 0x3210u;
                    const uint32_t lo = __byte_perm(v[r][0], v[r][1], sl), hi = __byte_perm(v[r][1], v[r][2], sl);
                    w[r][0] = up16_lo<WF>(lo); w[r][1] = up16_hi<WF>(lo);
                    w[r][2] = up16_lo<WF>(hi); w[r][3] = up16_hi<WF>(hi);
                }
            }
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                const float4 xv = *reinterpret_cast<const float4*>(xl + m * win);
                const float xk[4] = {xv.x, xv.y, xv.z, xv.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if constexpr (RT == 1) {
                        acc[m][0] = __fmaf_rn(xk[j], w[0][j], acc[m][0]);
                    } else {
#pragma unroll
                        for (int r = 0; r < RT; r += 2) {
                            const float2 t = __ffma2_rn(make_float2(xk[j], xk[j]), make_float2(w[r][j], w[r + 1][j]), make_float2(acc[m][r], acc[m][r + 1]));
                            acc[m][r] = t.x;
                            acc[m][r + 1] = t.y;
                        }
                    }
                }
            }
        };

        // groups of up to UC chunks, never across the end of a segment or of a window
        auto group_end = [&](unsigned c, unsigned s_hi, unsigned w_hi) { return min(min(K, s_hi), WINDOWS ? min(w_hi, c + 128 * UC) : c + 128 * UC); };
        bool first = true;                           // no segment has ended yet
        unsigned w_hi = win, w_lo = ~0u;             // end of the window of the group loaded last; start of the one in shared memory
        unsigned s_hi = second ? 2 * seg_len : seg_len;      // end of the segment of the group being multiplied
        unsigned c = second ? seg_len : 0, c_end = group_end(c, s_hi, w_hi);
        const unsigned c_stop = SPLIT && !second ? seg_len : K;
        if (second) {
#pragma unroll
            for (int r = 0; r < RT; ++r) pw[r] += seg_len * (unsigned)sizeof(WT) / 4;
        }
        load(raw[0], c, c_end);
        if (!WINDOWS && grp == (int)blockIdx.x) staged();
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int r = 0; r < RT; ++r) acc[m][r] = 0.0f;
        int buf = 0;
#pragma unroll 1
        while (c < c_stop) {
            if constexpr (WINDOWS) {
                if (one_window ? (w_lo != 0 && grp == (int)blockIdx.x) : (w_lo == ~0u || c - w_lo >= win)) {
                    w_lo = one_window ? 0 : c;
                    __syncthreads();                 // everybody has finished with the window before
                    stage(w_lo);
                    staged();
                }
            }
            const bool seg_done = c_end == min(K, s_hi);
            if (seg_done) s_hi += seg_len;
            if (WINDOWS && c_end == w_hi) w_hi += win;
            const unsigned nc_end = c_end < c_stop ? group_end(c_end, s_hi, w_hi) : c_end;
            const float* xl = xs + (!WINDOWS || one_window ? c : c - w_lo) + 4 * lane;
#pragma unroll
            for (int half = 0; half < 2; ++half) {   // (the buffers are registers: their index has to be a constant)
                if (buf == half) {
                    if (nc_end != c_end) load(raw[half ^ 1], c_end, nc_end);
                    if (c_end - c == 128 * UC) {
#pragma unroll
                        for (int u = 0; u < UC; ++u) multiply(raw[half][u], xl + 128 * u, by_word);
                    } else {
#pragma unroll
                        for (int u = 0; u < UC; ++u)
                            if (c + 128 * u < c_end) multiply(raw[half][u], xl + 128 * u, by_word && c + 128 * u + 128 <= c_end);
                    }
                }
            }
            buf ^= 1;
            if (seg_done) {
                float v[MT * RT];
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int r = 0; r < RT; ++r) { v[m * RT + r] = acc[m][r]; acc[m][r] = 0.0f; }
                lane_tree_scatter<MT * RT>(v, lane);
#pragma unroll
                for (int t = 0; t < Scatter<MT * RT>::kKeep; ++t) tot[t] = first ? v[t] : __fadd_rn(tot[t], v[t]);
                first = false;
            }
            c = c_end;
            c_end = nc_end;
        }
        constexpr int kSteps = Scatter<MT * RT>::kSteps, kKeep = Scatter<MT * RT>::kKeep;
        static_assert(!SPLIT || kKeep == 1, "room for one sum a lane");
        if constexpr (SPLIT) {
            // the second segments' sums meet the first ones' in shared memory, behind the activations
            float* sums = xs + MT * win + (warp * kKeep << 5) + lane;
            if (second) {
#pragma unroll
                for (int t = 0; t < kKeep; ++t) sums[t << 5] = tot[t];
            }
            __syncthreads();
            if (!second) {
#pragma unroll
                for (int t = 0; t < kKeep; ++t) tot[t] = __fadd_rn(tot[t], sums[t << 5]);
            }
            if (grp + (int)gridDim.x < groups) __syncthreads();
        }
        if (!second && (lane >> kSteps) == 0) {
            int base = 0, cnt = MT * RT;
#pragma unroll
            for (int i = 0; i < kSteps; ++i) { cnt >>= 1; base += ((lane >> i) & 1) * cnt; }
#pragma unroll
            for (int t = 0; t < kKeep; ++t) {
                const int idx = base + t;
                const int m = m0 + idx / RT, n = n0 + idx % RT;
                if (m < M && n < N) y[m * ldy + n] = b ? __fadd_rn(tot[t], __ldg(b + n)) : tot[t];
            }
        }
    }
}

template <int WF, int MT, int RT, bool SPLIT, bool WINDOWS>
cudaError_t launch_w(const LaunchArgs& a, const AnyGrid& g)
{
    static bool configured[kMaxDevices];             // function attributes belong to a device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    auto kern = decode_any_kernel<WF, MT, RT, SPLIT, WINDOWS>;
    if (!configured[dev]) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kAnySmemBytes1);
        if (e != cudaSuccess) return e;
        configured[dev] = true;
    }
    const unsigned win = (unsigned)g.window;
    const int64_t grid = a.max_blocks > 0 && g.blocks_x > a.max_blocks ? a.max_blocks : g.blocks_x;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    cfg.gridDim = dim3((unsigned)grid, (unsigned)g.batch_blocks);
    cfg.blockDim = dim3(32 * g.warps);
    cfg.dynamicSmemBytes = (size_t)MT * win * 4 + (SPLIT ? kAnySplitBytes : 0);
    cfg.stream = a.stream;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, a.x, static_cast<const typename WeightElem<WF>::type*>(a.W), a.b, a.y, (int)a.M, (int)a.N,
                              (unsigned)a.K, (unsigned)a.seg_len, (long long)a.ldy, win, (int)g.groups);
}

template <int WF, int MT, int RT, bool SPLIT>
cudaError_t launch_t(const LaunchArgs& a, int sms)
{
    const AnyGrid g = any_grid({MT, RT, SPLIT}, a.M, a.N, a.K, sms);
    if constexpr (!SPLIT) {
        if (g.window < a.K) return launch_w<WF, MT, RT, SPLIT, true>(a, g);
    }
    return launch_w<WF, MT, RT, SPLIT, false>(a, g);
}

template <int WF, int MT>
cudaError_t launch_m(const LaunchArgs& a, int sms)
{
    const AnyLayout& l = a.any_layout;
    if constexpr (MT < 8) {
        if (l.split) {
            if constexpr (MT == 4) {
                if (l.rt == 4) return launch_t<WF, MT, 4, true>(a, sms);
            }
            return l.rt == 2 ? launch_t<WF, MT, 2, true>(a, sms) : launch_t<WF, MT, 1, true>(a, sms);
        }
    }
    if (l.rt == 4) return launch_t<WF, MT, 4, false>(a, sms);
    return l.rt == 2 ? launch_t<WF, MT, 2, false>(a, sms) : launch_t<WF, MT, 1, false>(a, sms);
}

}  // namespace

#define DET_CAT2(a, b) a##b
#define DET_CAT(a, b) DET_CAT2(a, b)
cudaError_t DET_CAT(launch_decode_any_wf, DET_WF)(const LaunchArgs& a)
{
    const int sms = a.sm_count > 0 ? a.sm_count : 148;
    if (!any_layout_fits(a.any_layout, a.K, a.S)) return cudaErrorInvalidValue;
    switch (a.any_layout.mt) {
    case 1: return launch_m<DET_WF, 1>(a, sms);
    case 2: return launch_m<DET_WF, 2>(a, sms);
    case 4: return launch_m<DET_WF, 4>(a, sms);
    default: return launch_m<DET_WF, 8>(a, sms);
    }
}

}  // namespace detlin
