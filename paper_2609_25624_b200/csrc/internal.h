// Internal declarations shared by the host-side translation units of libdet_linear.
#pragma once
#include <cuda_runtime.h>
#include <cuda.h>
#include <cstdint>
#include <cstddef>
#include "det_linear.h"

namespace detlin {

constexpr int kOrderVersion = 2;
constexpr int kSegmentGranule = 256;   // segment boundaries are multiples of this many k elements
constexpr int64_t kDecodeNoSplitRows = 16384;   // decode bucket: weight matrices with at least this many rows are not split
constexpr int kDecodeMaxSegments = 8;  // most K segments the decode kernel folds inside a thread block
constexpr unsigned long long kDefaultWaitLimitNs = 2000000000ull;   // bound of one device-side wait: 2 s
constexpr int kDecodeMaxM = 64;        // decode bucket edge: rule R2 puts batches of up to 64 rows in the decode bucket

enum KernelId : int { kKernelGeneric = 0, kKernelDecode = 1, kKernelPrefill = 2 };

// Device-side status word written by kernels that give up a bounded wait.
struct DeviceStatus {
    unsigned int timeout_flag;   // nonzero: some wait expired
    unsigned int where;          // which wait (diagnostic); of several, the highest number
};

// LaunchArgs::test_flags beyond the test hooks: the decode kernel also waits for the previous kernel in the stream before it
// touches W and b, and before it lets the next kernel start (callers for whom W and b are not parameters that were complete long
// before)
constexpr int kFlagLateWeights = 4;

constexpr int kMaxDevices = 64;     // per-device caches (function attributes, symbol addresses)

void set_error(const char* fmt, ...);
det_status_t fill_params(int64_t M, int64_t N, int64_t K, det_linear_params_t* out);

// Decode for any K: batch rows and weight rows of a warp, and whether two warps share a row's two segments (in sixteen-warp blocks that
// hold all of K).  mt = 0: none chosen yet.
struct AnyLayout { int mt, rt, split; };
struct AnyGrid {
    int warps, row_warps, blocks_per_sm;         // warps of a block, those of them that have rows of their own
    int64_t window;                              // k elements of the activations in shared memory
    int64_t groups, batch_blocks, blocks_x;      // blocks_x thread blocks walk the row groups of each batch block
};
constexpr int kAnySmemBytes = 110 * 1024;        // activations of one window of K with two blocks of 8 warps per SM ...
constexpr int kAnySmemBytes1 = 220 * 1024;       // ... or one block of 16
constexpr int kAnySplitBytes = 8 * 32 * 4;       // split: the second segments' sums, one a lane
AnyGrid any_grid(const AnyLayout& l, int64_t M, int64_t N, int64_t K, int sm_count);
bool any_layout_fits(const AnyLayout& l, int64_t K, int S);
AnyLayout any_layout_for(int64_t M, int64_t N, int64_t K, int S, int wfmt, int sm_count);
// Searches for a layout or a tiling made by the calling thread (det_test_schedule_searches).
void count_schedule_search();

// ---- kernel launchers (defined in the .cu files) -------------------------------------------
struct LaunchArgs {
    const float* x;
    const void* W;        // [N,K] in weight format wfmt
    int wfmt;             // det_weight_format_t
    const float* b;
    float* y;             // final output [M,N], row pitch ldy
    int64_t ldy;          // floats between consecutive rows of y (N unless the plan is a column shard)
    float* partials;      // [S,M,N] when S > 1, else nullptr
    uint64_t partial_floats;   // what it holds: with room for whole tiles, and counters, the prefill kernel folds in place
    unsigned* tile_counters;   // prefill with S > 1: zeroed counters per output tile and warp (the TMA-fed kernel folds in place), or nullptr
    unsigned* sync;       // TMA-fed prefill kernel: zeroed ticket and hand-over flags
    float* handoff;       // prefill in equal stretches: accumulators on their way from one block to the next, or nullptr
    int64_t M, N, K;
    int64_t seg_len;
    int S;
    cudaStream_t stream;
    DeviceStatus* status; // device pointer
    int sm_count;
    int max_blocks;       // 0 = automatic
    int variant;          // 0 = automatic
    AnyLayout any_layout; // decode for any K
    unsigned long long wait_limit_ns;   // bound of one device-side wait (TMA-fed kernels)
    int test_flags;       // decode kernel test hooks (0 outside the tests)
};

cudaError_t launch_generic(const LaunchArgs& a, int bucket);
// Second pass of split-K: y[m,n] = (((P0 + P1) + P2) + ...) (+ b[n]); rule R3.
cudaError_t launch_combine(const LaunchArgs& a);

// Register-staged prefill kernel (the fallback without a schedule workspace; a.variant 15 .. 18 forces 5 .. 8 rows
// per thread).
cudaError_t launch_prefill(const LaunchArgs& a);
// Prefill kernel with both tiles fed by TMA (prefill_tma_kernel.cuh); block tile 16 tm rows x width columns.  Tensor maps,
// swizzled over the width of the box: map_x: x [M][K], box [16 tm][32]; map_w: W [N][K] in its format, box [width][32].
cudaError_t launch_prefill_tma(const LaunchArgs& a, int tm, int width, const CUtensorMap* map_w, const CUtensorMap* map_x);
// The same kernel fed by plain loads: any K, any alignment (x and W themselves, no tensor maps).  Without the hand-over
// workspace every unit of work gets a block of its own.
cudaError_t launch_prefill_plain(const LaunchArgs& a);
int prefill_tile_width(int64_t M, int64_t N, int64_t K, int S, int64_t seg_len, int tm, int sm_count);
// Device memory the TMA-fed kernel wants: split-K partials by tile with their counters; ticket, flags and accumulators of
// the hand-over between blocks (no accumulators when every unit of work gets a block of its own).
struct PrefillWorkspace { uint64_t partial_floats, counter_words, sync_words, handoff_floats; };
PrefillWorkspace prefill_workspace(int64_t M, int64_t N, int64_t K, int S, int64_t seg_len, int sm_count);
// tile height / 16 the prefill kernels use for batch size M (the register-staged kernel: rows per thread); schedule only
int prefill_rows_per_thread(int64_t M);
// Fixed-order RMSNorm of M rows of H elements (rmsnorm.cu).
cudaError_t launch_rmsnorm(const float* x, const float* g, float eps, int64_t M, int64_t H, float* y, cudaStream_t stream);
// Fixed-order decode attention (attention.cu); attention_smem_bytes = dynamic shared memory it needs.
size_t attention_smem_bytes(int G, int T, int D);
// test hook: force the number of thread blocks that share one (batch, KV head) row (1, 2, 4, 8, 16; 0 = automatic)
void attention_test_force_split(int c);
// the cluster size the launcher would use on a device with sm_count SMs (pure function of its arguments and of
// the forced split), and the dynamic shared memory of one block for it
int attention_split(int B, int Hkv, int G, int T, int D, int sm_count);
size_t attention_block_smem_bytes(int G, int T, int D, int C);
cudaError_t launch_attention_decode(const float* q, const float* k, const float* v, float scale, int B, int Hq, int Hkv, int T,
                                    int D, float* o, cudaStream_t stream);
// Read `bytes` at buf through L2 (evicts what was there without leaving dirty lines); sink: 4 bytes of device memory.
cudaError_t launch_l2_evict(const void* buf, size_t bytes, unsigned* sink, int sm_count, cudaStream_t stream);
// bytes (a multiple of 16) between pinned host memory and device memory, both 16-byte aligned
cudaError_t launch_copy_across_bus(const void* src, void* dst, size_t bytes, cudaStream_t stream);
cudaError_t launch_argmax(const float* y, int64_t M, int64_t N, int32_t* idx, cudaStream_t stream);

// Decode-kernel tiling chosen for a shape (numerically inert); used by the host to build the
// tensor maps with matching box sizes.
struct DecodeConfig {
    int mt, wm, rt, wr, sk, kc, stages;   // warp tile (mt x rt), warps (wm x wr) x sk segment groups, k per stage, ring depth
    int id;
};
// S = number of K segments of the order (it only scales the unit count in the schedule's cost model)
bool decode_config_for(int64_t M, int64_t N, int64_t K, int S, int wfmt, int variant, DecodeConfig* out);
int decode_num_variants();
// The longest K segment of the decode order.
inline int64_t decode_segment(int64_t K, int S)
{
    const int64_t granules = (K + kSegmentGranule - 1) / kSegmentGranule;
    return S > 1 ? (granules + S - 1) / S * kSegmentGranule : K;
}
// FP32 weights: does the multiply loop of a tiling load a chunk ahead?  The loads of a segment's first chunk, all of them before the
// first multiplication, then cost what the later chunks gain.  Times with against without, over the tilings of 161 shapes: segments of
// 128 to 256 elements 1.05 to 1.3 (M = 10, N = 22402, K = 208 13.4 us, without 10.8); 384 and 512 on average 0.95 in tiles of 8 rows a
// warp (M = 33, N = 6411, K = 880 18.6 and 21.0; M = 44, N = 22508, K = 264 35.0 and 38.6), 1.01 of 4; 768 0.91 and 0.97; 2048 0.82 and 0.89.  Up to four batch rows are bound by memory
// and gain later: segments of 512 to 1024 1.03, from 2048 on 0.83 to 1.0.
inline bool decode_loads_ahead(int rows_of_warp, int64_t M, int64_t K, int S)
{
    return decode_segment(K, S) >= (M <= 4 ? 2048 : rows_of_warp == 8 ? 257 : 768);
}
// map_w: box of a whole tile (rt * wr weight rows); map_g: of one row group (rt)
cudaError_t launch_decode(const LaunchArgs& a, const DecodeConfig& cfg, const CUtensorMap* map_w, const CUtensorMap* map_g, const CUtensorMap* map_x);
// resident blocks per SM of a tiling on the current device for an order with S segments (schedule information only)
int decode_config_occupancy(int wfmt, const DecodeConfig& cfg, int S);

}  // namespace detlin

struct det_linear_plan {
    det_linear_params_t prm;
    int device;
    int sm_count;
    float* partials;                 // device, S*M*n_count floats and more (prefill_workspace), or nullptr
    uint64_t partial_floats;
    unsigned* tile_counters;         // device, inside the partials allocation (prefill, S > 1) or nullptr
    uint64_t n_tile_counters;
    unsigned* sync;                  // device, prefill: ticket and hand-over flags of the TMA-fed kernel, or nullptr
    uint64_t n_sync;
    float* handoff;                  // device, in the same allocation: accumulators handed over from block to block, or nullptr
    int64_t n_begin, n_count, ldy;   // column shard computed by this plan (0, N, N for a whole layer)
    detlin::DeviceStatus* status;    // device
    float* x_stage;                  // device staging for det_linear_run_host
    float* y_stage;
    int forced_kernel;               // -1 automatic
    int max_blocks;
    int variant;
    unsigned long long wait_limit_ns;
    int test_flags;
    // the decode tiling chosen for this plan (schedule only; cached so that a run does no search)
    detlin::DecodeConfig decode_cfg;
    detlin::AnyLayout any_layout;    // decode for any K and alignment: likewise, chosen with the plan
    int decode_cfg_variant;          // variant the cached tiling was chosen for, -1 = none yet
    // tensor-map cache for the decode kernel (keyed by the pointers they were built for)
    const void* map_w_ptr;
    const void* map_x_ptr;
    int map_cfg_id;
    CUtensorMap map_w;
    CUtensorMap map_g;               // decode: one row group of a tile
    CUtensorMap map_x;
};

namespace detlin {

// One run on the plan's device buffers (capi.cu): alignment checks, choice of the kernel, tensor maps, launch.
det_status_t run_device(det_linear_plan_t* plan, const float* x, const void* W, const float* b, float* y, cudaStream_t stream);

}  // namespace detlin
