// Internal declarations shared by the translation units of libmoe.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "moe.h"

namespace moe {

typedef __nv_bfloat16 bf16;

constexpr int kMaxE = MOE_MAX_EXPERTS;
constexpr int kTileRows = 128;            // token rows per row tile of the grouped GEMMs
constexpr int kRouteTokPerBlock = 16;     // tokens of a unit: a row of the routers' histogram, a block of the permutation
constexpr int kHistCols = 2 * kMaxE + 1;  // per (expert, slot) pair counts + skipped count
constexpr int kInterleave = 16;           // W1/W3 rows are interleaved in groups of 16
constexpr int kDecodeMaxT = 256;          // up to here the small-batch path (weights read once) is used
constexpr int kTokensDPerExpert = 40;      // small batches with this many tokens per expert or more: token-major decode GEMM
constexpr int kTokensDMaxKept = 6;         // ... on layers with at most this many kept experts
// Large batches with at most so many pairs per kept expert (a forward call counts two per token, skipped or not)
// run gemm_pair_n, the others gemm_tokens_m: kPairMaxRows on rows of fewer than kPairWideH columns, kPairDownRows on
// wider ones of experts with fewer than kPairDeepF features, else kPairMaxRowsWide.  Whole step, gemm_pair_n (in both
// launches) against gemm_tokens_m, alternating runs, pairs per expert 1600 / 2048 / 4096 / 8192:
//   (h, f, experts)    64, 64, 8        -1 % / +8 % / +16 % / +16 %
//                      128, 448, 8      -4 / -4 / -3 / +9      256, 1024, 8     -6 / -7 / -1 / +8
//                      512, 1024, 8    -22 / -19 / -10 / -5    1024, 2048, 8   -12 / -10 / -7 / -5
//                      2048, 4096, 16   -8 / -7 / -7 / -5      4096, 1024, 8   -12 / -10 / -8 / -5
// On narrow layers an item is a few k-blocks long and the two CTAs spend it on handing over to each other.  Mixtral
// layer in 1.5 s loops at the power cap (ms): 8192 tokens (2048 a group) 4.77 vs 4.95, 16384 9.25 vs 9.45, 32768 (8192
// a group) 18.56 vs 18.57, 65536 37.5-39.0 vs 36.2.  There the board's power is the limit.
// Beyond kPairDownRows pairs per expert only the gate/up launch is theirs: in the down launch, whose items run over
// f / 64 k-blocks, pairs that started an item apart read weights and activations from HBM again (8192 tokens of the
// Mixtral layer 4.0 GB where gemm_tokens_m reads 2.1).  Search of 32768 tokens (6144 a group), three runs on one
// board: gemm_tokens_m 55.5-55.7 ms, pairs 53.4-54.2, pairs and gemm_tokens_m 53.5-53.6; forward of 32768 tokens
// 18.2-18.5, 18.1, 18.0-18.2.  Below the line that mixture against the pairs in both launches, pairs per expert 500 /
// 1024 / 1536 / 2048 / 3000 / 4096: Mixtral layer 1.01, 1.00, 1.02, 0.99, 1.00, 1.00 (a run differs by 2 %);
// 1024 / 2048 / 4000: (2048, 4096, 16) 1.03, 1.05, 1.04, (4096, 1024, 8) 1.05, 1.09, 1.09, (1024, 256, 8) 1.07, 1.13,
// 1.09.  Above it against gemm_tokens_m in both, 4500-5000 / 7000-8192: f 64 to 128 (h 512 to 4096) 1.02-1.05 /
// 1.04-1.08, f 192 and 256 0.91-0.98 / 0.97-1.00, f 512 and more 0.92-0.98 / 0.98-1.00; hence kPairDeepF: with one or
// two k-blocks in a down item a launch of either kind is its stores, and the pairs' half of the mixture wins too little.
constexpr int kPairMaxRows = 1536;
constexpr int kPairMaxRowsWide = 8192;
constexpr int kPairDownRows = 4096;
constexpr int kPairWideH = 512;
constexpr int kPairDeepF = 192;
// Top-k calls of more than kDecodeMaxT tokens with at most this many pairs per kept expert, half of the
// weight-major kernel's token tile, run that kernel: it cuts the last round into K-slices, and hardly any
// group needs a second tile.  Whole call in us, gemm_pair_n vs weight-major, layers of 16 experts (h, f):
//   pairs per expert   44          65          80-85 (four / one or two experts per token)
//   768, 512           46 vs 37    45 vs 37    52 vs 44    48 vs 43
//   1024, 2048         77 vs 70    83 vs 81    87 vs 73    87 vs 92-99
//   1536, 3072         118 vs 108  126 vs 120  130 vs 152  130 vs 143
//   2048, 4096         183 vs 170  188 vs 193  194 vs 191  200 vs 225
//   4096, 4096         312 vs 308  338 vs 341  347 vs 369  352 vs 389
//   6144, 512          123 vs 105  129 vs 110  133 vs 113  136 vs 123
// From 95 on the pairs won by up to a quarter except on the smallest weights.
constexpr int kFewRows = 64;
constexpr int kPairPad = 32;        // grain of its token tiles
// Up to here every block of the permutation counts the whole routing record itself (at 32 tokens a
// thread, in bytes, 255 tokens a thread at most); beyond, the routers' histogram and the scan do.
constexpr int kPermuteOwnT = 8192;
// Forward calls of at least so many tokens (64 tiles of 128) on rows of at least so many columns route on
// the tensor cores.  Error of the routing weights against 64 bits (2-norm, 8192 tokens), CUDA cores (one
// chain of h / 32 products per lane) vs tensor cores (chunks of 128 and a compensated sum): h 128
// 0.78e-7 vs 0.97e-7, h 2048 1.39e-7 vs 1.38e-7, h 4096 1.47e-7 vs 1.22e-7, h 8192 1.98e-7 vs 1.24e-7;
// whole call, 16384 tokens, 16 experts, h 6144, f 512: 1282 vs 1229 us.
constexpr int kRouterTcT = 64 * 128;
constexpr int kRouterTcH = 2048;
// Calibration on rows of at least so many columns has a router of its own (ratio_kernel); on narrower ones it runs the
// forward router, whose ratios it then gives to the last bit.  The forward router's bits stay what they are: in a
// stack a logit that moves in its last bit now and then flips a skip decision some layers on.  Calibration in us,
// forward router / ratio_kernel, 8 experts, 300, 8192 and 16384 tokens: h 1024 19.8 / 18.4, 24.1 / 21.5, 32.5 / 27.3;
// h 4096 23.9 / 19.4, 37.1 / 27.7, 56.8 / 52.9.  Error of the ratios against 64 bits (2-norm, 8192 tokens): h 1024
// 3.5e-7 / 2.6e-7, h 4096 (2000 tokens) 5.0e-7 / 2.6e-7.
// Few experts: the forward router computes 2 or 4 columns where ratio_kernel computes 8, so on rows of kRatioFewMinH
// to kRatioFewMaxH columns it stays ahead where the rest is equal: with 3 and 4 experts on batches that L2 no longer holds
// (h 2048, 4096, 6144, 8192, the same 67 MB: 32.3 / 30.0, 29.2 / 26.1, 29.6 / 28.1, 29.3 / 30.0; 88 MB: 41.9 / 41.5,
// 37.0 / 43.8, 33.3 / 35.1, 33.7 / 41.6; 134 MB: 56.0 / 56.7, 47.4 / 51.9, 57.6 / 64.2, 43.4 / 47.4; the line is the
// 4737th token of h 8192, with which its tiles go to four teams), with 2 experts from the second tile of a block on
// (h 1536, 4096, 8192: 2400 tokens 20.7 / 22.1, 23.3 / 23.2, 26.7 / 27.9; 16384 tokens of h 4096 47.2 / 51.9).  With 5
// and 6 experts either wins by turns (100 to 536 MB, h 1536 to 12288, ratio_kernel 0.82 to 1.17 of the forward router,
// 0.96 on average: it stays).  Beyond kRatioFewMaxH, the widest rows measured, ratio_kernel stays too: a router that is
// zero but for some columns then gives the ratios of the narrow one to the bit whatever the number of tokens, which
// two routers with sums in different orders do not.
constexpr int kRatioMinH = 1024;
constexpr int kRatioFewMinH = 1536;
constexpr int kRatioFewMaxH = 12288;
constexpr int kRatioTwoT = 148 * 16;
constexpr size_t kRatioFewBytes = (size_t)74 << 20;
inline bool calibrate_on_tiles(int T, int h, int r) {
  if (h < kRatioFewMinH || h > kRatioFewMaxH) return h >= kRatioMinH;
  if (r == 2) return T <= kRatioTwoT;
  return r > 4 || (size_t)T * h * 2 <= kRatioFewBytes;
}
constexpr int kDecodeKbPerItem = 112;      // k-blocks (of 64) per split-K item, decode down-proj

// Device-resident description of one permuted batch, written by the permutation (beyond kPermuteOwnT
// tokens by the scan, for the dense search by set_dense_meta) and read by every later kernel.
struct Meta {
  int32_t count[kMaxE];            // token-expert pairs that run, per kept expert (compact index)
  int32_t count_slot[kMaxE][2];    // the same, split by top-2 slot
  int32_t off[kMaxE + 1];          // first permuted row of each expert's group (padded groups)
  int32_t tile_prefix[kMaxE + 1];  // cumulative number of 128-row tiles
  int32_t n_skipped;
  int32_t n_touched;
  int32_t reserved;
};

struct KeptIds {
  int32_t id[kMaxE];  // compact index -> original expert id
};

// Programmatic dependent launch: a kernel launched this way may start while its predecessor
// in the stream is still draining; it must call pdl_wait() before touching anything the
// predecessor wrote (or still reads).  Every kernel on the forward path calls
// pdl_launch_dependents() and pdl_wait() first thing (the GEMMs after their set-up), so the
// stream order of all memory accesses is unchanged and only launch latency and prologues overlap.
// The one exception are the down launches of gemm_pair_n, gemm_weights_m and gemm_tokens_d: before they wait they
// read the batch description (Meta) and fetch weights (handover_wait in gemm_sm100.cu), and their MMA warps never wait.
// What that rests on: Meta is complete before the gate/up launch of the batch passes its own wait, and that launch
// triggers only then.  So nothing from the gate/up launch to the last down launch of a batch (the combine kernels between
// the column slabs of a host call among them) may write Meta or weights, nor may a kernel that does so trigger early
// and be followed by a down launch directly.
//
// THE RULE for every kernel launched with launch_pdl: whatever an earlier kernel of the stream
// may have written (token rows, routing records, permutation tables, the batch description,
// activations, expert outputs, the residual) is read with ld_l2() below (ld.global.cg), never
// through a `const T* __restrict__` parameter with a plain dereference or __ldg.  Such a kernel
// is resident while its predecessors still write, no kernel boundary invalidates the SM's L1 in
// between, and the non-coherent path (ld.global.nc, which the compiler may pick for const
// __restrict__ data) is only defined for data that does not change during the kernel's lifetime:
// an L1 line cached on this SM before the writer finished would be stale.  Only data that is
// constant from the creation of the handle on (router rows, expert weights) keeps __ldg or the
// streaming loads.  Operands that reach the SM through TMA are read at L2 by construction.
#ifdef __CUDACC__
__device__ __forceinline__ uint4 ld_l2(const uint4* p) { return __ldcg(p); }
__device__ __forceinline__ float4 ld_l2(const float4* p) { return __ldcg(p); }
__device__ __forceinline__ int ld_l2(const int32_t* p) { return __ldcg(p); }
__device__ __forceinline__ float ld_l2(const float* p) { return __ldcg(p); }
__device__ __forceinline__ int ld_l2(const uint8_t* p) { return (int)__ldcg(p); }
__device__ __forceinline__ float ld_l2(const __nv_bfloat16* p) {
  return __uint_as_float((uint32_t)__ldcg(reinterpret_cast<const unsigned short*>(p)) << 16);
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// MOE_NO_PDL=1 (read when a handle is created) launches everything with plain stream order.
inline bool g_pdl_enabled = true;

template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                       Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = g_pdl_enabled ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}
#endif

#ifdef __CUDACC__
// The same launch in plain stream order (the kernel's griddepcontrol instructions are no-ops).
template <typename... KArgs, typename... Args>
cudaError_t launch_plain(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                         Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}
#endif

// Stores the message moe_last_error() returns on this thread and returns `code` (api.cu).
int set_error(int code, const char* fmt, ...);

// ---- routing / permutation / element-wise kernels (route_permute.cu) --------------------
struct RouteOut {
  int32_t* idx;       // [T][2] compact expert index
  float* wn;          // [T][2]
  float* ratio;       // [T]
  uint8_t* skipped;   // [T]
  float* logits;      // [T][r] or null
  int32_t* blk_hist;  // [nblk][kHistCols] or null
  // user-visible routing record (all null when not requested)
  int32_t* s_idx;
  float* s_wn;
  float* s_ratio;
  uint8_t* s_skipped;
};

// w_const: Wg never changes (a handle's own rows) and may be read before the predecessor is done
cudaError_t launch_router(const bf16* x, const bf16* Wg, int T, int h, int r, float beta,
                          const KeptIds& kept, const RouteOut& out, cudaStream_t st, bool w_const = true);
// w_e1 / w_e0 of every token (calibration, calibrate_on_tiles)
cudaError_t launch_ratios(const bf16* x, const bf16* Wg, int T, int h, int r, float* ratio, cudaStream_t st,
                          bool w_const = true);
// Large forward batches (kRouterTcT, kRouterTcH): the logits on the tensor cores (gemm_sm100.cu), the
// decision as in launch_router.  Wg16 = the kept router rows padded with zero rows to kMaxE rows.
cudaError_t launch_router_tc(const bf16* x, const bf16* Wg16, int T, int h, int r, float beta,
                             const KeptIds& kept, const RouteOut& out, int* status, cudaStream_t st);
// T <= kDecodeMaxT: router with one block per token; permutation + gather with one block per token
cudaError_t launch_router_small(const bf16* x, const bf16* Wg, int T, int h, int r, float beta,
                                const KeptIds& kept, const RouteOut& out, cudaStream_t st);
cudaError_t launch_route_single(const bf16* x, const bf16* Wg, int h, int r, float beta,
                                const KeptIds& kept, const RouteOut& out, int pad, Meta* meta,
                                int32_t* pair_pos, bf16* xperm, int32_t* s_count,
                                int32_t* s_nskipped, int32_t* s_ntouched, int E, cudaStream_t st);
cudaError_t launch_permute_gather_small(const bf16* x, const int32_t* idx, const uint8_t* skipped, int T,
                                        int h, int r, int pad, Meta* meta, int32_t* pair_pos,
                                        bf16* xperm, int32_t* s_count,
                                        int32_t* s_nskipped, int32_t* s_ntouched, const KeptIds& kept,
                                        int E, cudaStream_t st);
cudaError_t launch_scan(const int32_t* blk_hist, int nblk, int r, int pad, int32_t* blk_base,
                        Meta* meta, int32_t* s_count, int32_t* s_nskipped, int32_t* s_ntouched,
                        const KeptIds& kept, int E, cudaStream_t st);
// T > kDecodeMaxT.  blk_base: the scan's result, or null for at most kPermuteOwnT tokens (the kernel
// then counts for itself and writes *meta and the record's counts).  active: skip flags (uint8,
// top2) or the number of slots that run (int32).
cudaError_t launch_permute(const bf16* x, const int32_t* idx, const void* active, bool top2, int T, int k, int h,
                           int r, int pad, const int32_t* blk_base, Meta* meta, int32_t* pair_pos, bf16* xperm,
                           int32_t* s_count, int32_t* s_nskipped, int32_t* s_ntouched, const KeptIds& kept,
                           int E, cudaStream_t st);
cudaError_t launch_combine(const float* O, int ksplit, size_t split_stride, const int32_t* pair_pos,
                           const float* wn, const bf16* residual, int T, int h, bf16* y,
                           cudaStream_t st, int col0 = 0, int cols = 0);  // columns col0 .. + cols (0: all)
// general top-k path (k slots per token instead of two)
cudaError_t launch_router_topk(const bf16* x, const bf16* Wg, int T, int h, int r, int k, float beta,
                               const KeptIds& kept, int32_t* idx, float* wn, int32_t* nact,
                               int32_t* u_idx, float* u_wn, int32_t* u_nact, float* logits,
                               cudaStream_t st);
cudaError_t launch_count_topk(const int32_t* idx, const int32_t* nact, int T, int k,
                              int32_t* blk_hist, cudaStream_t st);
cudaError_t launch_combine_topk(const float* O, int ksplit, size_t split_stride,
                                const int32_t* pair_pos, const float* wn, int k, int T, int h,
                                bf16* y, cudaStream_t st);
cudaError_t launch_coselection(const int32_t* idx, int T, int E, const KeptIds& kept, int32_t* counts,
                               cudaStream_t st);
cudaError_t launch_top2_distance(const float* O, int ksplit, size_t split_stride,
                                 const int32_t* pair_pos, int T, int h, float* dist, cudaStream_t st);
cudaError_t launch_rmsnorm(const bf16* x, int T, int h, float eps, bf16* out, cudaStream_t st);
cudaError_t launch_set_dense_meta(Meta* meta, int E, int rows_per_expert, int off_stride,
                                  cudaStream_t st);
// k-th smallest (0-based) of ratio[T] for k = k0 and k1 (= k0 or k0 + 1), written to out[0], out[1]
// (device memory or mapped host memory)
cudaError_t launch_select2(const float* ratio, int T, int k0, int k1, float* out, cudaStream_t st);
// brings every kernel of a calibration of up to MOE_NOALLOC_MAX_TOKENS tokens onto the device
cudaError_t load_calibration_kernels();
// W13[c][32q + s] = W1[id[c]][16q + s] (s < 16) | W3[id[c]][16q + s - 16] (s >= 16)
cudaError_t launch_interleave(const bf16* W1, const bf16* W3, const KeptIds& kept, int r, int f,
                              int h, bf16* W13, cudaStream_t st);

// ---- grouped GEMMs (gemm_sm100.cu) ----------------------------------------------------
enum GemmOut { kOutActBf16 = 0, kOutF32 = 1, kOutBf16 = 2 };

struct GemmArgs {
  const Meta* meta;
  int r;         // kept experts
  int K;         // contraction length (h for gate/up, f for down)
  int n_w_rows;  // weight rows per expert (2f interleaved for gate/up, h for down)
  int w_row0;    // pair kernel: the launch computes rows w_row0 (a multiple of 512) .. n_w_rows
  // token-side operand rows: a_row = a_row_base + a_off_mul * off[c] + 128 * m
  int a_row_base, a_off_mul;
  // output rows: out_row = out_row_base + out_off_mul * off[c] + 128 * m; column offset c * out_col_mul
  int out_row_base, out_off_mul;
  long long out_col_mul;
  long long out_ld;        // elements between output rows
  void* out;               // bf16 activations / fp32 outputs / bf16 expert outputs
  long long split_stride;  // elements between split-K partial planes (decode down-proj)
  int* status;             // device error word
  // weight-major kernel: arrival counters (kTailHeaderBytes, zero between launches) followed by
  // the partial tiles of the K-sliced tail items; null = no slicing
  float* tail;
  int tile_cap;  // pair kernel: largest token tile / 32, 0 = chosen by the kernel (tests set it)
};

constexpr size_t kTailHeaderBytes = 4096;  // four arrival counters per tail item
constexpr size_t kTailBufferBytes = kTailHeaderBytes + (size_t)1024 * 128 * 128 * 4;  // 1024 slots of 128 tokens

int gemm_init_driver_api();  // resolves cuTensorMapEncodeTiled; 0 on success
int make_map_2d(CUtensorMap* m, const void* base, uint64_t inner, uint64_t rows, uint32_t box_rows);
int make_map_3d(CUtensorMap* m, const void* base, uint64_t inner, uint64_t rows, uint64_t planes,
                uint32_t box_rows);

struct GemmMaps {
  CUtensorMap w;     // weights [planes = r][rows][K], box 64 x (256 or 128) x 1
  CUtensorMap t[4];  // token-side operand [rows][K], boxes of 16 / 32 / 64 / 128 rows
};

// Token rows are the 128-row MMA operand, weights the 256-wide one (large T).
cudaError_t launch_gemm_tokens_m(bool gate_up, GemmOut out_kind, const GemmMaps& maps,
                                 const GemmArgs& a, cudaStream_t st);
// On CTA pairs: weight rows are the 256-row MMA operand, up to 256 tokens the other (large T).
cudaError_t launch_gemm_pair_n(bool gate_up, GemmOut out_kind, const GemmMaps& maps,
                               const GemmArgs& a, cudaStream_t st);
// Weight rows are the 128-row MMA operand, tokens the narrow one (small T): weights stream once.
cudaError_t launch_gemm_tokens_d(bool gate_up, const GemmMaps& maps, const GemmArgs& a, int kb_per_item,
                                 cudaStream_t st);
cudaError_t launch_gemm_weights_m(bool gate_up, const GemmMaps& maps, const GemmArgs& a,
                                  int kb_per_item, int max_tokens_per_tile, cudaStream_t st);
// Single-token forward on the CUDA cores (T = 1 only): routing + gate/up matrix-vector kernel,
// then the down projection with the weighted sum of Eq. 2, which writes y.
cudaError_t gemv_single_setup();
bool gemv_single_fits(int h, int f);
cudaError_t launch_gemv_route_gate_up(const bf16* x, const bf16* Wg, const bf16* W13, int r, int h, int f,
                                      float beta, const KeptIds& kept, const RouteOut& ro, Meta* meta,
                                      int32_t* pair_pos, int32_t* s_count,
                                      int32_t* s_nskipped, int32_t* s_ntouched, int E, bf16* act,
                                      cudaStream_t st);
cudaError_t launch_gemv_down_combine(const bf16* act, const bf16* W2, const int32_t* idx,
                                     const uint8_t* skipped, const float* wn, const bf16* residual,
                                     int h, int f, bf16* y, cudaStream_t st);
// Plain CUDA-core kernels of the same contractions, for bring-up and debugging only
// (MOE_DEBUG_SIMT=1); never selected otherwise.
cudaError_t launch_simt_gate_up(const bf16* A, const bf16* W13, const GemmArgs& a, int cap_rows,
                                cudaStream_t st);
cudaError_t launch_simt_down(const bf16* A, const bf16* W2, const GemmArgs& a, int cap_rows,
                             GemmOut out_kind, cudaStream_t st);
cudaError_t gemm_set_attributes();
// Test hook: one CTA runs the GEMMs' bounded wait on a barrier nobody arrives on, then their
// abort path (see moe_test_hooks.h).
cudaError_t launch_wait_expiry(int* status, unsigned long long limit_ns, cudaStream_t st);
cudaError_t launch_wait_expiry_pair(int* status, unsigned long long limit_ns, int cta, cudaStream_t st);

// ---- search (search.cu) ---------------------------------------------------------------
// Where the enumeration finds the expert outputs.  Dense (topk_idx == null): Yall[T][E][h].
// Pruned work: only each token's K = E - r + 2 top-ranked experts were evaluated;
// topk_idx[T][K] lists them in rank order and their outputs are rows of a permuted buffer,
// row (t / chunk_tokens) * chunk_rows + pair_pos[t][rank].
struct EnumSource {
  const int32_t* topk_idx;
  const int32_t* pair_pos;
  int chunk_tokens;
  int chunk_rows;
  int k_stride;  // ranked experts recorded per token in topk_idx / pair_pos (>= E - r + 2)
};
int enumerate_num_blocks(int T, int nC);
bool enumerate_takes_list(int nC);
// host_subsets: the masks in host memory; the copy `subsets` in device memory is read only where
// !enumerate_takes_list(nC).  status_out (or null): where *status goes with the losses.
cudaError_t launch_enumerate(const float* logits, const bf16* Yall, int T, int E, int r, int h,
                             const uint32_t* subsets, const uint32_t* host_subsets, int nC, float* partial,
                             double* loss_sq, float* losses, const float* Fref, const EnumSource& src,
                             const int* status, int* status_out, cudaStream_t st);

}  // namespace moe
