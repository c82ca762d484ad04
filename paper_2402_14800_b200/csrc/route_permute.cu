// Router, token permutation, combine and the small element-wise kernels.
//
//   router_kernel   Sec. 3.1 (logits, softmax, top-2, Eq. 1), Sec. 3.2 (kept experts only),
//                   Sec. 3.3 (skip test), App. A.2 (weight 1 after a skip); several tokens per warp
//                   (large forward batches: router_tc_kernel, on the tensor cores).
//   ratio_kernel    Sec. 3.3: w_e1 / w_e0 for calibration, on warp-level tensor-core instructions, as
//                   router_topk_kernel (App. A.2).
//   scan / permute  stable counting sort of the token-expert pairs that run, by expert (no atomics,
//                   the order is a function of the routing alone), and the copy of the routed rows
//                   of x into that order.
//   combine         Eq. 2: y = bf16(residual + w~_e0 o_e0 + w~_e1 o_e1), slot 0 first.
//
// Every kernel here that is launched as a programmatic dependent reads what earlier kernels of
// the stream wrote with ld_l2 (the rule beside launch_pdl): token rows, routing records,
// histograms, the batch description, expert outputs, the residual.  The router rows never
// change and keep ld.global.nc.
#include "common.h"
#include "route_device.cuh"

namespace moe {

namespace {

// Small batches: one block per token, all loads of a thread independent of each other, so the
// kernel costs a couple of memory round trips instead of a serial walk over the row.
template <int R>
__global__ void __launch_bounds__(256)
router_small_kernel(const bf16* x, const bf16* __restrict__ Wg, int T, int h, int r,
                    float beta, KeptIds kept, RouteOut o) {
  pdl_launch_dependents();
  pdl_wait();
  __shared__ float s_part[8][R];
  const int t = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nvec = h >> 3;
  float acc[R];
#pragma unroll
  for (int c = 0; c < R; ++c) acc[c] = 0.f;
  const uint4* xr = reinterpret_cast<const uint4*>(x + (size_t)t * h);
  for (int v = threadIdx.x; v < nvec; v += 256) {
    float xf[8];
    unpack8(ld_l2(xr + v), xf);
#pragma unroll
    for (int c = 0; c < R; ++c) {
      if (c < r) {
        float wf[8];
        unpack8(__ldg(reinterpret_cast<const uint4*>(Wg + (size_t)c * h) + v), wf);
#pragma unroll
        for (int k = 0; k < 8; ++k) acc[c] = fmaf(xf[k], wf[k], acc[c]);
      }
    }
  }
#pragma unroll
  for (int c = 0; c < R; ++c) {
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], s);
    if (lane == 0) s_part[warp][c] = acc[c];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    float l[R];
#pragma unroll
    for (int c = 0; c < R; ++c) {
      float v = 0.f;
#pragma unroll
      for (int w = 0; w < 8; ++w) v += s_part[w][c];
      l[c] = v;
    }
    int e0, e1;
    bool skip;
    route_decide<R>(l, r, beta, t, kept, o, e0, e1, skip);
  }
}

// A single token (batch-1 decoding): routing, the (trivial) permutation, the batch description
// and the copy of the token's row in one block, in place of the two launches above.  The
// records it writes are those of router_small_kernel + permute_gather_small_kernel for T = 1.
template <int R>
__global__ void __launch_bounds__(256)
route_single_kernel(const bf16* x, const bf16* __restrict__ Wg, int h, int r, float beta,
                    KeptIds kept, RouteOut o, int pad, Meta* meta, int32_t* __restrict__ pair_pos,
                    bf16* __restrict__ xperm, int32_t* s_count,
                    int32_t* s_nskipped, int32_t* s_ntouched, int E) {
  pdl_launch_dependents();
  pdl_wait();
  __shared__ float s_part[8][R];
  __shared__ int s_p[2];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nvec = h >> 3;
  float acc[R];
#pragma unroll
  for (int c = 0; c < R; ++c) acc[c] = 0.f;
  const uint4* xr = reinterpret_cast<const uint4*>(x);
  for (int v = threadIdx.x; v < nvec; v += 256) {
    float xf[8];
    unpack8(ld_l2(xr + v), xf);
#pragma unroll
    for (int c = 0; c < R; ++c) {
      if (c < r) {
        float wf[8];
        unpack8(__ldg(reinterpret_cast<const uint4*>(Wg + (size_t)c * h) + v), wf);
#pragma unroll
        for (int k = 0; k < 8; ++k) acc[c] = fmaf(xf[k], wf[k], acc[c]);
      }
    }
  }
#pragma unroll
  for (int c = 0; c < R; ++c) {
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], s);
    if (lane == 0) s_part[warp][c] = acc[c];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    float l[R];
#pragma unroll
    for (int c = 0; c < R; ++c) {
      float v = 0.f;
#pragma unroll
      for (int w = 0; w < 8; ++w) v += s_part[w][c];
      l[c] = v;
    }
    int e0, e1;
    bool skip;
    route_decide<R>(l, r, beta, 0, kept, o, e0, e1, skip);
    if (skip) e1 = -1;
    publish_single(e0, e1, pad, kept, meta, pair_pos, s_count, s_nskipped, s_ntouched, E,
                   s_p[0], s_p[1]);
  }
  __syncthreads();
  const int p0 = s_p[0], p1 = s_p[1];
  uint4* d0 = reinterpret_cast<uint4*>(xperm + (size_t)p0 * h);
  uint4* d1 = reinterpret_cast<uint4*>(xperm + (size_t)(p1 < 0 ? p0 : p1) * h);
  for (int v = threadIdx.x; v < nvec; v += 256) {
    const uint4 val = ld_l2(xr + v);
    d0[v] = val;
    if (p1 >= 0) d1[v] = val;
  }
}

// Small batches: permutation and gather in one launch, one block per token.  Every block
// recomputes the (tiny) histogram and offsets from the routing record (by ballots: with loops over
// the record the stage took 16.9 us at 256 tokens and 14.5 at 128, now 12.6 and 11.5), places its own token's
// pairs and copies the token's row to them; block 0 also publishes the batch description.
// Padding rows of the groups are left as they are: in the weight-major GEMM a token row only
// feeds its own accumulator column, and the columns of padding rows are never stored.
__global__ void __launch_bounds__(kDecodeMaxT)
permute_gather_small_kernel(const bf16* x, const int32_t* idx, const uint8_t* skipped, int T, int h, int r, int pad,
                            Meta* meta, int32_t* __restrict__ pair_pos,
                            bf16* __restrict__ xperm,
                            int32_t* s_count, int32_t* s_nskipped, int32_t* s_ntouched, KeptIds kept,
                            int E) {
  pdl_launch_dependents();
  pdl_wait();
  // thread i looks at token i; a ballot per expert and slot counts a warp's tokens
  constexpr int kWarps = kDecodeMaxT / 32;
  __shared__ int s_part[3][kWarps][kMaxE];  // slot-0 pairs, slot-1 pairs, pairs of tokens before t
  __shared__ int s_e[2], s_p[2];
  const int i = threadIdx.x, warp = i >> 5, lane = i & 31;
  const int t = blockIdx.x;
  int e0 = -1, e1 = -1;
  if (i < T) {
    e0 = ld_l2(idx + 2 * i);
    e1 = ld_l2(skipped + i) ? -1 : ld_l2(idx + 2 * i + 1);
  }
  if (i == t) { s_e[0] = e0; s_e[1] = e1; }
  const unsigned before = t >= 32 * (warp + 1) ? 0xffffffffu : (t > 32 * warp ? (1u << (t - 32 * warp)) - 1u : 0u);
  for (int c = 0; c < r; ++c) {
    const unsigned m0 = __ballot_sync(0xffffffffu, e0 == c), m1 = __ballot_sync(0xffffffffu, e1 == c);
    if (lane == c) {
      s_part[0][warp][c] = __popc(m0);
      s_part[1][warp][c] = __popc(m1);
      s_part[2][warp][c] = __popc(m0 & before) + __popc(m1 & before);
    }
  }
  __syncthreads();
  if (warp == 0) {
    const bool on = lane < r;
    int c0 = 0, c1 = 0, rank = 0;
    if (on) {
#pragma unroll
      for (int w = 0; w < kWarps; ++w) { c0 += s_part[0][w][lane]; c1 += s_part[1][w][lane]; rank += s_part[2][w][lane]; }
    }
    const int cnt = c0 + c1, padded = (cnt + pad - 1) / pad * pad, mine = (cnt + kTileRows - 1) / kTileRows;
    int end = padded, tiles = mine;  // inclusive sums over the experts
#pragma unroll
    for (int s = 1; s < kMaxE; s <<= 1) {
      const int a = __shfl_up_sync(0xffffffffu, end, s), b = __shfl_up_sync(0xffffffffu, tiles, s);
      if (lane >= s) { end += a; tiles += b; }
    }
    const int pos = end - padded + rank;  // of the next pair of this lane's expert
    const int f0 = s_e[0], f1 = s_e[1];
    const int p0 = __shfl_sync(0xffffffffu, pos, f0 & 31), p1 = __shfl_sync(0xffffffffu, pos, f1 & 31);
    if (lane < 2) {
      const int p = lane == 0 ? p0 : (f1 < 0 ? -1 : p1);
      s_p[lane] = p;
      pair_pos[2 * t + lane] = p;
    }
    if (t == 0) {
      const int pairs = __reduce_add_sync(0xffffffffu, cnt);
      const int touched = __popc(__ballot_sync(0xffffffffu, cnt > 0));
      if (lane < kMaxE) {
        meta->count[lane] = cnt;
        meta->count_slot[lane][0] = c0;
        meta->count_slot[lane][1] = c1;
        meta->off[lane + 1] = end;
        meta->tile_prefix[lane + 1] = tiles;
        if (s_count && lane < E) { s_count[2 * lane] = 0; s_count[2 * lane + 1] = 0; }
      }
      __syncwarp();
      if (s_count && on) { s_count[2 * kept.id[lane]] = c0; s_count[2 * kept.id[lane] + 1] = c1; }
      if (lane == kMaxE - 1) {
        meta->off[0] = 0;
        meta->tile_prefix[0] = 0;
        meta->n_skipped = 2 * T - pairs;
        meta->n_touched = touched;
        meta->reserved = 0;
        if (s_count) { *s_nskipped = 2 * T - pairs; *s_ntouched = touched; }
      }
    }
  }
  __syncthreads();
  const int nvec = h >> 3;
  const uint4* src = reinterpret_cast<const uint4*>(x + (size_t)t * h);
  const int p0 = s_p[0], p1 = s_p[1];
  uint4* d0 = reinterpret_cast<uint4*>(xperm + (size_t)p0 * h);
  uint4* d1 = reinterpret_cast<uint4*>(xperm + (size_t)(p1 < 0 ? p0 : p1) * h);
  for (int v = i; v < nvec; v += blockDim.x) {
    const uint4 val = ld_l2(src + v);
    d0[v] = val;
    if (p1 >= 0) d1[v] = val;
  }
}

// Forward batches of more than kDecodeMaxT tokens (up to kRouterTcT on wide rows), and calibration on narrow rows: a
// warp takes the logits of TB tokens.  A lane walks the
// same 8-element slices of the TB rows and of the router rows, so a slice of a router row is read
// and unpacked once for TB tokens; the products of two tokens go through one fma.rn.f32x2.  A logit
// is one chain of fused multiply-adds per lane (slices, then elements, in order) and a butterfly over
// the lanes, whatever the batch and the tokens beside it.
//   - The router rows are copied to shared memory once per block, before the wait for the
//     predecessor (they never change), where they fit beside the ring: read through L1 they cost a
//     chain of L2 round trips per slice, 62 us for 611 tokens.  Longer rows (beyond h = 5824 with 8
//     experts) pass through the same memory in two halves of as many columns as fit: while the warps
//     of the block work on one, all threads fetch the next into the other, with the token slices'
//     groups.  The block then walks its tokens in step, a barrier per part; the sums are the same.
//     (Read through L1 instead: layer of 16 experts, h 6144, f 512, whole forward of 300 tokens 138 us
//     against 121, of 16384 tokens 1324 against 1282; and rows that a caller has just written may not be
//     read that way at all, see the rule beside launch_pdl.)
//   - The token rows come through a ring of kRouteStages slices per warp, filled with cp.async.cg
//     (which reads at L2, as the rule beside launch_pdl asks): a lane copies exactly the bytes it
//     will use itself, so no barrier is needed, and the loads in flight cost no registers.
// Bound by the issue slots of the fp32 work and, beside them, the shared-memory port; 134 MB of token
// rows at 16384 tokens take 20 us to stream.  Router launch, before (one warp per token, router rows
// through L1; a tensor-core kernel from 8192 tokens on: 33 us at 8192) -> after: 611 tokens 19.4 ->
// 10.3 us, 4000 26.7 -> 14.9, 16384 88.9 -> 40.2.
__device__ __forceinline__ uint64_t pack_f32x2(float lo, float hi) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ void fma_f32x2(uint64_t& acc, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ void split_f32x2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ void cp_async16(void* dst_shared, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
               ::"r"((uint32_t)__cvta_generic_to_shared(dst_shared)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Sums N values (a power of two up to 32) over the 32 lanes, halving the values a lane carries at
// every exchange; lane l returns the total of value l / (32 / N).
template <int N, int OFF = 16>
__device__ __forceinline__ float reduce_scatter(const float (&v)[N], int lane) {
  if constexpr (OFF == 0) {
    return v[0];
  } else if constexpr (N == 1) {
    const float one[1] = {v[0] + __shfl_xor_sync(0xffffffffu, v[0], OFF)};
    return reduce_scatter<1, OFF / 2>(one, lane);
  } else {
    const bool up = lane & OFF;
    float half[N / 2];
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
      const float got = __shfl_xor_sync(0xffffffffu, up ? v[i] : v[i + N / 2], OFF);
      half[i] = (up ? v[i + N / 2] : v[i]) + got;
    }
    return reduce_scatter<N / 2, OFF / 2>(half, lane);
  }
}

// R = experts computed (>= r), RP = R rounded up to a power of two, TB = tokens per warp.  A team of
// kTeamWarps warps takes the kRouteTokPerBlock tokens of one row of the permutation's histogram;
// a block of 16 warps is several teams, and the blocks go round until the tokens are done.
constexpr int kRouteStages = 4;
constexpr int kRouteWarps = 16;
template <int R> struct RouteCfg {
  static constexpr int kRP = R <= 2 ? 2 : (R <= 4 ? 4 : (R <= 8 ? 8 : 16));
  static constexpr int kTB = R <= 8 ? 4 : 2;
  static constexpr int kN = kRP * kTB;
  static constexpr int kTeamWarps = kRouteTokPerBlock / kTB;
  static constexpr int kTeams = kRouteWarps / kTeamWarps;
  static constexpr size_t kRingBytes = (size_t)kRouteWarps * kRouteStages * kTB * 32 * 16;
};
constexpr size_t kRouteSmemMax = 227 * 1024 - 8 * 1024;  // dynamic part; the records are static

// 16-byte vectors of a router row that shared memory holds at a time: the whole row, or a part of it (a
// whole number of slices; at least 9 for every R) of which two fit.
template <int R> inline int route_part(int h, int r) {
  const size_t room = kRouteSmemMax - RouteCfg<R>::kRingBytes;
  if ((size_t)r * h * 2 <= room) return h >> 3;
  return (int)(room / 2 / ((size_t)r * 512)) * 32;
}

// Starts the copy of vectors v0 .. of the r router rows, at most `part` of each, to dst[row][part]
// (WHOLE: of the whole rows, which lie one after the other).  Every thread of the block calls it.
template <bool WHOLE>
__device__ __forceinline__ void fetch_router_part(uint4* dst, const bf16* Wg, int v0, int part, int nvec, int r) {
  const uint4* src = reinterpret_cast<const uint4*>(Wg) + v0;
  if (WHOLE) {
    for (int i = threadIdx.x; i < r * nvec; i += 32 * kRouteWarps) cp_async16(dst + i, src + i);
    return;
  }
  const int len = min(part, nvec - v0);
  for (int c = 0; c < r; ++c)
    for (int i = threadIdx.x; i < len; i += 32 * kRouteWarps) cp_async16(dst + c * part + i, src + (size_t)c * nvec + i);
}

// Logits of this warp's tokens t0 .. t0 + TB - 1 (tokens past the end repeat the last): lane l
// returns the one of token q / RP and expert q % RP, q = l / (32 / N); experts beyond r repeat the
// last.  WHOLE: s_w holds the router rows [r][nvec].  Otherwise it holds two parts [2][r][part], the
// first of which is in `half` or on its way there, and all warps of the block call this together, those
// that have no tokens (t0 >= T) to fetch their shares of the parts; the first part comes round again
// behind the last one, for the next call.
template <int R, bool WHOLE>
__device__ __forceinline__ float warp_logits(const bf16* x, uint4* s_w, const bf16* Wg, int part, int& half,
                                             int t0, int T, int h, int r, uint4* ring) {
  const bool on = WHOLE || t0 < T;
  constexpr int RP = RouteCfg<R>::kRP, TB = RouteCfg<R>::kTB, N = RouteCfg<R>::kN;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nvec = h >> 3;
  uint64_t acc[TB / 2][R];  // two tokens each
#pragma unroll
  for (int i = 0; i < TB / 2; ++i)
#pragma unroll
    for (int c = 0; c < R; ++c) acc[i][c] = 0ull;
  const uint4* xr[TB];
#pragma unroll
  for (int i = 0; i < TB; ++i) xr[i] = reinterpret_cast<const uint4*>(x + (size_t)min(t0 + i, T - 1) * h) + lane;
  uint4* mine = ring + warp * (kRouteStages * TB * 32) + lane;  // [stage][token][lane]
  auto fetch = [&](int v, int s) {  // slice v / 32 into stage s
    if (on && v + lane < nvec) {
#pragma unroll
      for (int i = 0; i < TB; ++i) cp_async16(mine + (s * TB + i) * 32, xr[i] + v);
    }
    cp_async_commit();
  };
#pragma unroll
  for (int s = 0; s < kRouteStages - 1; ++s) fetch(32 * s, s);
  int s = 0, left = 0;  // vectors of the present part still to come
  const uint4* w = s_w + lane;
#pragma unroll 1
  for (int v = 0; v < nvec; v += 32, left -= 32) {
    cp_async_wait<kRouteStages - 2>();
    if (!WHOLE && left <= 0) {
      // this part was fetched with or before a token slice that has arrived; no warp reads the other half now
      __syncthreads();
      w = s_w + half * r * part + lane - v;
      half ^= 1;
      left = part;
      const int next = v + part < nvec ? v + part : 0;
      fetch_router_part<WHOLE>(s_w + half * r * part, Wg, next, part, nvec, r);  // committed with the slice below
    }
    if (!on) {
      cp_async_commit();
      continue;
    }
    uint64_t xf[TB / 2][8];
#pragma unroll
    for (int i = 0; i < TB / 2; ++i) {
      float lo[8], hi[8];
      unpack8(mine[(s * TB + 2 * i) * 32], lo);
      unpack8(mine[(s * TB + 2 * i + 1) * 32], hi);
#pragma unroll
      for (int e = 0; e < 8; ++e) xf[i][e] = pack_f32x2(lo[e], hi[e]);
    }
    fetch(v + 32 * (kRouteStages - 1), s == 0 ? kRouteStages - 1 : s - 1);
    if (v + lane < nvec) {
      constexpr int kBatch = 2;  // router slices in flight
#pragma unroll
      for (int c0 = 0; c0 < R; c0 += kBatch) {
        uint4 wv[kBatch];
#pragma unroll
        for (int b = 0; b < kBatch; ++b) wv[b] = w[(size_t)min(c0 + b, r - 1) * (WHOLE ? nvec : part) + v];
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
          if (c0 + b < R) {
            float wf[8];
            unpack8(wv[b], wf);
#pragma unroll
            for (int e = 0; e < 8; ++e)
#pragma unroll
              for (int i = 0; i < TB / 2; ++i)
                fma_f32x2(acc[i][c0 + b < R ? c0 + b : 0], xf[i][e], pack_f32x2(wf[e], wf[e]));
          }
        }
      }
    }
    if (++s == kRouteStages) s = 0;
  }
  float val[N];
#pragma unroll
  for (int q = 0; q < N; ++q) val[q] = 0.f;
#pragma unroll
  for (int i = 0; i < TB / 2; ++i)
#pragma unroll
    for (int c = 0; c < R; ++c) split_f32x2(acc[i][c], val[2 * i * RP + c], val[(2 * i + 1) * RP + c]);
  return reduce_scatter<N>(val, lane);
}

// Top-2 routing.
template <int R, bool WHOLE>
__global__ void __launch_bounds__(32 * kRouteWarps, 1)
router_kernel(const bf16* x, const bf16* Wg, int T, int h, int r, int part, float beta, KeptIds kept,
              RouteOut o, bool w_const) {
  pdl_launch_dependents();
  using Cfg = RouteCfg<R>;
  constexpr int RP = Cfg::kRP, TB = Cfg::kTB, N = Cfg::kN;
  extern __shared__ uint4 ring[];
  __shared__ float s_l[kRouteWarps][N];
  __shared__ int s_e[Cfg::kTeams][kRouteTokPerBlock][2];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int team = warp / Cfg::kTeamWarps, tw = warp % Cfg::kTeamWarps;
  uint4* s_w = ring + Cfg::kRingBytes / 16;
  if (w_const) fetch_router_part<WHOLE>(s_w, Wg, 0, part, h >> 3, r);
  pdl_wait();
  if (!w_const) fetch_router_part<WHOLE>(s_w, Wg, 0, part, h >> 3, r);
  cp_async_commit();
  if (WHOLE) {
    cp_async_wait<0>();
    __syncthreads();
  }
  const int units = (T + kRouteTokPerBlock - 1) / kRouteTokPerBlock;
  int half = 0;
  // with the rows in parts all warps of the block stay in step: a team goes on while the first has a unit
  for (int u = blockIdx.x + gridDim.x * team; u - (WHOLE ? 0 : (int)gridDim.x * team) < units; u += gridDim.x * Cfg::kTeams) {
    const int t0 = u * kRouteTokPerBlock;
    const float mine = warp_logits<R, WHOLE>(x, s_w, Wg, part, half, t0 + tw * TB, T, h, r, ring);
    if (!WHOLE && u >= units) continue;
    if (lane % (32 / N) == 0) s_l[warp][lane / (32 / N)] = mine;
    __syncwarp();
    const int i = tw * TB + lane, t = t0 + i;
    int e0 = -1, e1 = -1;
    bool skip = false;
    if (lane < TB && t < T) {
      float l[R];
#pragma unroll
      for (int c = 0; c < R; ++c) l[c] = s_l[warp][lane * RP + c];
      route_decide<R>(l, r, beta, t, kept, o, e0, e1, skip);
      if (skip) e1 = -1;
    }
    __syncwarp();
    if (!o.blk_hist) continue;
    // pair counts of the unit, by the team's threads
    if (lane < TB) { s_e[team][i][0] = e0; s_e[team][i][1] = e1; }
    constexpr int kTeamThreads = 32 * Cfg::kTeamWarps;
    asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "n"(kTeamThreads) : "memory");
    const int col = threadIdx.x - team * kTeamThreads;
    if (col < kHistCols) {
      const int n_tok = min(kRouteTokPerBlock, T - t0);
      int n = 0;
      if (col == 2 * kMaxE) {
        for (int q = 0; q < n_tok; ++q) n += s_e[team][q][1] < 0;
      } else {
        const int c = col >> 1, slot = col & 1;
        for (int q = 0; q < n_tok; ++q) n += (s_e[team][q][slot] == c);
      }
      o.blk_hist[(size_t)u * kHistCols + col] = n;
    }
    asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "n"(kTeamThreads) : "memory");
  }
  if (!WHOLE) cp_async_wait<0>();  // the first part, fetched once more behind the last
}

// Calibration (where calibrate_on_tiles says so), the top-k and the search router: a team of TW warps takes
// tiles of 8 NT tokens in turn, its warps sharing the columns of a row (blocks of 64 columns); a block of
// kRouteWarps warps is one team or several.  The products of 16 columns of up to 16 tokens with 8 router rows are
// one mma.sync.m16n8k16: a [T x h] x [h x 16] contraction is bound by reading the token rows, which a handful of
// warp-level instructions keeps up with, and tokens go from global memory to the instruction's registers without
// passing through shared or tensor memory (the order of the columns inside a block is free, so the 16 bytes of a
// row that a lane reads are its operands of two instructions).  Whole calibration call, before (router_kernel) ->
// after, us: h 4096, 8 experts, 300 tokens 23.9 -> 19.4, 8192 37.1 -> 27.7, 16384 56.8 -> 52.9, 32768 97.4 -> 85.8;
// h 2048, 16 experts, 16384 tokens 60.3 -> 36.5.  With 2 to 4 experts router_kernel, which then has half the arithmetic,
// stays ahead on long batches.  Forms that were slower (16384 tokens, when this one took 50): one warp that decides
// while the others wait 67, 8 tokens as the narrow operand (twice the instructions) 61, prefetching deeper to L2 58-60;
// a column phase of its own per block changed nothing.  Top-k calls in a row of layers with few columns or experts lose
// 1-3 us to the router of chains of multiply-adds that ran before (E 4, h 512, f 64, 1000 tokens 33.4 -> 35.7 us a
// call; alone the launch takes as long); tiles for teams of 4 warps or two blocks per SM did not change that.
//   - A logit: sums of 64 products by the tensor core, added up by each warp in column order and then over the
//     warps, both as compensated fp32 sums (the tensor core drops bits that an IEEE addition would round, which
//     costs little over 64 products and too much over a row).
//   - The router rows wait in shared memory in operand order, fetched before the wait for the predecessor where
//     they never change; rows too long for it (h beyond 10880 with 8 experts, 4416 with 16) are read at L2.
//   - A lane has 8 NT slots of 16 bytes; a slot is refilled, from the next tile if need be, as soon as it is used, in
//     order, so that fewer than that are in flight on average.
//   - After a tile's one barrier every warp of the team adds up and decides its share of the tokens.

// d += A (16 tokens x 16 columns) B (16 columns x 8 router rows)
__device__ __forceinline__ void mma_16x8(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// Compensated sum: `lost` collects exactly what each addition drops (Knuth's two-sum), the sum is acc + lost.
// Adding zero changes neither.
__device__ __forceinline__ void add_compensated(float& acc, float& lost, float v) {
  const float sum = __fadd_rn(acc, v), part = __fsub_rn(sum, acc);
  lost = __fadd_rn(lost, __fadd_rn(__fsub_rn(acc, __fsub_rn(sum, part)), __fsub_rn(v, part)));
  acc = sum;
}
// (an infinite sum has lost NaN)
__device__ __forceinline__ float closed_sum(float acc, float lost) { return lost == lost ? acc + lost : acc; }

constexpr int kRouteSlots = 4;  // blocks of 64 columns that a warp has in flight
constexpr size_t kTileSmemMax = 227 * 1024 - 9 * 1024;  // dynamic part; the records are static
// R = experts computed (>= r; 8 or 16), NT = groups of 8 tokens in a tile, TW = warps of a team
template <int R, int NT, int TW> struct TileCfg {
  static constexpr int kTeams = kRouteWarps / TW;
  static constexpr int kPlanes = R > 8 ? 2 : 1;         // 8 router rows each
  static constexpr int kTokens = 8 * NT;
  static constexpr int kStride = R > 8 ? 20 : 12;       // floats per token: spreads the tokens over the banks
  static constexpr int kPart = kTokens * kStride;       // floats a warp leaves, twice (sums, what they lost)
  static constexpr size_t kPartBytes = (size_t)4 * kRouteWarps * kPart * 4;
  static size_t w_bytes(int h) { return (size_t)((h + 63) / 64) * kPlanes * 1024; }
  // a tile's decision: kRP lanes per token, kTPP tokens per pass, kLanes lanes with the same logit
  static constexpr int kRP = R;
  static constexpr int kTPW = kTokens > TW ? kTokens / TW : 1;  // tokens of a warp
  static constexpr int kTPP = kTPW * kRP > 32 ? 32 / kRP : kTPW;
  static constexpr int kLanes = 32 / (kTPP * kRP);
};

// 16 bytes of a token row, read at L2 (the rule beside launch_pdl); their 256 bytes are fetched to L2 along with them.
// `once`: a batch that L2 does not hold; the lines in flight are not allocated in L1 either, which holds few of
// them beside the shared memory (14000 / 16384 / 32768 tokens of h 4096 from DRAM 52.1 / 54.8 / 91.8 -> 49.6 / 51.3 /
// 85.4 us; 8192 tokens, from L2, 27.9 -> 30.9).
__device__ __forceinline__ uint4 ld_row(const uint4* p, bool once) {
  uint4 v;
  if (once)
    asm volatile("ld.relaxed.gpu.global.L1::no_allocate.L2::256B.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  else
    asm volatile("ld.global.cg.L2::256B.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}
constexpr size_t kRouteOnceBytes = (size_t)96 << 20;
template <int N> __device__ __forceinline__ void named_sync(int id) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(N) : "memory");
}
// Calls decide(t0, n, mine) for all tokens, up to kTPP of them at a time (t0 .. t0 + n - 1; none if n <= 0), by a
// converged warp: a lane brings the logit of token t0 + lane / kLanes / kRP and expert lane / kLanes % kRP (beyond
// n and r: anything).
// WHOLE: the router rows pass through shared memory.
template <int R, int NT, int TW, bool WHOLE, class Decide>
__device__ __forceinline__ void route_tiles(const bf16* x, const bf16* Wg, int T, int h, int r, bool w_const,
                                            Decide&& decide) {
  using Cfg = TileCfg<R, NT, TW>;
  constexpr int PL = Cfg::kPlanes, S = Cfg::kStride, U = kRouteSlots;
  constexpr int kMembers = 32 * TW;
  extern __shared__ uint4 s_dyn[];
  uint4* s_w = s_dyn + Cfg::kPartBytes / 16;        // [block of 64 columns][plane][half][lane]
  const int team = threadIdx.x / kMembers, warp = threadIdx.x / 32 % TW;
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  float* s_part = reinterpret_cast<float*>(s_dyn) + team * 4 * TW * Cfg::kPart;  // [2][warp][sum, lost][token][S]
  const int nvec = h >> 3, blocks = (h + 63) >> 6;
  auto fetch_w = [&]() {
    if (!WHOLE) return;
    for (int i = threadIdx.x; i < blocks * PL * 64; i += 32 * kRouteWarps) {
      const int row = (i >> 2 & 7) + 8 * (i / 64 % PL), v = 8 * (i / (64 * PL)) + 4 * (i >> 5 & 1) + (i & 3);
      if (row >= r) continue;  // whatever lies there only reaches the sums of experts that do not exist
      if (v < nvec) cp_async16(s_w + i, reinterpret_cast<const uint4*>(Wg) + (size_t)row * nvec + v);
      else s_w[i] = make_uint4(0u, 0u, 0u, 0u);
    }
  };
  if (w_const) fetch_w();
  pdl_wait();
  if (!w_const) fetch_w();

  const int tiles = (T + Cfg::kTokens - 1) / Cfg::kTokens, stride = (int)gridDim.x * Cfg::kTeams;
  const int rounds = (blocks + U * TW - 1) / (U * TW);
  const bool once = (size_t)T * h * 2 > kRouteOnceBytes;
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
  uint4 slot[U][NT][2];  // [block][8 tokens][half]
  const uint4* row[NT];
  // one team for the whole block: neighbouring warps, neighbouring blocks; small teams: a warp reads 512 bytes
  // of a row at a time
  constexpr bool kDeal = TW == kRouteWarps;
  auto block_of = [&](int b, int u) { return kDeal ? (b * U + u) * TW + warp : (b * TW + warp) * U + u; };
  auto set_rows = [&](int tile) {
#pragma unroll
    for (int n = 0; n < NT; ++n)
      row[n] = reinterpret_cast<const uint4*>(x) + (size_t)min(tile * Cfg::kTokens + 8 * n + g, T - 1) * nvec + q;
  };
  auto fill = [&](int c, uint4 (&dst)[NT][2]) {
    if (8 * c + 8 <= nvec) {
#pragma unroll
      for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int o = 0; o < 2; ++o) dst[n][o] = ld_row(row[n] + 8 * c + 4 * o, once);
    } else if (8 * c < nvec) {  // the last, partly filled block
#pragma unroll
      for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int o = 0; o < 2; ++o) dst[n][o] = 8 * c + 4 * o + q < nvec ? ld_row(row[n] + 8 * c + 4 * o, once) : zero;
    }
  };
  auto take = [&](int tile, int b) {  // this warp's tokens
    constexpr int RP = Cfg::kRP, TPP = Cfg::kTPP, kLanes = Cfg::kLanes;
    const int used = min(TW, kDeal ? blocks : (blocks + U - 1) / U);  // warps that have columns
    const int i = lane / kLanes / RP, c = min(lane / kLanes % RP, R - 1);
    if (warp * Cfg::kTPW >= Cfg::kTokens) return;
#pragma unroll
    for (int p = 0; p < Cfg::kTPW / TPP; ++p) {
      const int first = warp * Cfg::kTPW + p * TPP;
      const float* from = s_part + b * TW * 2 * Cfg::kPart + (first + i) * S + c;
      float sum = 0.f, drop = 0.f;
      for (int w = lane % kLanes; w < used; w += kLanes) {
        add_compensated(sum, drop, from[w * 2 * Cfg::kPart]);
        drop += from[w * 2 * Cfg::kPart + Cfg::kPart];
      }
#pragma unroll
      for (int o = 1; o < kLanes; o <<= 1) {  // lower lane first on both sides: the same bits
        const float s1 = __shfl_xor_sync(0xffffffffu, sum, o), d1 = __shfl_xor_sync(0xffffffffu, drop, o);
        const bool up = lane & o;
        float acc = up ? s1 : sum;
        drop = up ? d1 + drop : drop + d1;
        add_compensated(acc, drop, up ? sum : s1);
        sum = acc;
      }
      decide(tile * Cfg::kTokens + first, min(TPP, T - tile * Cfg::kTokens - first), closed_sum(sum, drop));
    }
  };
  int tile = blockIdx.x + gridDim.x * team;
  if (tile < tiles) {
    set_rows(tile);
#pragma unroll
    for (int u = 0; u < U; ++u) fill(block_of(0, u), slot[u]);
  }
  if (WHOLE) {
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
  }
  int it = 0;
  for (; tile < tiles; tile += stride, ++it) {
    float acc[PL][4], lost[PL][4];
#pragma unroll
    for (int p = 0; p < PL; ++p)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[p][i] = lost[p][i] = 0.f;
#pragma unroll 1
    for (int b = 0; b < rounds; ++b) {
      const bool last = b + 1 == rounds, more = !last || tile + stride < tiles;
      if (last && more) set_rows(tile + stride);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int c = block_of(b, u);
        if (c < blocks) {
#pragma unroll
          for (int p = 0; p < PL; ++p) {
            float sum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int o = 0; o < 2; ++o) {
              uint4 w;
              if (WHOLE) w = s_w[((c * PL + p) * 2 + o) * 32 + lane];
              else w = 8 * c + 4 * o + q < nvec
                           ? ld_l2(reinterpret_cast<const uint4*>(Wg) + (size_t)min(g + 8 * p, r - 1) * nvec + 8 * c + 4 * o + q)
                           : zero;
              const uint4 lo = slot[u][0][o], hi = NT > 1 ? slot[u][NT - 1][o] : zero;
              mma_16x8(sum, lo.x, hi.x, lo.y, hi.y, w.x, w.y);
              mma_16x8(sum, lo.z, hi.z, lo.w, hi.w, w.z, w.w);
            }
#pragma unroll
            for (int i = 0; i < 2 * NT; ++i) add_compensated(acc[p][i], lost[p][i], sum[i]);
          }
        }
        if (more) fill(block_of(last ? 0 : b + 1, u), slot[u]);
      }
    }
    const int b = it & 1;
    float* mine = s_part + (b * TW + warp) * 2 * Cfg::kPart;
#pragma unroll
    for (int p = 0; p < PL; ++p)
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        float* at = mine + (8 * n + g) * S + 8 * p + 2 * q;
        *reinterpret_cast<float2*>(at) = make_float2(acc[p][2 * n], acc[p][2 * n + 1]);
        *reinterpret_cast<float2*>(at + Cfg::kPart) = make_float2(lost[p][2 * n], lost[p][2 * n + 1]);
      }
    __syncwarp();
    named_sync<kMembers>(1 + team);
    take(tile, b);
  }
}

// Calibration: w_e1 / w_e0 of every token.
template <int R, int NT, int TW, bool WHOLE>
__global__ void __launch_bounds__(32 * kRouteWarps, 1)
ratio_kernel(const bf16* x, const bf16* Wg, int T, int h, int r, float* __restrict__ ratio, bool w_const) {
  pdl_launch_dependents();
  using Cfg = TileCfg<R, NT, TW>;
  const int lane = threadIdx.x & 31;
  route_tiles<R, NT, TW, WHOLE>(x, Wg, T, h, r, w_const, [&](int t0, int n, float mine) {
    constexpr int kPer = Cfg::kRP * Cfg::kLanes;  // lanes of a token
    const int i = lane / kPer;
    float l[R], w0, w1, p1;
#pragma unroll
    for (int c = 0; c < R; ++c) l[c] = __shfl_sync(0xffffffffu, mine, i * kPer + c * Cfg::kLanes);
    if (lane % kPer || i >= n) return;
    int e0, e1;
    bool skip;
    route_choose<R>(l, r, 0.f, e0, e1, skip, w0, w1, p1);
    ratio[t0 + i] = p1;
  });
}

// ---------------------------------------------------------------------------------- scan

// One block.  Warp c scans the per-block counts of expert c over the blocks in order, which
// gives every block its first position inside the expert's group; thread 0 then lays the
// groups out (each padded to `pad` rows) and counts the 128-row tiles.
__global__ void __launch_bounds__(1024)
scan_kernel(const int32_t* blk_hist, int nblk, int r, int pad,
            int32_t* __restrict__ blk_base, Meta* meta, int32_t* s_count, int32_t* s_nskipped,
            int32_t* s_ntouched, KeptIds kept, int E) {
  pdl_launch_dependents();
  pdl_wait();
  __shared__ int s_tot[kMaxE][2];
  __shared__ int s_skipped;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp < r) {
    int run = 0, run0 = 0;
    // the loads of a step do not depend on the running sums: let several steps be in flight
#pragma unroll 4
    for (int b0 = 0; b0 < nblk; b0 += 32) {
      const int b = b0 + lane;
      int v0 = 0, v1 = 0;
      if (b < nblk) {
        v0 = ld_l2(blk_hist + (size_t)b * kHistCols + 2 * warp);
        v1 = ld_l2(blk_hist + (size_t)b * kHistCols + 2 * warp + 1);
      }
      const int v = v0 + v1;
      int inc = v;
#pragma unroll
      for (int s = 1; s < 32; s <<= 1) {
        const int n = __shfl_up_sync(0xffffffffu, inc, s);
        if (lane >= s) inc += n;
      }
      if (b < nblk) blk_base[(size_t)b * kMaxE + warp] = run + inc - v;
      run += __shfl_sync(0xffffffffu, inc, 31);
      int t0 = v0;
#pragma unroll
      for (int s = 16; s > 0; s >>= 1) t0 += __shfl_xor_sync(0xffffffffu, t0, s);
      run0 += t0;
    }
    if (lane == 0) { s_tot[warp][0] = run0; s_tot[warp][1] = run - run0; }
  } else if (warp == kMaxE) {
    int n = 0;
    for (int b = lane; b < nblk; b += 32) n += ld_l2(blk_hist + (size_t)b * kHistCols + 2 * kMaxE);
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) n += __shfl_xor_sync(0xffffffffu, n, s);
    if (lane == 0) s_skipped = n;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int off = 0, tiles = 0, touched = 0;
    meta->off[0] = 0;
    meta->tile_prefix[0] = 0;
    for (int c = 0; c < kMaxE; ++c) {
      const int n0 = c < r ? s_tot[c][0] : 0, n1 = c < r ? s_tot[c][1] : 0;
      const int n = n0 + n1;
      meta->count[c] = n;
      meta->count_slot[c][0] = n0;
      meta->count_slot[c][1] = n1;
      off += (n + pad - 1) / pad * pad;
      tiles += (n + kTileRows - 1) / kTileRows;
      touched += (n > 0);
      meta->off[c + 1] = off;
      meta->tile_prefix[c + 1] = tiles;
    }
    meta->n_skipped = s_skipped;
    meta->n_touched = touched;
    meta->reserved = 0;
    if (s_count) {
      for (int e = 0; e < E; ++e) { s_count[2 * e] = 0; s_count[2 * e + 1] = 0; }
      for (int c = 0; c < r; ++c) {
        s_count[2 * kept.id[c]] = s_tot[c][0];
        s_count[2 * kept.id[c] + 1] = s_tot[c][1];
      }
      *s_nskipped = s_skipped;
      *s_ntouched = touched;
    }
  }
}

// ------------------------------------------------------------------------------- permute

// Permutation and gather of batches beyond kDecodeMaxT tokens: block (b, y) places the pairs of the
// kRouteTokPerBlock tokens of unit b and copies column share y of their rows to the places.
// TOP2: two slots per token, the second off where `active` (the skip flag) is set; otherwise k slots,
// the first `active` of them on.
// Position of a pair = start of its expert's group + pairs of that expert in earlier units + pairs of
// that expert among the earlier tokens of the unit.  blk_base == null (at most kPermuteOwnT tokens):
// every block counts the pairs of the whole routing record and of the units before its own itself,
// which costs a block a few microseconds and saves the launches of a histogram and a scan; block
// (0, 0) publishes the batch description.  Else both come from the scan.
// The rows between a group's end and its padded end are zeroed (the tensor cores draw less power on
// zeros than on stale rows).
// Bound by the copy (x once, its k places once); before, as memset + count + scan + scatter + gather
// with x read once per slot: 611 tokens, two slots 21 -> 10.8 us of kernel time and three launches
// less; 8192 tokens, six slots 172 -> 135 us.
__device__ __forceinline__ void count_pair(uint64_t (&n)[2], int e) {  // one byte per expert
  const uint64_t one = 1ull << (8 * (e & 7));
  if (e < 8) n[0] += one;
  else n[1] += one;
}

template <bool TOP2>
__global__ void __launch_bounds__(256)
permute_kernel(const bf16* x, const int32_t* idx, const void* active, int T, int k, int h, int r, int pad,
               const int32_t* blk_base, Meta* meta, int32_t* __restrict__ pair_pos, bf16* __restrict__ xperm,
               int32_t* s_count, int32_t* s_nskipped, int32_t* s_ntouched, KeptIds kept, int E) {
  pdl_launch_dependents();
  pdl_wait();
  __shared__ int s_part[3][8][kMaxE];  // slot-0 pairs, other pairs, pairs of earlier units; per warp
  __shared__ int s_off[kMaxE], s_cnt[kMaxE], s_end[kMaxE], s_base[kMaxE];
  __shared__ int s_e[kRouteTokPerBlock][kMaxE];
  __shared__ int s_pos[kRouteTokPerBlock][kMaxE];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int t0 = blockIdx.x * kRouteTokPerBlock;
  auto n_active = [&](int t) {
    if (TOP2) return ld_l2(reinterpret_cast<const uint8_t*>(active) + t) ? 1 : 2;
    return ld_l2(reinterpret_cast<const int32_t*>(active) + t);
  };
  if (blk_base == nullptr) {
    uint64_t n0[2] = {0, 0}, n1[2] = {0, 0}, nb[2] = {0, 0};
    for (int t = tid; t < T; t += 256) {
      const int n = n_active(t);
      const int32_t* e = idx + (size_t)t * k;
      const int first = ld_l2(e);
      count_pair(n0, first);
      if (t < t0) count_pair(nb, first);
      for (int m = 1; m < n; ++m) {
        const int em = ld_l2(e + m);
        count_pair(n1, em);
        if (t < t0) count_pair(nb, em);
      }
    }
    for (int c = 0; c < r; ++c) {
      const int q = c >> 3, s = 8 * (c & 7);
      const unsigned v0 = __reduce_add_sync(0xffffffffu, (unsigned)((q ? n0[1] : n0[0]) >> s) & 255u);
      const unsigned v1 = __reduce_add_sync(0xffffffffu, (unsigned)((q ? n1[1] : n1[0]) >> s) & 255u);
      const unsigned vb = __reduce_add_sync(0xffffffffu, (unsigned)((q ? nb[1] : nb[0]) >> s) & 255u);
      if (lane == 0) { s_part[0][warp][c] = (int)v0; s_part[1][warp][c] = (int)v1; s_part[2][warp][c] = (int)vb; }
    }
  }
  // the unit's own pairs
  if (tid < kRouteTokPerBlock * kMaxE) {
    const int tl = tid / kMaxE, m = tid % kMaxE, t = t0 + tl;
    s_e[tl][m] = (m < k && t < T && m < n_active(t)) ? ld_l2(idx + (size_t)t * k + m) : -1;
  }
  __syncthreads();
  if (warp == 0) {
    const bool on = lane < r;
    int off, cnt, padded, base;
    if (blk_base == nullptr) {
      int c0 = 0, c1 = 0, before = 0;
      for (int w = 0; on && w < 8; ++w) {
        c0 += s_part[0][w][lane];
        c1 += s_part[1][w][lane];
        before += s_part[2][w][lane];
      }
      cnt = c0 + c1;
      padded = (cnt + pad - 1) / pad * pad;
      const int mine_tiles = (cnt + kTileRows - 1) / kTileRows;
      int end = padded, tiles = mine_tiles;  // inclusive sums over the experts
#pragma unroll
      for (int s = 1; s < kMaxE; s <<= 1) {
        const int a = __shfl_up_sync(0xffffffffu, end, s), b = __shfl_up_sync(0xffffffffu, tiles, s);
        if (lane >= s) { end += a; tiles += b; }
      }
      off = end - padded;
      base = off + before;
      if (blockIdx.x == 0 && blockIdx.y == 0) {
        const int pairs = __reduce_add_sync(0xffffffffu, cnt);
        const int touched = __popc(__ballot_sync(0xffffffffu, cnt > 0));
        if (lane < kMaxE) {
          meta->count[lane] = cnt;
          meta->count_slot[lane][0] = TOP2 ? c0 : cnt;
          meta->count_slot[lane][1] = TOP2 ? c1 : 0;
          meta->off[lane + 1] = end;
          meta->tile_prefix[lane + 1] = tiles;
          if (s_count && lane < E) { s_count[2 * lane] = 0; s_count[2 * lane + 1] = 0; }
        }
        __syncwarp();
        if (s_count && on) { s_count[2 * kept.id[lane]] = c0; s_count[2 * kept.id[lane] + 1] = c1; }
        if (lane == kMaxE - 1) {
          meta->off[0] = 0;
          meta->tile_prefix[0] = 0;
            meta->n_skipped = T * k - pairs;
          meta->n_touched = touched;
          meta->reserved = 0;
          if (s_count) { *s_nskipped = T * k - pairs; *s_ntouched = touched; }
        }
      }
    } else {
      off = on ? ld_l2(&meta->off[lane]) : 0;
      cnt = on ? ld_l2(&meta->count[lane]) : 0;
      padded = on ? ld_l2(&meta->off[lane + 1]) - off : 0;
      base = on ? off + ld_l2(blk_base + (size_t)blockIdx.x * kMaxE + lane) : 0;
    }
    if (on) { s_off[lane] = off; s_cnt[lane] = cnt; s_end[lane] = off + padded; s_base[lane] = base; }
  }
  __syncthreads();
  if (tid < kRouteTokPerBlock * kMaxE) {
    const int tl = tid / kMaxE, m = tid % kMaxE, c = s_e[tl][m];
    int pos = -1;
    if (c >= 0) {
      int rank = 0;
      for (int i = 0; i < tl; ++i)
        for (int q = 0; q < k; ++q) rank += (s_e[i][q] == c);
      pos = s_base[c] + rank;
    }
    s_pos[tl][m] = pos;
    if (blockIdx.y == 0 && m < k && t0 + tl < T) pair_pos[(size_t)(t0 + tl) * k + m] = pos;
  }
  __syncthreads();
  const int nvec = h >> 3;
  const int share = (nvec + gridDim.y - 1) / gridDim.y;
  const int v0 = blockIdx.y * share, v1 = min(nvec, v0 + share);
  uint4* rows = reinterpret_cast<uint4*>(xperm);
  for (int tl = warp; tl < kRouteTokPerBlock && t0 + tl < T; tl += 8) {
    const uint4* src = reinterpret_cast<const uint4*>(x + (size_t)(t0 + tl) * h);
    constexpr int kAhead = 8;  // loads in flight per lane
    for (int v = v0 + lane; v < v1; v += 32 * kAhead) {
      uint4 val[kAhead];
#pragma unroll
      for (int a = 0; a < kAhead; ++a)
        if (v + 32 * a < v1) val[a] = ld_l2(src + v + 32 * a);
      for (int m = 0; m < k; ++m) {
        const int pos = s_pos[tl][m];
        if (pos < 0) continue;
        uint4* dst = rows + (size_t)pos * nvec;
#pragma unroll
        for (int a = 0; a < kAhead; ++a)
          if (v + 32 * a < v1) dst[v + 32 * a] = val[a];
      }
    }
  }
  for (int c = blockIdx.x; c < r; c += gridDim.x)
    for (int row = s_off[c] + s_cnt[c] + warp; row < s_end[c]; row += 8)
      for (int v = v0 + lane; v < v1; v += 32) rows[(size_t)row * nvec + v] = make_uint4(0u, 0u, 0u, 0u);
}

// ------------------------------------------------------------------------------- combine

__global__ void __launch_bounds__(128)
combine_kernel(const float* O, int ksplit, size_t split_stride, const int32_t* pair_pos,
               const float* wn, const bf16* residual, int T, int h, int v0, int v1, bf16* y) {
  pdl_launch_dependents();
  pdl_wait();
  const int t = blockIdx.x;
  const int p0 = ld_l2(pair_pos + 2 * t), p1 = ld_l2(pair_pos + 2 * t + 1);
  const float w0 = ld_l2(wn + 2 * t), w1 = ld_l2(wn + 2 * t + 1);
  for (int v = v0 + blockIdx.y * blockDim.x + threadIdx.x; v < v1; v += gridDim.y * blockDim.x) {
    float a[8], b[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) { a[k] = 0.f; b[k] = 0.f; }
#pragma unroll 4
    for (int s = 0; s < ksplit; ++s) {
      const float4* o0 = reinterpret_cast<const float4*>(O + s * split_stride + (size_t)p0 * h) + 2 * v;
      const float4 q0 = ld_l2(o0), q1 = ld_l2(o0 + 1);
      a[0] += q0.x; a[1] += q0.y; a[2] += q0.z; a[3] += q0.w;
      a[4] += q1.x; a[5] += q1.y; a[6] += q1.z; a[7] += q1.w;
      if (p1 >= 0) {
        const float4* o1 = reinterpret_cast<const float4*>(O + s * split_stride + (size_t)p1 * h) + 2 * v;
        const float4 r0 = ld_l2(o1), r1 = ld_l2(o1 + 1);
        b[0] += r0.x; b[1] += r0.y; b[2] += r0.z; b[3] += r0.w;
        b[4] += r1.x; b[5] += r1.y; b[6] += r1.z; b[7] += r1.w;
      }
    }
    float z[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) z[k] = (p1 >= 0) ? fmaf(w1, b[k], w0 * a[k]) : w0 * a[k];
    if (residual) {
      float rf[8];
      unpack8(ld_l2(reinterpret_cast<const uint4*>(residual + (size_t)t * h) + v), rf);
#pragma unroll
      for (int k = 0; k < 8; ++k) z[k] += rf[k];
    }
    uint4 outv;
    outv.x = pack2(z[0], z[1]); outv.y = pack2(z[2], z[3]);
    outv.z = pack2(z[4], z[5]); outv.w = pack2(z[6], z[7]);
    reinterpret_cast<uint4*>(y + (size_t)t * h)[v] = outv;
  }
}


// ------------------------------------------------------------------ general top-k path

// Top-k routing with the generalised skipping rule of App. A.2:
//   e_0..e_{k-1} = kept experts with the k largest logits (ties to the lower index),
//   p_m = exp(l_em - l_e0);  keep the top i* = min i : sum_{m>i} p_m <= beta * sum_{m<=k} p_m;
//   weights p_m / sum_{m<=i*} p_m.  The fp32 summation orders are fixed: total ascending in m,
//   tails from the smallest upwards, kept mass ascending in m.
// Ranking by counting, one lane per (token, kept expert): the rank of expert c is the number of kept
// experts that beat it (larger logit, or equal logit and lower index), so the expert of rank m is
// the m-th choice; the three sums are one lane's per token (k <= 16 values).
template <int R, int NT, int TW, bool WHOLE>
__global__ void __launch_bounds__(32 * kRouteWarps, 1)
router_topk_kernel(const bf16* x, const bf16* Wg, int T, int h, int r, int k, float beta, KeptIds kept,
                   int32_t* __restrict__ idx, float* __restrict__ wn, int32_t* __restrict__ nact,
                   int32_t* u_idx, float* u_wn, int32_t* u_nact, float* logits) {
  pdl_launch_dependents();
  using Cfg = TileCfg<R, NT, TW>;
  constexpr int RP = Cfg::kRP, TPP = Cfg::kTPP, kLanes = Cfg::kLanes;
  __shared__ float s_p[kRouteWarps][TPP][RP];
  __shared__ int s_sel[kRouteWarps][TPP][RP];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  route_tiles<R, NT, TW, WHOLE>(x, Wg, T, h, r, true, [&](int t0, int n, float mine) {
    const int i = lane / kLanes / RP, c = lane / kLanes % RP;
    int rank = 0;
    float top = -INFINITY;
    for (int d = 0; d < r; ++d) {
      const float o = __shfl_sync(0xffffffffu, mine, (i * RP + d) * kLanes);
      rank += (o > mine) || (o == mine && d < c);
      top = d == 0 || o > top ? o : top;
    }
    if (lane % kLanes == 0) {  // logits that compare with nothing (NaN) leave ranks unclaimed: name some expert
      s_sel[warp][i][c] = min(c, r - 1);
      s_p[warp][i][c] = 0.f;
    }
    __syncwarp();
    if (c < r && lane % kLanes == 0) {
      if (logits && i < n) logits[(size_t)(t0 + i) * r + c] = mine;
      if (rank < k) {
        s_sel[warp][i][rank] = c;
        s_p[warp][i][rank] = expf(mine - top);
      }
    }
    __syncwarp();
    const int t = t0 + lane;
    if (lane < n) {
      const float* p = s_p[warp][lane];
      const int* sel = s_sel[warp][lane];
      // i* = the smallest i in 1..k whose dropped mass p_i + .. + p_{k-1} (added from the smallest
      // value upwards) is at most beta times the whole mass p_0 + .. + p_{k-1} (added in rank order)
      float whole = 0.f;
      for (int m = 0; m < k; ++m) whole += p[m];
      const float bound = beta * whole;
      float dropped = 0.f;  // mass beyond rank istar - 1, for istar = k, k - 1, ..: walk down while it fits
      int istar = k;
      while (istar > 1 && dropped + p[istar - 1] <= bound) { dropped += p[istar - 1]; --istar; }
      float kept_mass = 0.f;
      for (int m = 0; m < istar; ++m) kept_mass += p[m];
      for (int m = 0; m < k; ++m) {
        const float w = m < istar ? p[m] / kept_mass : 0.f;
        const int e = sel[m];
        idx[(size_t)t * k + m] = e;
        wn[(size_t)t * k + m] = w;
        if (u_idx) u_idx[(size_t)t * k + m] = kept.id[e];
        if (u_wn) u_wn[(size_t)t * k + m] = w;
      }
      nact[t] = istar;
      if (u_nact) u_nact[t] = istar;
    }
    __syncwarp();
  });
}

// Per block of kRouteTokPerBlock tokens: active pairs per expert, in the column layout scan_kernel reads
// (the pairs go to the slot-0 column, the skipped pairs to the last column).
__global__ void __launch_bounds__(kHistCols < 64 ? 64 : kHistCols)
count_topk_kernel(const int32_t* __restrict__ idx, const int32_t* __restrict__ nact, int T, int k,
                  int32_t* __restrict__ blk_hist) {
  const int t0 = blockIdx.x * kRouteTokPerBlock;
  const int col = threadIdx.x;
  if (col >= kHistCols) return;
  int n = 0;
  const int t1 = min(T, t0 + kRouteTokPerBlock);
  if (col == 2 * kMaxE) {
    for (int t = t0; t < t1; ++t) n += k - nact[t];
  } else if ((col & 1) == 0) {
    const int c = col >> 1;
    for (int t = t0; t < t1; ++t)
      for (int m = 0; m < nact[t]; ++m) n += (idx[(size_t)t * k + m] == c);
  }
  blk_hist[(size_t)blockIdx.x * kHistCols + col] = n;
}

__global__ void __launch_bounds__(128)
combine_topk_kernel(const float* O, int ksplit, size_t split_stride, const int32_t* pair_pos, const float* wn,
                    int k, int T, int h, bf16* y) {
  pdl_launch_dependents();
  pdl_wait();
  constexpr int kAhead = 4;  // slots whose loads are in flight together
  __shared__ int s_p[kMaxE];
  __shared__ float s_w[kMaxE];
  const int t = blockIdx.x;
  const int nvec = h >> 3;
  if (threadIdx.x < kMaxE) {
    const bool on = (int)threadIdx.x < k;
    s_p[threadIdx.x] = on ? ld_l2(pair_pos + (size_t)t * k + threadIdx.x) : -1;
    s_w[threadIdx.x] = on ? ld_l2(wn + (size_t)t * k + threadIdx.x) : 0.f;
  }
  __syncthreads();
  for (int v = blockIdx.y * blockDim.x + threadIdx.x; v < nvec; v += gridDim.y * blockDim.x) {
    float z[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) z[q] = 0.f;
    for (int m0 = 0; m0 < k; m0 += kAhead) {
      float4 q0[kAhead], q1[kAhead];
#pragma unroll
      for (int m = 0; m < kAhead; ++m) {
        q0[m] = q1[m] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (s_p[m0 + m] >= 0) {
          const float4* o = reinterpret_cast<const float4*>(O + (size_t)s_p[m0 + m] * h) + 2 * v;
          q0[m] = ld_l2(o);
          q1[m] = ld_l2(o + 1);
        }
      }
#pragma unroll
      for (int m = 0; m < kAhead; ++m) {
        if (s_p[m0 + m] < 0) continue;
        float a[8] = {q0[m].x, q0[m].y, q0[m].z, q0[m].w, q1[m].x, q1[m].y, q1[m].z, q1[m].w};
        for (int s = 1; s < ksplit; ++s) {
          const float4* o = reinterpret_cast<const float4*>(O + s * split_stride + (size_t)s_p[m0 + m] * h) + 2 * v;
          const float4 r0 = ld_l2(o), r1 = ld_l2(o + 1);
          a[0] += r0.x; a[1] += r0.y; a[2] += r0.z; a[3] += r0.w;
          a[4] += r1.x; a[5] += r1.y; a[6] += r1.z; a[7] += r1.w;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) z[q] = fmaf(s_w[m0 + m], a[q], z[q]);
      }
    }
    uint4 outv;
    outv.x = pack2(z[0], z[1]); outv.y = pack2(z[2], z[3]);
    outv.z = pack2(z[4], z[5]); outv.w = pack2(z[6], z[7]);
    reinterpret_cast<uint4*>(y + (size_t)t * h)[v] = outv;
  }
}

// --------------------------------------------------------------------------- co-selection

// counts[a][b] += 1 for every token whose top-2 is (a, b) (App. A.1).  Integer counts: block
// histograms in shared memory, then integer atomics, so the result is exact and order-free.
__global__ void __launch_bounds__(256)
coselection_kernel(const int32_t* __restrict__ idx, int T, int E, KeptIds kept,
                   int32_t* __restrict__ counts) {
  __shared__ int s_c[kMaxE * kMaxE];
  for (int i = threadIdx.x; i < kMaxE * kMaxE; i += blockDim.x) s_c[i] = 0;
  __syncthreads();
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < T; t += gridDim.x * blockDim.x)
    atomicAdd(&s_c[kept.id[idx[2 * t]] * kMaxE + kept.id[idx[2 * t + 1]]], 1);
  __syncthreads();
  for (int i = threadIdx.x; i < kMaxE * kMaxE; i += blockDim.x) {
    const int a = i / kMaxE, b = i % kMaxE;
    if (a < E && b < E && s_c[i]) atomicAdd(&counts[a * E + b], s_c[i]);
  }
}

// ------------------------------------------------------------------------- top-2 distance

// D_t = || E_e0(x_t) - E_e1(x_t) ||_2, the quantity App. A.2 observes to be concentrated.
__global__ void __launch_bounds__(256)
top2_distance_kernel(const float* O, int ksplit, size_t split_stride, const int32_t* pair_pos, int T,
                     int h, float* __restrict__ dist) {
  __shared__ float s_part[8];
  pdl_launch_dependents();
  pdl_wait();
  const int t = blockIdx.x;
  const int p0 = ld_l2(pair_pos + 2 * t), p1 = ld_l2(pair_pos + 2 * t + 1);
  float acc = 0.f;
  if (p1 >= 0) {
    for (int i = threadIdx.x; i < h; i += blockDim.x) {
      float a = 0.f, b = 0.f;
      for (int s = 0; s < ksplit; ++s) {
        a += ld_l2(O + s * split_stride + (size_t)p0 * h + i);
        b += ld_l2(O + s * split_stride + (size_t)p1 * h + i);
      }
      const float d = a - b;
      acc = fmaf(d, d, acc);
    }
  }
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, s);
  if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    float tot = 0.f;
    for (int w = 0; w < 8; ++w) tot += s_part[w];
    dist[t] = sqrtf(tot);
  }
}

// ------------------------------------------------------------------------------- rmsnorm

__global__ void __launch_bounds__(256)
rmsnorm_kernel(const bf16* x, int T, int h, float eps, bf16* out) {
  pdl_launch_dependents();
  pdl_wait();
  __shared__ float s_part[8];
  const int t = blockIdx.x;
  const int nvec = h >> 3;
  const uint4* xr = reinterpret_cast<const uint4*>(x + (size_t)t * h);
  float ss = 0.f;
  for (int v = threadIdx.x; v < nvec; v += blockDim.x) {
    float f[8];
    unpack8(ld_l2(xr + v), f);
#pragma unroll
    for (int k = 0; k < 8; ++k) ss = fmaf(f[k], f[k], ss);
  }
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, s);
  if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = ss;
  __syncthreads();
  float tot = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) tot += s_part[w];
  const float inv = 1.0f / sqrtf(tot / (float)h + eps);
  for (int v = threadIdx.x; v < nvec; v += blockDim.x) {
    float f[8];
    unpack8(ld_l2(xr + v), f);
    uint4 o;
    o.x = pack2(f[0] * inv, f[1] * inv); o.y = pack2(f[2] * inv, f[3] * inv);
    o.z = pack2(f[4] * inv, f[5] * inv); o.w = pack2(f[6] * inv, f[7] * inv);
    reinterpret_cast<uint4*>(out + (size_t)t * h)[v] = o;
  }
}

// ---------------------------------------------------------------------------- dense meta

__global__ void set_dense_meta_kernel(Meta* meta, int E, int rows, int off_stride) {
  if (threadIdx.x != 0) return;
  const int tiles = (rows + kTileRows - 1) / kTileRows;
  for (int c = 0; c <= kMaxE; ++c) {
    const int cc = c < E ? c : E;
    meta->off[c] = cc * off_stride;
    meta->tile_prefix[c] = cc * tiles;
    if (c < kMaxE) {
      meta->count[c] = c < E ? rows : 0;
      meta->count_slot[c][0] = meta->count[c];
      meta->count_slot[c][1] = 0;
    }
  }
  meta->n_skipped = 0;
  meta->n_touched = E;
  meta->reserved = 0;
}

// -------------------------------------------------------------------------------- select

__device__ __forceinline__ uint32_t float_key(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_float(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// Exact k0-th and k1-th smallest (0-based, k1 = k0 or k0 + 1).  The ratios lie in 0 .. 1, so one histogram
// of 2048 even bins leaves a handful of candidates around rank k0, which are ranked by counting.  Where more
// than kSelCand values share the bin (equal ratios, values outside 0 .. 1) the bit patterns are selected by
// radix: digits of 11, 11 and 10 bits, the counts of a digit in shared memory.  Then one more pass for the
// smallest key above the k0-th, if it is wanted and not among the candidates.  NV > 0: up to NV keys per thread
// stay in registers (NV * 1024 values); NV = 0: every pass reads the values again.  One block: bound by the
// latency of its passes (the first radix digit alone, few exponents and so few bins, serialised its additions).
constexpr int kSelThreads = 1024;
constexpr int kSelCand = 1024;
// monotone in the key
__device__ __forceinline__ int even_bin(uint32_t key) {
  if (key <= 0x80000000u) return 0;     // +0 and below
  if (key >= 0xbf800000u) return 2047;  // 1 and above
  return (int)(key_float(key) * 2048.f);
}
template <int NV>
__global__ void __launch_bounds__(kSelThreads)
select2_kernel(const float* v, int n, int k0, int k1, float* out) {
  pdl_wait();
  __shared__ unsigned hist[2048];
  __shared__ unsigned s_warp[32];
  __shared__ unsigned s_prefix, s_rank, s_count, s_next;
  __shared__ uint32_t s_cand[kSelCand];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint32_t keys[NV > 0 ? NV : 1];
  if (NV > 0) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int p = tid + i * kSelThreads;
      keys[i] = p < n ? float_key(ld_l2(v + p)) : 0u;
    }
  }
  auto each = [&](auto&& f) {
    if (NV > 0) {
#pragma unroll
      for (int i = 0; i < NV; ++i)
        if (tid + i * kSelThreads < n) f(keys[i]);
    } else {
      for (int p = tid; p < n; p += kSelThreads) f(float_key(ld_l2(v + p)));
    }
  };
  // counts in hist[] -> s_prefix = bin that holds rank `rank`, s_rank = rank inside it, s_count = values in it
  auto find_bin = [&](unsigned rank) {
    // exclusive sums over the bins, two bins a thread; the thread whose bin holds the rank says so
    const unsigned h0 = hist[2 * tid], h1 = hist[2 * tid + 1];
    unsigned inc = h0 + h1;
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
      const unsigned up = __shfl_up_sync(0xffffffffu, inc, s);
      if (lane >= s) inc += up;
    }
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    const unsigned before = __reduce_add_sync(0xffffffffu, lane < warp ? s_warp[lane] : 0u) + inc - h0 - h1;
    if (rank >= before && rank < before + h0 + h1) {
      const bool second = rank >= before + h0;
      s_prefix = (uint32_t)(2 * tid + (second ? 1 : 0));
      s_rank = rank - before - (second ? h0 : 0u);
      s_count = second ? h1 : h0;
    }
    __syncthreads();
  };
  auto clear_bins = [&]() {
    hist[2 * tid] = 0u;
    hist[2 * tid + 1] = 0u;
    __syncthreads();
  };
  clear_bins();
  each([&](uint32_t key) { atomicAdd(&hist[even_bin(key)], 1u); });
  __syncthreads();
  find_bin((unsigned)k0);
  const int bin = (int)s_prefix;
  unsigned rank = s_rank, count = s_count;
  uint32_t prefix = 0, next = 0;
  bool have_next = false;
  if (count <= kSelCand) {
    __syncthreads();  // everyone has read what find_bin left
    if (tid == 0) s_count = 0u;
    __syncthreads();
    each([&](uint32_t key) { if (even_bin(key) == bin) s_cand[atomicAdd(&s_count, 1u)] = key; });
    __syncthreads();
    if (tid < (int)count) {
      const uint32_t mine = s_cand[tid];
      unsigned less = 0, same = 0;
      for (unsigned i = 0; i < count; ++i) {
        less += s_cand[i] < mine;
        same += s_cand[i] == mine;
      }
      // equal keys write equal values
      if (less <= rank && rank < less + same) s_prefix = mine;
      if (less <= rank + 1 && rank + 1 < less + same) s_next = mine;
    }
    __syncthreads();
    prefix = s_prefix;
    have_next = rank + 1 < count;
    next = s_next;
  } else {
    uint32_t mask = 0;
    rank = (unsigned)k0;
#pragma unroll
    for (int pass = 0; pass < 3; ++pass) {
      const int shift = pass == 0 ? 21 : (pass == 1 ? 10 : 0);
      const uint32_t digit = pass == 2 ? 1023u : 2047u;
      clear_bins();
      each([&](uint32_t key) {
        if ((key & mask) == prefix) atomicAdd(&hist[(key >> shift) & digit], 1u);
      });
      __syncthreads();
      find_bin(rank);
      prefix |= s_prefix << shift;
      rank = s_rank;
      count = s_count;
      mask |= digit << shift;
    }
    have_next = rank + 1 < count;
    next = prefix;
  }
  if (k1 == k0) {
    next = prefix;
  } else if (!have_next) {  // the k0-th is the last of its value, or of its bin
    uint32_t best = 0xffffffffu;
    each([&](uint32_t key) { if (key > prefix) best = min(best, key); });
    best = __reduce_min_sync(0xffffffffu, best);
    if (lane == 0) s_warp[warp] = best;
    __syncthreads();
    next = __reduce_min_sync(0xffffffffu, s_warp[lane]);
  }
  if (tid == 0) {
    out[0] = key_float(prefix);
    out[1] = key_float(next);
  }
}

// ---------------------------------------------------------------------------- interleave

__global__ void __launch_bounds__(256)
interleave_kernel(const bf16* __restrict__ W1, const bf16* __restrict__ W3, KeptIds kept, int r,
                  int f, int h, bf16* __restrict__ W13) {
  const long long rows = (long long)r * 2 * f;
  const int lane = threadIdx.x & 31;
  const int nvec = h >> 3;
  for (long long row = (long long)blockIdx.x * 8 + (threadIdx.x >> 5); row < rows;
       row += (long long)gridDim.x * 8) {
    const int c = (int)(row / (2 * f));
    const int R = (int)(row % (2 * f));
    const int q = R / (2 * kInterleave), s = R % (2 * kInterleave);
    const bf16* src = (s < kInterleave)
        ? W1 + ((size_t)kept.id[c] * f + (size_t)q * kInterleave + s) * h
        : W3 + ((size_t)kept.id[c] * f + (size_t)q * kInterleave + s - kInterleave) * h;
    const uint4* sv = reinterpret_cast<const uint4*>(src);
    uint4* dv = reinterpret_cast<uint4*>(W13 + (size_t)row * h);
    for (int v = lane; v < nvec; v += 32) dv[v] = __ldg(sv + v);
  }
}

}  // namespace

// ------------------------------------------------------------------------------ launchers

// One block per SM at most; `work` blocks have something to do.
template <typename... KArgs, typename... Args>
static cudaError_t launch_route(void (*kernel)(KArgs...), int work, size_t smem, cudaStream_t st, Args&&... args) {
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRouteSmemMax);
    if (e != cudaSuccess) return e;
  }
  return launch_pdl(kernel, dim3(work < 148 ? work : 148), dim3(32 * kRouteWarps), smem, st, args...);
}

cudaError_t launch_router(const bf16* x, const bf16* Wg, int T, int h, int r, float beta,
                          const KeptIds& kept, const RouteOut& out, cudaStream_t st, bool w_const) {
#define MOE_ROUTER(R)                                                                                          \
  {                                                                                                            \
    const int part = route_part<R>(h, r);                                                                             \
    const bool whole = part == (h >> 3);                                                                       \
    const size_t smem = RouteCfg<R>::kRingBytes + (size_t)(whole ? 1 : 2) * r * part * 16;                     \
    const int units = (T + kRouteTokPerBlock - 1) / kRouteTokPerBlock;                                         \
    return launch_route(whole ? router_kernel<R, true> : router_kernel<R, false>, units, smem, st, x, Wg, T, h, \
                        r, part, beta, kept, out, w_const);                                                    \
  }
  switch (r) {
    case 2: MOE_ROUTER(2)
    case 3: case 4: MOE_ROUTER(4)
    case 5: case 6: MOE_ROUTER(6)
    case 7: case 8: MOE_ROUTER(8)
    default: MOE_ROUTER(kMaxE)
  }
#undef MOE_ROUTER
}

// One block per SM at most.  Up to 8 tokens per SM: a tile of 8 for the whole block, the shortest way to one
// tile's end.  Then, up to two tiles of 16 per block, the whole block again; beyond, and for narrow rows that
// leave 16 warps little to share, four teams, which run out of step and so keep more loads in flight.  Router
// rows that do not fit shared memory are read once per tile and warp: the whole block shares them.  Calibration
// in us, one team / four teams, 2000, 4096, 8192, 16384 tokens: h 4096, 8 experts 20.4 / 23.2, 24.6 / 24.8, 31.1 / 27.9,
// 56.4 / 50.8, 16 experts 23.3 / 27.1, 28.0 / 29.0, 36.4 / 32.1; h 2048 19.4 / 20.7, 22.0 / 21.0, 27.0 / 23.7, 36.9 / 30.8;
// h 1024 18.7 / 18.5, 21.2 / 19.0, 24.8 / 21.3; top-k call on h 128, 8192 tokens 79.2 / 72.5.
constexpr int kRouteShort = 148 * 8;
inline bool route_in_teams(int T, int h, bool whole) { return whole && (h < 2048 || T > 2 * 148 * 16); }
template <typename... KArgs, typename... Args>
static cudaError_t launch_tiles(void (*kernel)(KArgs...), int tiles, size_t smem, cudaStream_t st, Args&&... args) {
  if (smem > 32 * 1024) {  // with the records (static) possibly more than the default limit of 48 KB
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTileSmemMax);
    if (e != cudaSuccess) return e;
  }
  return launch_pdl(kernel, dim3(tiles < 148 ? tiles : 148), dim3(32 * kRouteWarps), smem, st, args...);
}

#define MOE_TILES_LAUNCH(kernel, R, NT, TW, whole, ...)                                                       \
  return launch_tiles(kernel<R, NT, TW, whole>, (T + 8 * NT - 1) / (8 * NT),                                  \
                      TileCfg<R, NT, TW>::kPartBytes + (whole ? TileCfg<R, NT, TW>::w_bytes(h) : 0), st, x, Wg, T, h, r, \
                      __VA_ARGS__)
#define MOE_TILES_R(kernel, R, ...)                                                                           \
  {                                                                                                           \
    const bool whole = TileCfg<R, 2, 4>::kPartBytes + TileCfg<R, 2, 4>::w_bytes(h) <= kTileSmemMax;         \
    if (route_in_teams(T, h, whole) && T > kRouteShort) MOE_TILES_LAUNCH(kernel, R, 2, 4, true, __VA_ARGS__); \
    if (T > kRouteShort && whole) MOE_TILES_LAUNCH(kernel, R, 2, kRouteWarps, true, __VA_ARGS__);             \
    if (T > kRouteShort) MOE_TILES_LAUNCH(kernel, R, 2, kRouteWarps, false, __VA_ARGS__);                     \
    if (whole) MOE_TILES_LAUNCH(kernel, R, 1, kRouteWarps, true, __VA_ARGS__);                                \
    MOE_TILES_LAUNCH(kernel, R, 1, kRouteWarps, false, __VA_ARGS__);                                          \
  }
// (with fewer than 8 experts the tensor core computes 8 columns all the same)
#define MOE_TILES_SWITCH(kernel, ...)                                                                         \
  if (r <= 8) MOE_TILES_R(kernel, 8, __VA_ARGS__)                                                             \
  MOE_TILES_R(kernel, kMaxE, __VA_ARGS__)

cudaError_t launch_ratios(const bf16* x, const bf16* Wg, int T, int h, int r, float* ratio, cudaStream_t st,
                          bool w_const) {
  MOE_TILES_SWITCH(ratio_kernel, ratio, w_const)
}

cudaError_t launch_router_small(const bf16* x, const bf16* Wg, int T, int h, int r, float beta,
                                const KeptIds& kept, const RouteOut& out, cudaStream_t st) {
  switch (r) {
    case 2: return launch_pdl(router_small_kernel<2>, dim3(T), dim3(256), 0, st, x, Wg, T, h, r, beta, kept, out);
    case 3: case 4: return launch_pdl(router_small_kernel<4>, dim3(T), dim3(256), 0, st, x, Wg, T, h, r, beta, kept, out);
    case 5: case 6: return launch_pdl(router_small_kernel<6>, dim3(T), dim3(256), 0, st, x, Wg, T, h, r, beta, kept, out);
    case 7: case 8: return launch_pdl(router_small_kernel<8>, dim3(T), dim3(256), 0, st, x, Wg, T, h, r, beta, kept, out);
    default: return launch_pdl(router_small_kernel<kMaxE>, dim3(T), dim3(256), 0, st, x, Wg, T, h, r, beta, kept, out);
  }
  return cudaGetLastError();
}

cudaError_t launch_route_single(const bf16* x, const bf16* Wg, int h, int r, float beta,
                                const KeptIds& kept, const RouteOut& out, int pad, Meta* meta,
                                int32_t* pair_pos, bf16* xperm, int32_t* s_count,
                                int32_t* s_nskipped, int32_t* s_ntouched, int E, cudaStream_t st) {
#define MOE_ROUTE_SINGLE(R)                                                                        \
  return launch_pdl(route_single_kernel<R>, dim3(1), dim3(256), 0, st, x, Wg, h, r, beta, kept, out, \
                    pad, meta, pair_pos, xperm, s_count, s_nskipped, s_ntouched, E)
  switch (r) {
    case 2: MOE_ROUTE_SINGLE(2);
    case 3: case 4: MOE_ROUTE_SINGLE(4);
    case 5: case 6: MOE_ROUTE_SINGLE(6);
    case 7: case 8: MOE_ROUTE_SINGLE(8);
    default: MOE_ROUTE_SINGLE(kMaxE);
  }
#undef MOE_ROUTE_SINGLE
}

cudaError_t launch_permute_gather_small(const bf16* x, const int32_t* idx, const uint8_t* skipped, int T,
                                        int h, int r, int pad, Meta* meta, int32_t* pair_pos,
                                        bf16* xperm, int32_t* s_count,
                                        int32_t* s_nskipped, int32_t* s_ntouched, const KeptIds& kept,
                                        int E, cudaStream_t st) {
  return launch_pdl(permute_gather_small_kernel, dim3(T), dim3(kDecodeMaxT), 0, st, x, idx, skipped, T, h,
                    r, pad, meta, pair_pos, xperm, s_count, s_nskipped, s_ntouched, kept, E);
}

cudaError_t launch_scan(const int32_t* blk_hist, int nblk, int r, int pad, int32_t* blk_base,
                        Meta* meta, int32_t* s_count, int32_t* s_nskipped, int32_t* s_ntouched,
                        const KeptIds& kept, int E, cudaStream_t st) {
  return launch_pdl(scan_kernel, dim3(1), dim3(1024), 0, st, blk_hist, nblk, r, pad, blk_base, meta,
                    s_count, s_nskipped, s_ntouched, kept, E);
}

cudaError_t launch_permute(const bf16* x, const int32_t* idx, const void* active, bool top2, int T, int k, int h,
                           int r, int pad, const int32_t* blk_base, Meta* meta, int32_t* pair_pos, bf16* xperm,
                           int32_t* s_count, int32_t* s_nskipped, int32_t* s_ntouched, const KeptIds& kept,
                           int E, cudaStream_t st) {
  const int units = (T + kRouteTokPerBlock - 1) / kRouteTokPerBlock;
  // column shares: enough blocks to keep every SM copying, at least 64 vectors each
  int ny = 148 * 4 / units, most = (h >> 3) / 64;
  if (ny > most) ny = most;
  if (ny < 1) ny = 1;
  return launch_pdl(top2 ? permute_kernel<true> : permute_kernel<false>, dim3(units, ny), dim3(256), 0, st, x, idx,
                    active, T, k, h, r, pad, blk_base, meta, pair_pos, xperm, s_count, s_nskipped, s_ntouched,
                    kept, E);
}

cudaError_t launch_combine(const float* O, int ksplit, size_t split_stride, const int32_t* pair_pos,
                           const float* wn, const bf16* residual, int T, int h, bf16* y,
                           cudaStream_t st, int col0, int cols) {
  const int v0 = col0 >> 3, v1 = cols ? v0 + (cols >> 3) : h >> 3;
  int ychunks = (v1 - v0 + 127) / 128;
  if (T > 4096) ychunks = 1;  // plenty of blocks already
  return launch_pdl(combine_kernel, dim3(T, ychunks), dim3(128), 0, st, O, ksplit, split_stride,
                    pair_pos, wn, residual, T, h, v0, v1, y);
}

cudaError_t launch_router_topk(const bf16* x, const bf16* Wg, int T, int h, int r, int k, float beta,
                               const KeptIds& kept, int32_t* idx, float* wn, int32_t* nact,
                               int32_t* u_idx, float* u_wn, int32_t* u_nact, float* logits,
                               cudaStream_t st) {
  MOE_TILES_SWITCH(router_topk_kernel, k, beta, kept, idx, wn, nact, u_idx, u_wn, u_nact, logits)
}

cudaError_t launch_count_topk(const int32_t* idx, const int32_t* nact, int T, int k,
                              int32_t* blk_hist, cudaStream_t st) {
  const int nblk = (T + kRouteTokPerBlock - 1) / kRouteTokPerBlock;
  count_topk_kernel<<<nblk, kHistCols < 64 ? 64 : kHistCols, 0, st>>>(idx, nact, T, k, blk_hist);
  return cudaGetLastError();
}

cudaError_t launch_combine_topk(const float* O, int ksplit, size_t split_stride,
                                const int32_t* pair_pos, const float* wn, int k, int T, int h,
                                bf16* y, cudaStream_t st) {
  int ychunks = ((h >> 3) + 127) / 128;
  if (T > 4096) ychunks = 1;
  return launch_pdl(combine_topk_kernel, dim3(T, ychunks), dim3(128), 0, st, O, ksplit, split_stride, pair_pos,
                    wn, k, T, h, y);
}

cudaError_t launch_coselection(const int32_t* idx, int T, int E, const KeptIds& kept, int32_t* counts,
                               cudaStream_t st) {
  int blocks = (T + 255) / 256;
  if (blocks > 148 * 4) blocks = 148 * 4;
  coselection_kernel<<<blocks, 256, 0, st>>>(idx, T, E, kept, counts);
  return cudaGetLastError();
}

cudaError_t launch_top2_distance(const float* O, int ksplit, size_t split_stride,
                                 const int32_t* pair_pos, int T, int h, float* dist, cudaStream_t st) {
  return launch_pdl(top2_distance_kernel, dim3(T), dim3(256), 0, st, O, ksplit, split_stride, pair_pos,
                    T, h, dist);
}

cudaError_t launch_rmsnorm(const bf16* x, int T, int h, float eps, bf16* out, cudaStream_t st) {
  return launch_pdl(rmsnorm_kernel, dim3(T), dim3(256), 0, st, x, T, h, eps, out);
}

cudaError_t launch_set_dense_meta(Meta* meta, int E, int rows_per_expert, int off_stride,
                                  cudaStream_t st) {
  set_dense_meta_kernel<<<1, 32, 0, st>>>(meta, E, rows_per_expert, off_stride);
  return cudaGetLastError();
}

cudaError_t launch_select2(const float* ratio, int T, int k0, int k1, float* out, cudaStream_t st) {
  if (T <= 8 * kSelThreads) return launch_pdl(select2_kernel<8>, dim3(1), dim3(kSelThreads), 0, st, ratio, T, k0, k1, out);
  if (T <= 16 * kSelThreads) return launch_pdl(select2_kernel<16>, dim3(1), dim3(kSelThreads), 0, st, ratio, T, k0, k1, out);
  if (T <= 32 * kSelThreads) return launch_pdl(select2_kernel<32>, dim3(1), dim3(kSelThreads), 0, st, ratio, T, k0, k1, out);
  return launch_pdl(select2_kernel<0>, dim3(1), dim3(kSelThreads), 0, st, ratio, T, k0, k1, out);
}

// Under lazy module loading a kernel's code comes onto the device, and takes device memory, when it is first
// launched or asked about: asks about every kernel that a calibration of up to 16384 tokens can run.
template <int R> static cudaError_t load_routers(cudaError_t e) {
  cudaFuncAttributes a;
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, router_kernel<R, true>);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, router_kernel<R, false>);
  return e;
}
template <int R> static cudaError_t load_ratios(cudaError_t e) {  // the forms of MOE_TILES_R
  cudaFuncAttributes a;
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, ratio_kernel<R, 2, 4, true>);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, ratio_kernel<R, 2, kRouteWarps, true>);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, ratio_kernel<R, 2, kRouteWarps, false>);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, ratio_kernel<R, 1, kRouteWarps, true>);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, ratio_kernel<R, 1, kRouteWarps, false>);
  return e;
}
cudaError_t load_calibration_kernels() {
  cudaError_t e = load_ratios<kMaxE>(load_ratios<8>(cudaSuccess));
  e = load_routers<2>(load_routers<4>(load_routers<6>(load_routers<8>(load_routers<kMaxE>(e)))));
  cudaFuncAttributes a;
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, select2_kernel<8>);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, select2_kernel<16>);
  return e;
}

cudaError_t launch_interleave(const bf16* W1, const bf16* W3, const KeptIds& kept, int r, int f,
                              int h, bf16* W13, cudaStream_t st) {
  interleave_kernel<<<148 * 8, 256, 0, st>>>(W1, W3, kept, r, f, h, W13);
  return cudaGetLastError();
}

}  // namespace moe
