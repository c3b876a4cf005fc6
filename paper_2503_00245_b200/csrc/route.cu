// Router (logits + softmax + top-k + gate weights), token->expert grouping, row gather,
// gate-weighted combine and the one-off weight packing kernels.
#include <algorithm>

#include "common.cuh"

namespace cosmoe {

// ------------------------------------------------------------------------------------ router
// Threads split the d axis and keep E partial logits each; shuffle trees finish them; one warp then
// does the E-wide softmax and the top-k with one or two experts per lane (E <= 64).
// Selection runs on the logits: softmax is monotonic, so top_k(W) = top_k(R) (Eq. 2, Eq. 3), and
// the logits carry more bits than the fp32 probabilities.  Ties go to the lower expert index.
template <typename XT>
__device__ __forceinline__ void load_x8(const XT* p, float* f);
template <>
__device__ __forceinline__ void load_x8<float>(const float* p, float* f) {
  const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
  f[0] = a.x, f[1] = a.y, f[2] = a.z, f[3] = a.w, f[4] = b.x, f[5] = b.y, f[6] = b.z, f[7] = b.w;
}
template <>
__device__ __forceinline__ void load_x8<__nv_bfloat16>(const __nv_bfloat16* p, float* f) {
  unpack8(*reinterpret_cast<const uint4*>(p), f);
}

constexpr int kRouteWarps = 8;

// Partial logits of one token over the chunks [c_begin, c_end) step c_step of the d axis.  The token's
// chunks are fetched eight at a time before any arithmetic, so a warp pays one memory round trip per group.
template <typename XT, int EMAX>
__device__ __forceinline__ void route_partial(const XT* __restrict__ xr, const uint16_t* __restrict__ w_router, int E,
                                              int c_begin, int c_end, int c_step, float* acc) {
  const bool vec = (E % 8) == 0;
  for (int cb = c_begin; cb < c_end; cb += 8 * c_step) {
    float xv[8][8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int c = cb + u * c_step;
      if (c < c_end) {
        load_x8<XT>(xr + c * 8, xv[u]);
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) xv[u][i] = 0.f;
      }
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int c = min(cb + u * c_step, c_end - 1);  // clamped rows meet zero inputs
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const uint16_t* wr = w_router + (size_t)(c * 8 + i) * E;
        if (vec) {
#pragma unroll
          for (int e8 = 0; e8 < EMAX / 8; ++e8) {
            if (e8 * 8 < E) {
              float wv[8];
              unpack8(__ldg(reinterpret_cast<const uint4*>(wr) + e8), wv);
#pragma unroll
              for (int j = 0; j < 8; ++j) acc[e8 * 8 + j] = fmaf(xv[u][i], wv[j], acc[e8 * 8 + j]);
            }
          }
        } else {
#pragma unroll
          for (int e = 0; e < EMAX; ++e)
            if (e < E) acc[e] = fmaf(xv[u][i], bf16_to_float(__ldg(wr + e)), acc[e]);
        }
      }
    }
  }
}

// Many tokens: one warp per token, lanes split the d axis.
template <typename XT, int EMAX>
__global__ void __launch_bounds__(kRouteWarps * 32)
    route_kernel(const XT* __restrict__ x, const uint16_t* __restrict__ w_router, const float* __restrict__ bias, int T,
                 int d, int E, int k, int renorm, int32_t* __restrict__ topk_idx, float* __restrict__ topk_w,
                 float* __restrict__ probs) {
  __shared__ float s_logit[kRouteWarps][EMAX];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int t = blockIdx.x * kRouteWarps + wib;
  pdl_launch_dependents();
  pdl_wait();
  if (t >= T) return;
  float acc[EMAX];
#pragma unroll
  for (int e = 0; e < EMAX; ++e) acc[e] = 0.f;
  route_partial<XT, EMAX>(x + (size_t)t * d, w_router, E, lane, d / 8, 32, acc);
#pragma unroll
  for (int e = 0; e < EMAX; ++e)
    if (e < E) acc[e] = warp_sum(acc[e]);
  if (lane == 0) {
#pragma unroll
    for (int e = 0; e < EMAX; ++e)
      if (e < E) s_logit[wib][e] = acc[e];
  }
  __syncwarp();
  const float l0 = lane < E ? s_logit[wib][lane] + (bias ? bias[lane] : 0.f) : 0.f;
  const float l1 = lane + 32 < E ? s_logit[wib][lane + 32] + (bias ? bias[lane + 32] : 0.f) : 0.f;
  warp_route_finish(l0, l1, E, k, renorm, lane, topk_idx + (size_t)t * k, topk_w + (size_t)t * k,
                    probs ? probs + (size_t)t * E : nullptr);
}

// Many tokens: the logits of 16 tokens per CTA on the tensor cores (mma.sync m16n8k8: 16 tokens x 8 experts; N is far
// below a tcgen05 tile).  W_r lies transposed in shared memory, [expert][feature], the experts' rows 64 bytes beyond a
// multiple of 128 apart; the 16 warps split the features in units of 32.  A lane takes 8 consecutive features of a row at a
// time, of x straight from memory (all of a warp's loads of a round in flight together) and of W_r alike: the order of
// the contraction inside a unit is free.  fp32 rows go in as three bf16 terms.  An MMA cuts its sums instead of rounding them:
// eight products in one (m16n8k8), everything else is added in fp32, in pairs.  Relative error of the probabilities against 64
// bits, 512 bf16 tokens at d 1024: 7.9e-8, as with fp32 multiply-adds (64 products in one accumulator: 10.2e-8).
// The last CTA to finish groups the pairs by expert, a stable counting sort: every warp counts and then scatters a
// contiguous run of them.  One launch instead of two, and no second walk over the routing by a lone CTA in rounds.
// Bound by latency: one round trip to x, then a CTA's chain of barriers.  Under ncu, cold, 2048 tokens at d 2048: 12.5 us for 8
// experts where the staged router and the grouping took 11.4 + 7.4; other expert counts had a router that read W_r through L1
// a value at a time: a whole layer of 272 tokens, 16 experts at d 344 51.2 -> 36.6 us, 107 tokens, 2 experts at d 352 38.9 -> 27.8.
constexpr int kRtWarps = 16, kRtTokens = 16, kRtUnit = 32, kRtBatch = 4;
struct RtShape {
  int e8, row_bytes, part_off, smem;  // experts rounded up to 8; bytes between two experts' rows; partial logits; total
};
static __host__ __device__ inline RtShape rt_shape(int d, int E) {
  RtShape r{};
  r.e8 = (E + 7) / 8 * 8;
  r.row_bytes = (d + kRtUnit - 1) / kRtUnit * kRtUnit * 2;
  r.row_bytes += (r.row_bytes & 127) == 64 ? 0 : 64;
  r.part_off = r.e8 * r.row_bytes;
  const int part = kRtWarps * kRtTokens * r.e8 * 4, count = kRtWarps * MOE_MAX_EXPERTS * 4;
  r.smem = r.part_off + (part > count ? part : count);
  return r;
}

template <typename XT>
__global__ void __launch_bounds__(kRtWarps * 32)
    route_tile_kernel(const XT* __restrict__ x, const uint16_t* __restrict__ w_router, const float* __restrict__ bias, int T,
                      int d, int E, int k, int renorm, int32_t* topk_idx, float* __restrict__ topk_w,
                      float* __restrict__ probs, Grouping grp, Scatter sc, DeviceState* st) {
  constexpr int NT = sizeof(XT) == 4 ? 3 : 1;  // bf16 terms of a value
  extern __shared__ __align__(128) unsigned char rt_smem[];
  const RtShape sh = rt_shape(d, E);
  float* const part = reinterpret_cast<float*>(rt_smem + sh.part_off);  // [warp][token][expert]
  __shared__ int s_last, s_base[MOE_MAX_EXPERTS + 1], s_count[MOE_MAX_EXPERTS];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_launch_dependents();
  if (tid < MOE_MAX_EXPERTS) s_count[tid] = 0;
  const int units = (d + kRtUnit - 1) / kRtUnit;
  for (uint32_t i = tid * 128u, n = (uint32_t)d * E * 2u; i < n; i += kRtWarps * 32 * 128u)  // (W_r: its lines into L2 ...)
    asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const unsigned char*>(w_router) + i));
  pdl_wait();  // (... its values, like x, may come from the kernel before)
  const int t0 = blockIdx.x * kRtTokens, g = lane >> 2, q = lane & 3;
  const XT* const row0 = x + (size_t)min(t0 + g, T - 1) * d;
  const XT* const row1 = x + (size_t)min(t0 + g + 8, T - 1) * d;
  uint4 a[kRtBatch][2][NT];
  auto fetch = [&](int u0) {
#pragma unroll
    for (int j = 0; j < kRtBatch; ++j)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = (u0 + j * kRtWarps) * kRtUnit + q * 8;
        const bool in = c < d;  // (what lies past the row: zeros, in place of its first eight values)
        const XT* src = (h ? row1 : row0) + (in ? c : 0);
        if constexpr (NT == 1) {
          a[j][h][0] = ldcg_now(reinterpret_cast<const uint4*>(src));
          if (!in) a[j][h][0] = make_uint4(0u, 0u, 0u, 0u);
        } else {
          float f[8];
          load_x8<XT>(src, f);
          uint16_t tm[8][3];
#pragma unroll
          for (int i = 0; i < 8; ++i) split3(in ? f[i] : 0.f, tm[i]);
#pragma unroll
          for (int t = 0; t < NT; ++t)
            a[j][h][t] = make_uint4(tm[0][t] | (uint32_t)tm[1][t] << 16, tm[2][t] | (uint32_t)tm[3][t] << 16,
                                    tm[4][t] | (uint32_t)tm[5][t] << 16, tm[6][t] | (uint32_t)tm[7][t] << 16);
        }
      }
  };
  if (NT == 1) fetch(warp);  // on its way while W_r is laid out (fp32 rows: no registers for that)
  constexpr int kRowsFly = 4;  // rows of W_r a thread has on their way at a time (d <= 2048: one round trip)
  for (int e8 = 0; e8 < sh.e8; e8 += 8)
    for (int r0 = tid; r0 < units * kRtUnit; r0 += kRowsFly * kRtWarps * 32) {
      uint16_t v[kRowsFly][8];
#pragma unroll
      for (int u = 0; u < kRowsFly; ++u) {
        const int r = r0 + u * kRtWarps * 32;
        if ((E & 7) == 0) {
          const uint4 w = ldcg_now(reinterpret_cast<const uint4*>(w_router + (size_t)min(r, d - 1) * E + e8));
          *reinterpret_cast<uint4*>(v[u]) = r < d ? w : make_uint4(0u, 0u, 0u, 0u);
        } else {
#pragma unroll
          for (int e = 0; e < 8; ++e) v[u][e] = r < d && e8 + e < E ? __ldcg(w_router + (size_t)r * E + e8 + e) : (uint16_t)0;
        }
      }
#pragma unroll
      for (int u = 0; u < kRowsFly; ++u) {
        const int r = r0 + u * kRtWarps * 32;
        if (r >= units * kRtUnit) break;
#pragma unroll
        for (int e = 0; e < 8; ++e) *reinterpret_cast<uint16_t*>(rt_smem + (e8 + e) * sh.row_bytes + r * 2) = v[u][e];
      }
    }
  __syncthreads();
  float* const mine = part + (warp * kRtTokens + g) * sh.e8 + 2 * q;
  for (int u0 = warp; u0 < units || u0 == warp; u0 += kRtWarps * kRtBatch) {
    if (NT != 1 || u0 != warp) fetch(u0);
    for (int e8 = 0; e8 < sh.e8; e8 += 8) {
      const unsigned char* wrow = rt_smem + (e8 + g) * sh.row_bytes + q * 16;
      float sum[4];
#pragma unroll
      for (int j0 = 0; j0 < kRtBatch; j0 += 2) {
        float m[8][4];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const uint4 b = *reinterpret_cast<const uint4*>(wrow + min(u0 + (j0 + j) * kRtWarps, units - 1) * (kRtUnit * 2));
          const uint4(&r)[2][NT] = a[j0 + j];
#pragma unroll
          for (int i = 0; i < 4; ++i) m[4 * j + i][0] = m[4 * j + i][1] = m[4 * j + i][2] = m[4 * j + i][3] = 0.f;
#pragma unroll
          for (int t = NT - 1; t >= 0; --t) {  // (what the small terms' sums lose is far below the first one's last place)
            mma8(m[4 * j], r[0][t].x, r[1][t].x, b.x), mma8(m[4 * j + 1], r[0][t].y, r[1][t].y, b.y);
            mma8(m[4 * j + 2], r[0][t].z, r[1][t].z, b.z), mma8(m[4 * j + 3], r[0][t].w, r[1][t].w, b.w);
          }
        }
#pragma unroll
        for (int n = 4; n > 0; n >>= 1)
#pragma unroll
          for (int j = 0; j < n; ++j) add4(m[j], m[j + n]);
#pragma unroll
        for (int i = 0; i < 4; ++i) sum[i] = j0 == 0 ? m[0][i] : sum[i] + m[0][i];
      }
      float* dst = mine + e8;  // D: tokens g and g + 8, experts 2q and 2q + 1
      if (u0 == warp) {
        dst[0] = sum[0], dst[1] = sum[1], dst[8 * sh.e8] = sum[2], dst[8 * sh.e8 + 1] = sum[3];
      } else {
        dst[0] += sum[0], dst[1] += sum[1], dst[8 * sh.e8] += sum[2], dst[8 * sh.e8 + 1] += sum[3];
      }
    }
  }
  __syncthreads();
  int my_e = 0, my_pos = 0;  // (lane j: the token's j-th choice)
  {
    const int t = t0 + warp;  // a warp finishes one token
    if (t < T) {
      float l0 = 0.f, l1 = 0.f;
      auto logit = [&](int e) {  // the warps' shares, in pairs
        const float* p = part + warp * sh.e8 + e;
        const int step = kRtTokens * sh.e8;
        float v[kRtWarps];
#pragma unroll
        for (int w = 0; w < kRtWarps; ++w) v[w] = p[w * step];
#pragma unroll
        for (int n = kRtWarps / 2; n > 0; n >>= 1)
#pragma unroll
          for (int w = 0; w < n; ++w) v[w] += v[w + n];
        return bias ? v[0] + bias[e] : v[0];
      };
      if (lane < E) l0 = logit(lane);
      if (lane + 32 < E) l1 = logit(lane + 32);
      int e;
      float wt;
      unsigned long long selected;
      warp_route_top(l0, l1, E, k, renorm, lane, probs ? probs + (size_t)t * E : nullptr, e, wt, selected);
      if (lane < k) {
        topk_idx[(size_t)t * k + lane] = e, topk_w[(size_t)t * k + lane] = wt;
        if (sc.rows) my_e = e, my_pos = atomicAdd(&s_count[e], 1);
      }
    }
  }
  if (sc.rows) {
    // ---- the CTA takes places for its tokens and copies their rows there
    const int t = min(t0 + warp, T - 1), chunks = d / 8;
    const XT* const row = x + (size_t)t * d;
    constexpr int kFly = sizeof(XT) == 4 ? 4 : 8;
    float f[kFly][8];
    auto get = [&](int c0) {
#pragma unroll
      for (int u = 0; u < kFly; ++u)
        if (c0 + 32 * u < chunks) load_x8<XT>(row + (c0 + 32 * u) * 8, f[u]);
    };
    get(lane);
    __syncthreads();
    if (tid < E && s_count[tid] > 0) s_base[tid] = (int)atomicAdd(&st->route_count[tid], (unsigned)s_count[tid]);
    __syncthreads();
    if (t0 + warp >= T) return;
    if (lane < k) {
      my_pos += s_base[my_e];
      sc.pos[(size_t)t * k + lane] = my_pos;
    }
    for (int c0 = lane; __any_sync(0xffffffffu, c0 < chunks); c0 += 32 * kFly) {
      if (c0 != lane) get(c0);
      for (int j = 0; j < k; ++j) {
        const size_t r = (size_t)__shfl_sync(0xffffffffu, my_e, j) * T + __shfl_sync(0xffffffffu, my_pos, j);
        uint4* const dst = reinterpret_cast<uint4*>(sc.rows) + r * chunks;
#pragma unroll
        for (int u = 0; u < kFly; ++u)
          if (c0 + 32 * u < chunks)
            dst[c0 + 32 * u] = make_uint4(pack_bf16x2(f[u][0], f[u][1]), pack_bf16x2(f[u][2], f[u][3]), pack_bf16x2(f[u][4], f[u][5]),
                                          pack_bf16x2(f[u][6], f[u][7]));
      }
    }
    return;
  }
  if (!grp.perm) return;
  // ---- the last CTA groups the pairs
  __syncthreads();
  if (tid == 0) {
    // (release: the CTA's routing, ordered before this thread by the barrier; acquire: the other CTAs')
    const unsigned old = atom_add_acq_rel(&st->route_done, 1u);
    s_last = old == gridDim.x - 1u;
    if (s_last) st->route_done = 0u;
  }
  __syncthreads();
  if (!s_last) return;
  int* const count = reinterpret_cast<int*>(part);  // [warp][expert]
  for (int i = tid; i < kRtWarps * MOE_MAX_EXPERTS; i += kRtWarps * 32) count[i] = 0;
  __syncthreads();
  const int n = T * k, per = (n + kRtWarps * 32 - 1) / (kRtWarps * 32) * 32;
  const int lo = warp * per, hi = min(n, lo + per);
  int* const wc = count + warp * MOE_MAX_EXPERTS;
  const unsigned below = (1u << lane) - 1u;
  constexpr int kKeep = 8;  // pairs per lane kept in registers between the two walks
  int keep[kKeep];
#pragma unroll
  for (int i = 0; i < kKeep; ++i) {
    const int p = lo + i * 32 + lane;
    keep[i] = p < hi ? __ldcg(topk_idx + p) : -1;
  }
  auto each = [&](auto&& body) {
#pragma unroll
    for (int i = 0; i < kKeep; ++i)
      if (lo + i * 32 < hi) body(lo + i * 32 + lane, keep[i]);
    for (int p0 = lo + kKeep * 32; p0 < hi; p0 += 32) body(p0 + lane, p0 + lane < hi ? __ldcg(topk_idx + p0 + lane) : -1);
  };
  each([&](int, int e) {
    const unsigned peers = __match_any_sync(0xffffffffu, e);
    if (e >= 0 && (peers & below) == 0u) wc[e] += __popc(peers);
    __syncwarp();
  });
  __syncthreads();
  if (tid < MOE_MAX_EXPERTS) {
    int run = 0;
    for (int w = 0; w < kRtWarps; ++w) {
      const int c = count[w * MOE_MAX_EXPERTS + tid];
      count[w * MOE_MAX_EXPERTS + tid] = run;  // within the expert: where the warp's pairs start
      run += c;
    }
    s_base[tid] = run;
  }
  __syncthreads();
  if (warp == 0) {
    const int c0 = s_base[lane], c1 = s_base[lane + 32];
    int a0 = c0, a1 = c1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v0 = __shfl_up_sync(0xffffffffu, a0, o), v1 = __shfl_up_sync(0xffffffffu, a1, o);
      if (lane >= o) a0 += v0, a1 += v1;
    }
    const int tot0 = __shfl_sync(0xffffffffu, a0, 31);
    __syncwarp();
    s_base[lane] = a0 - c0, s_base[lane + 32] = tot0 + a1 - c1;
    if (lane < E) grp.offsets[lane] = a0 - c0;
    if (lane + 32 < E) grp.offsets[lane + 32] = tot0 + a1 - c1;
    if (lane == 0) grp.offsets[E] = n;
  }
  __syncthreads();
  each([&](int p, int e) {
    const unsigned peers = __match_any_sync(0xffffffffu, e);
    const int base = e >= 0 ? s_base[e] + wc[e] : 0;
    __syncwarp();
    if (e >= 0) {
      const int slot = base + __popc(peers & below);
      grp.perm[slot] = p;
      grp.inv[p] = slot;
      if ((peers & below) == 0u) wc[e] += __popc(peers);
    }
    __syncwarp();
  });
}

// Few tokens (decode): one CTA per token, all 256 threads split the d axis so the weight rows are
// fetched in a single round trip; warp 0 finishes.
template <typename XT, int EMAX>
__global__ void __launch_bounds__(kRouteWarps * 32)
    route_block_kernel(const XT* __restrict__ x, const uint16_t* __restrict__ w_router, const float* __restrict__ bias,
                       int T, int d, int E, int k, int renorm, int32_t* __restrict__ topk_idx,
                       float* __restrict__ topk_w, float* __restrict__ probs) {
  __shared__ float s_part[kRouteWarps][EMAX];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  pdl_launch_dependents();
  pdl_wait();
  const int t = blockIdx.x;
  float acc[EMAX];
#pragma unroll
  for (int e = 0; e < EMAX; ++e) acc[e] = 0.f;
  route_partial<XT, EMAX>(x + (size_t)t * d, w_router, E, threadIdx.x, d / 8, kRouteWarps * 32, acc);
#pragma unroll
  for (int e = 0; e < EMAX; ++e)
    if (e < E) acc[e] = warp_sum(acc[e]);
  if (lane == 0) {
#pragma unroll
    for (int e = 0; e < EMAX; ++e)
      if (e < E) s_part[wib][e] = acc[e];
  }
  __syncthreads();
  if (wib != 0) return;
  float l0 = 0.f, l1 = 0.f;
  if (lane < E) {
    for (int w = 0; w < kRouteWarps; ++w) l0 += s_part[w][lane];
    if (bias) l0 += bias[lane];
  }
  if (lane + 32 < E) {
    for (int w = 0; w < kRouteWarps; ++w) l1 += s_part[w][lane + 32];
    if (bias) l1 += bias[lane + 32];
  }
  warp_route_finish(l0, l1, E, k, renorm, lane, topk_idx + (size_t)t * k, topk_w + (size_t)t * k,
                    probs ? probs + (size_t)t * E : nullptr);
}

// more than a decode step's tokens (16 would be a tile of a single CTA: those take a CTA per token), and W_r fits into shared
// memory (two CTAs' share of an SM: d = 2048 up to 16 experts)
bool route_tile_applies(const moe_config& c, int T) {
  return T > MOE_STREAM_MAX_TOKENS && rt_shape(c.d_model, c.n_experts).smem <= 112 * 1024;
}

template <typename XT>
static int launch_route_t(moe_ctx* ctx, const void* x, int T, const moe_weights* w, int32_t* idx, float* wt,
                          float* probs, cudaStream_t s, const Grouping* grp, const Scatter* sc) {
  const moe_config& c = ctx->cfg;
  const XT* xp = (const XT*)x;
  const uint16_t* wr = (const uint16_t*)w->w_router;
  const RtShape sh = rt_shape(c.d_model, c.n_experts);
  if (route_tile_applies(c, T)) {
    MOE_TRY(allow_full_smem<route_tile_kernel<XT>>(ctx));
    MOE_CUDA_TRY(launch_pdl(route_tile_kernel<XT>, dim3((T + kRtTokens - 1) / kRtTokens), dim3(kRtWarps * 32), (size_t)sh.smem, s,
                            xp, wr, w->b_router, T, c.d_model, c.n_experts, c.top_k, c.renorm, idx, wt, probs,
                            grp ? *grp : Grouping{nullptr, nullptr, nullptr}, sc ? *sc : Scatter{nullptr, nullptr}, ctx->d_state));
    ctx->launches++;
    return MOE_OK;
  }
  const dim3 block(kRouteWarps * 32);
  const bool few = T <= 64;
  const dim3 grid(few ? T : (T + kRouteWarps - 1) / kRouteWarps);
#define ROUTE_CASE(EM)                                                                                                \
  MOE_CUDA_TRY(launch_pdl(few ? route_block_kernel<XT, EM> : route_kernel<XT, EM>, grid, block, 0, s, xp, wr, w->b_router, \
                          T, c.d_model, c.n_experts, c.top_k, c.renorm, idx, wt, probs))
  if (c.n_experts <= 8)
    ROUTE_CASE(8);
  else if (c.n_experts <= 16)
    ROUTE_CASE(16);
  else if (c.n_experts <= 32)
    ROUTE_CASE(32);
  else
    ROUTE_CASE(64);
#undef ROUTE_CASE
  ctx->launches++;
  return grp ? launch_permute(ctx, idx, T, grp->offsets, grp->perm, grp->inv, s) : MOE_OK;
}

int launch_route(moe_ctx* ctx, const void* x, int T, const moe_weights* w, int32_t* idx, float* wt, float* probs,
                 cudaStream_t s, const Grouping* grp, const Scatter* sc) {
  if (ctx->cfg.x_dtype == MOE_F32) return launch_route_t<float>(ctx, x, T, w, idx, wt, probs, s, grp, sc);
  return launch_route_t<__nv_bfloat16>(ctx, x, T, w, idx, wt, probs, s, grp, sc);
}

// ------------------------------------------------------------------------------------ grouping
// One CTA: histogram of the T*k pairs by expert, exclusive scan, then a stable scatter that walks
// the pairs in order, 1024 at a time (rank inside a warp by match_any, across warps by a scan).
constexpr int kPermThreads = 1024;

__global__ void __launch_bounds__(kPermThreads)
    permute_kernel(const int32_t* __restrict__ topk_idx, int n, int E, int32_t* __restrict__ offsets,
                   int32_t* __restrict__ perm, int32_t* __restrict__ inv, DeviceState* st) {
  __shared__ int s_base[MOE_MAX_EXPERTS];
  __shared__ int s_wc[kPermThreads / 32][MOE_MAX_EXPERTS];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_launch_dependents();
  pdl_wait();
  if (tid < MOE_MAX_EXPERTS) s_base[tid] = 0;
  __syncthreads();
  for (int p = tid; p < n; p += kPermThreads) {
    const int e = topk_idx[p];
    if (e < 0 || e >= E)
      flag_error(st, MOE_ERR_STATE, 0x100u);
    else
      atomicAdd(&s_base[e], 1);
  }
  __syncthreads();
  if (tid == 0) {
    int run = 0;
    for (int e = 0; e < E; ++e) {
      const int c = s_base[e];
      offsets[e] = run;
      s_base[e] = run;
      run += c;
    }
    offsets[E] = run;
  }
  __syncthreads();
  for (int p0 = 0; p0 < n; p0 += kPermThreads) {
    for (int i = tid; i < (kPermThreads / 32) * MOE_MAX_EXPERTS; i += kPermThreads) (&s_wc[0][0])[i] = 0;
    __syncthreads();
    const int p = p0 + tid;
    int e = -1;
    if (p < n) {
      e = topk_idx[p];
      if (e < 0 || e >= E) e = -1;
    }
    const unsigned peers = __match_any_sync(0xffffffffu, e);
    const int rank = __popc(peers & ((1u << lane) - 1u));
    if (e >= 0 && rank == 0) s_wc[warp][e] = __popc(peers);
    __syncthreads();
    if (tid < E) {
      int run = s_base[tid];
      for (int w = 0; w < kPermThreads / 32; ++w) {
        const int c = s_wc[w][tid];
        s_wc[w][tid] = run;
        run += c;
      }
      s_base[tid] = run;
    }
    __syncthreads();
    if (e >= 0) {
      const int slot = s_wc[warp][e] + rank;
      perm[slot] = p;
      inv[p] = slot;
    }
    __syncthreads();
  }
}

int launch_permute(moe_ctx* ctx, const int32_t* idx, int T, int32_t* offsets, int32_t* perm, int32_t* inv,
                   cudaStream_t s) {
  const moe_config& c = ctx->cfg;
  MOE_CUDA_TRY(launch_pdl(permute_kernel, dim3(1), dim3(kPermThreads), 0, s, idx, T * c.top_k, c.n_experts, offsets, perm, inv,
                          ctx->d_state));
  ctx->launches++;
  return MOE_OK;
}

// ------------------------------------------------------------------------------------ gather
// xperm[s][:] = bf16(x[perm[s] / k][:])  (operand rows of the tensor-core path, grouped by expert).  A warp per row, up to
// eight 16-byte chunks per lane on their way at a time, no index arithmetic per chunk.  (Rows cut into parts so that few rows
// fill the SMs: 58.3 against 56.4 us for 512 tokens at d 1024 -- the next kernel's CTAs find the SMs occupied.)
constexpr int kRowWarps = 8;
template <typename XT>
__global__ void __launch_bounds__(kRowWarps * 32)
    gather_rows_kernel(const XT* __restrict__ x, const int32_t* __restrict__ perm, int n_slots, int k, int d, uint4* __restrict__ out) {
  constexpr int kFly = sizeof(XT) == 4 ? 4 : 8;
  const int chunks = d / 8, lane = threadIdx.x & 31, s = blockIdx.x * kRowWarps + (threadIdx.x >> 5);
  pdl_launch_dependents();
  pdl_wait();
  if (s >= n_slots) return;
  const XT* row = x + (size_t)(perm[s] / k) * d;
  uint4* dst = out + (size_t)s * chunks;
  for (int c0 = lane; c0 < chunks; c0 += 32 * kFly) {
    float f[kFly][8];
#pragma unroll
    for (int u = 0; u < kFly; ++u)
      if (c0 + 32 * u < chunks) load_x8<XT>(row + (c0 + 32 * u) * 8, f[u]);
#pragma unroll
    for (int u = 0; u < kFly; ++u)
      if (c0 + 32 * u < chunks)
        dst[c0 + 32 * u] = make_uint4(pack_bf16x2(f[u][0], f[u][1]), pack_bf16x2(f[u][2], f[u][3]),
                                      pack_bf16x2(f[u][4], f[u][5]), pack_bf16x2(f[u][6], f[u][7]));
  }
}

int launch_gather_rows(moe_ctx* ctx, const void* x, const int32_t* perm, int n_slots, void* xperm, cudaStream_t s) {
  const moe_config& c = ctx->cfg;
  const dim3 grid((n_slots + kRowWarps - 1) / kRowWarps), block(kRowWarps * 32);
  if (c.x_dtype == MOE_F32)
    MOE_CUDA_TRY(launch_pdl(gather_rows_kernel<float>, grid, block, 0, s, (const float*)x, perm, n_slots, c.top_k, c.d_model,
                            (uint4*)xperm));
  else
    MOE_CUDA_TRY(launch_pdl(gather_rows_kernel<__nv_bfloat16>, grid, block, 0, s, (const __nv_bfloat16*)x, perm, n_slots, c.top_k,
                            c.d_model, (uint4*)xperm));
  ctx->launches++;
  return MOE_OK;
}

// ------------------------------------------------------------------------------------ combine
// y[t][c] = sum_j w[t][j] * out_slots[inv[t*k+j]][c], j ascending, fp32, one rounding to the output type; PL planes of partial
// sums of a cut contraction are added in order.  A warp per part of a row: a token's slots and weights are read once and
// handed round by shuffles, and all planes' loads of a choice are on their way together.
template <typename YT, int PL>
__global__ void __launch_bounds__(kRowWarps * 32)
    combine_kernel(const float* __restrict__ out_slots, const float* __restrict__ wt, const int32_t* __restrict__ inv, int T, int k,
                   int d, int parts, YT* __restrict__ y) {
  constexpr int kFly = PL == 1 ? 4 : 2;
  const int quads = d / 4, lane = threadIdx.x & 31, wid = blockIdx.x * kRowWarps + (threadIdx.x >> 5);
  const int t = wid / parts, part = wid - t * parts;
  pdl_launch_dependents();
  pdl_wait();
  if (t >= T) return;
  const int my_slot = lane < k ? inv[(size_t)t * k + lane] : 0;
  const float my_w = lane < k ? wt[(size_t)t * k + lane] : 0.f;
  const size_t plane = (size_t)T * k * quads;
  const int per = (quads + parts - 1) / parts, q_lo = part * per, q_hi = min(quads, q_lo + per);
  for (int q0 = q_lo + lane; __any_sync(0xffffffffu, q0 < q_hi); q0 += 32 * kFly) {
    float4 acc[kFly];
#pragma unroll
    for (int u = 0; u < kFly; ++u) acc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int j = 0; j < k; ++j) {
      const float w = __shfl_sync(0xffffffffu, my_w, j);
      const float4* src = reinterpret_cast<const float4*>(out_slots) + (size_t)__shfl_sync(0xffffffffu, my_slot, j) * quads;
      float4 o[PL][kFly];
#pragma unroll
      for (int pl = 0; pl < PL; ++pl)
#pragma unroll
        for (int u = 0; u < kFly; ++u) o[pl][u] = src[pl * plane + min(q0 + 32 * u, quads - 1)];
#pragma unroll
      for (int u = 0; u < kFly; ++u) {
        float4 s = o[0][u];
#pragma unroll
        for (int pl = 1; pl < PL; ++pl) s.x += o[pl][u].x, s.y += o[pl][u].y, s.z += o[pl][u].z, s.w += o[pl][u].w;
        acc[u].x = fmaf(w, s.x, acc[u].x), acc[u].y = fmaf(w, s.y, acc[u].y);
        acc[u].z = fmaf(w, s.z, acc[u].z), acc[u].w = fmaf(w, s.w, acc[u].w);
      }
    }
#pragma unroll
    for (int u = 0; u < kFly; ++u) {
      const int q = q0 + 32 * u;
      if (q >= q_hi) continue;
      if constexpr (sizeof(YT) == 4)
        reinterpret_cast<float4*>(y + (size_t)t * d)[q] = acc[u];
      else
        reinterpret_cast<uint2*>(y + (size_t)t * d)[q] = make_uint2(pack_bf16x2(acc[u].x, acc[u].y), pack_bf16x2(acc[u].z, acc[u].w));
    }
  }
}

template <typename YT>
static int launch_combine_t(moe_ctx* ctx, const float* out_slots, const float* wt, const int32_t* inv, int T, YT* y, int planes,
                            cudaStream_t s) {
  const moe_config& c = ctx->cfg;
  // enough warps to fill the SMs where there are few tokens, but no part shorter than one round of loads
  const int round = planes == 1 ? 128 : 64, most = std::max(1, (c.d_model / 4 + round - 1) / round);
  const int parts = std::min(most, std::max(1, (16 * ctx->sm_count + T - 1) / T));
  const dim3 grid(((unsigned)T * parts + kRowWarps - 1) / kRowWarps), block(kRowWarps * 32);
#define COMBINE(PL) MOE_CUDA_TRY(launch_pdl(combine_kernel<YT, PL>, grid, block, 0, s, out_slots, wt, inv, T, c.top_k, c.d_model, parts, y))
  switch (planes) {
    case 1: COMBINE(1); break;
    case 2: COMBINE(2); break;
    case 3: COMBINE(3); break;
    default: COMBINE(4); break;
  }
#undef COMBINE
  ctx->launches++;
  return MOE_OK;
}

static_assert(kKSplitMax == 4, "combine_kernel's instantiations");
int launch_combine(moe_ctx* ctx, const float* out_slots, const float* wt, const int32_t* inv, int T, void* y,
                   int planes, cudaStream_t s) {
  return ctx->cfg.x_dtype == MOE_F32 ? launch_combine_t(ctx, out_slots, wt, inv, T, (float*)y, planes, s)
                                     : launch_combine_t(ctx, out_slots, wt, inv, T, (__nv_bfloat16*)y, planes, s);
}

// out[i] = sum over the planes, in order (n a multiple of 4)
__global__ void sum_planes_kernel(const float4* __restrict__ in, long long quads, int planes, float4* __restrict__ out) {
  pdl_launch_dependents();
  pdl_wait();
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < quads; i += (long long)gridDim.x * blockDim.x) {
    float4 o = in[i];
    for (int pl = 1; pl < planes; ++pl) {
      const float4 o2 = in[i + pl * quads];
      o.x += o2.x, o.y += o2.y, o.z += o2.z, o.w += o2.w;
    }
    out[i] = o;
  }
}

int launch_sum_planes(moe_ctx* ctx, const float* in, long long n, int planes, float* out, cudaStream_t s) {
  const long long quads = n / 4, want = (quads + 255) / 256;
  const int grid = (int)(want < 16ll * ctx->sm_count ? want : 16ll * ctx->sm_count);
  MOE_CUDA_TRY(launch_pdl(sum_planes_kernel, dim3(grid), dim3(256), 0, s, (const float4*)in, quads, planes, (float4*)out));
  ctx->launches++;
  return MOE_OK;
}

// The planes of [rows][n] partial sums added in order and split into bf16 head and remainder: out [rows][hi n | lo n]
__global__ void split_planes_kernel(const float4* __restrict__ in, int rows, int n, int planes, uint2* __restrict__ out) {
  const int quads = n / 4;
  const long long total = (long long)rows * quads;
  pdl_launch_dependents();
  pdl_wait();
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    float4 o = in[i];
    for (int pl = 1; pl < planes; ++pl) {
      const float4 o2 = in[i + pl * total];
      o.x += o2.x, o.y += o2.y, o.z += o2.z, o.w += o2.w;
    }
    const uint2 hi = make_uint2(pack_bf16x2(o.x, o.y), pack_bf16x2(o.z, o.w));
    const uint2 lo = make_uint2(pack_bf16x2(o.x - __uint_as_float(hi.x << 16), o.y - __uint_as_float(hi.x & 0xffff0000u)),
                                pack_bf16x2(o.z - __uint_as_float(hi.y << 16), o.w - __uint_as_float(hi.y & 0xffff0000u)));
    const long long r = i / quads;
    out[r * quads + i] = hi;  // row r starts at 2 r quads
    out[r * quads + i + quads] = lo;
  }
}

int launch_split_planes(moe_ctx* ctx, const float* in, int rows, int n, int planes, void* out, cudaStream_t s) {
  const long long want = ((long long)rows * (n / 4) + 255) / 256;
  const int grid = (int)(want < 16ll * ctx->sm_count ? want : 16ll * ctx->sm_count);
  MOE_CUDA_TRY(launch_pdl(split_planes_kernel, dim3(grid), dim3(256), 0, s, (const float4*)in, rows, n, planes, (uint2*)out));
  ctx->launches++;
  return MOE_OK;
}

// ------------------------------------------------------------------------------------ packing
// in [B][R][C] -> out[b][c][sub][r] with nsub interleaved row kinds: a tiled transpose.
__global__ void pack_transpose_kernel(const uint16_t* __restrict__ in, uint16_t* __restrict__ out, int R, int C,
                                      int nsub, int sub) {
  __shared__ uint16_t tile[32][33];
  const int b = blockIdx.z;
  const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  const uint16_t* src = in + (size_t)b * R * C;
  uint16_t* dst = out + (size_t)b * C * nsub * R;
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int r = r0 + i, c = c0 + threadIdx.x;
    if (r < R && c < C) tile[i][threadIdx.x] = src[(size_t)r * C + c];
  }
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int c = c0 + i, r = r0 + threadIdx.x;
    if (r < R && c < C) dst[((size_t)c * nsub + sub) * R + r] = tile[threadIdx.x][i];
  }
}

// out[b][c][sub][:] = in[b][c][:]  (rows copied into an interleaved layout, 16 bytes per thread)
__global__ void pack_rows_kernel(const uint4* __restrict__ in, uint4* __restrict__ out, long long rows, int chunks,
                                 int nsub, int sub) {
  const long long total = rows * chunks;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const long long r = i / chunks;
    const int c = (int)(i - r * chunks);
    out[(r * nsub + sub) * chunks + c] = in[i];
  }
}

static int pack_one(const void* in, void* out, int B, int R, int C, int nsub, int sub, cudaStream_t s) {
  const dim3 grid((C + 31) / 32, (R + 31) / 32, B), block(32, 8);
  if (grid.y > 65535u || grid.z > 65535u) return MOE_ERR_UNSUPPORTED;
  pack_transpose_kernel<<<grid, block, 0, s>>>((const uint16_t*)in, (uint16_t*)out, R, C, nsub, sub);
  MOE_CUDA_TRY(cudaGetLastError());
  return MOE_OK;
}

}  // namespace cosmoe

using namespace cosmoe;

extern "C" {

int moe_pack_dense(int32_t d, int32_t f, int32_t n_experts, const void* w_gate, const void* w_up, const void* w_down,
                   void* gud_out, void* stream) {
  if (d <= 0 || f <= 0 || n_experts <= 0 || !w_gate || !w_up || !w_down || !gud_out) return MOE_ERR_INVALID_ARG;
  if (d % 8 || f % 8) return MOE_ERR_UNSUPPORTED;
  cudaStream_t s = (cudaStream_t)stream;
  int rc = pack_one(w_gate, gud_out, n_experts, d, f, 3, 0, s);
  if (rc == MOE_OK) rc = pack_one(w_up, gud_out, n_experts, d, f, 3, 1, s);
  if (rc == MOE_OK) {
    pack_rows_kernel<<<148 * 8, 256, 0, s>>>((const uint4*)w_down, (uint4*)gud_out, (long long)n_experts * f, d / 8, 3, 2);
    MOE_CUDA_TRY(cudaGetLastError());
  }
  return rc;
}

int moe_pack_wd(int32_t d, int32_t f, int32_t r, int32_t n_experts, const void* gL, const void* gR, const void* uL,
                const void* uR, const void* dL, const void* dR, void* wd_a, void* wd_b, void* wd_c, void* wd_d,
                void* stream) {
  if (d <= 0 || f <= 0 || r <= 0 || n_experts <= 0 || !gL || !gR || !uL || !uR || !dL || !dR || !wd_a || !wd_b ||
      !wd_c || !wd_d)
    return MOE_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  int rc = pack_one(gL, wd_a, n_experts, d, r, 2, 0, s);
  if (rc == MOE_OK) rc = pack_one(uL, wd_a, n_experts, d, r, 2, 1, s);
  if (rc == MOE_OK) rc = pack_one(gR, wd_b, n_experts, r, f, 2, 0, s);
  if (rc == MOE_OK) rc = pack_one(uR, wd_b, n_experts, r, f, 2, 1, s);
  if (rc == MOE_OK) rc = pack_one(dL, wd_c, n_experts, f, r, 1, 0, s);
  if (rc == MOE_OK) rc = pack_one(dR, wd_d, n_experts, r, d, 1, 0, s);
  return rc;
}

}  // extern "C"
