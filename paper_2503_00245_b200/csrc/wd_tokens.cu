// Decode of a layer with weight-decomposed experts (Eq. 1) for several tokens (T <= 16), and the per-slot expert FFN
// of the streaming path: ONE launch that streams every selected expert's factors once and does the arithmetic on
// the tensor cores.
//
//   product 0   t = x [gL | uL]                           rows (j, gate|up) of d values   wd_a [S][r][2][d]
//   product 1   h_c = silu(t_g . gR_c) * (t_u . uR_c)     pairs of rows of r values       wd_b [S][f][2][r]
//   product 2   v = h dL                                  rows of f values                wd_c [S][r][f]
//   product 3   y = sum_a w_a (v_a dR_a)                  rows of r values                wd_d [S][d][r]
//
// Every product is a skinny GEMM per active expert: out[slot][row] = W[row][:] . in[slot][:], at most 8 tokens at a
// time.  It is bound by the bytes of the factors, so the weights go through a ring of shared-memory stages filled
// with bulk asynchronous copies, and the arithmetic goes to mma.sync m16n8k16 (16 weight rows x 8 tokens): the
// instruction count does not grow with the tokens of an expert.  (N = 8 tokens is far below a tcgen05 tile; the MMA
// only has to keep out of the way of the stream.)  The input vectors are kept as THREE bf16 terms whose sum is the
// fp32 value (8 + 8 + 8 significand bits), each with accumulators of its own, so t, h and v carry fp32 precision as
// in the one-token kernels; bf16 token rows are one exact term.
//
// Rows of (active expert x product) are dealt to the CTAs (one per SM) evenly, row by row, while there are many active experts;
// with eight CTAs or more for each a CTA works for one of them (kAlignCtas); in product 3 the CTAs split
// the output columns instead, each summing all experts itself, so every value has one writer and a fixed order of
// summation: no atomics, results bit-identical from call to call.  Between the products the CTAs meet at an arrival
// counter that runs over launches, with a bounded wait.
//
// A CTA's rows of a product are walked in groups of up to 4 tiles of 16 rows; a group goes through the contraction
// in slices of at most 448 values.  Roles, talking through mbarriers only (all waits bounded):
//   weight producer thread a stage = one tile's slice, in at most two tiled TMA loads of 16 rows x 224 values (one copy
//                          per row: 100 cycles of the issuing thread per KB, a third of the copy bandwidth).  The
//                          weights depend on nothing but the routing, so it runs ahead across the meetings as far as
//                          the ring allows;
//   vector producer warp   meets the other CTAs, then brings the slices of the input vectors, one copy per token;
//   8 consumer warps       split a slice's 32-value units; a unit's input fragments stay in registers for all tiles
//                          of the group.  A lane fetches 8 consecutive values of a row at a time (16 bytes) and the two
//                          MMA steps of a unit take them in that order, weights and vectors alike: the order of the
//                          contraction inside a unit is free;
//   2 epilogue warps       add the 8 warps' partial sums in order, SiLU * mul, split into terms, store.
// Measured on B200, d 1600, f 4352, r 800, 8 experts, 2 active, T = 5, two layers (about 170 MB of factors each, 26 us at
// the copy bandwidth): 134 to 139 us, by GPU.  The kernel before it (fp32 multiply-adds, one warp for vectors, barriers and epilogues, a
// router launch of 10 us) took 430 to 470.  What a layer's 66 us go to: three meetings and the refill behind them (about 15), the
// router (4), the products at 4 to 5 TB/s.
#include <cuda.h>

#include "common.cuh"

namespace cosmoe {

namespace {

constexpr int kConsWarps = 8;
constexpr int kTeams = 2, kTeamWarps = kConsWarps / kTeams;
constexpr int kEpiWarp0 = kConsWarps;
constexpr int kEpiWarps = 2;  // (12 warps in all: three per SM sub-partition, 168 registers each)
constexpr int kWeightWarp = kEpiWarp0 + kEpiWarps;
constexpr int kVectorWarp = kWeightWarp + 1;
constexpr int kThreads = (kVectorWarp + 1) * 32;
static_assert(kThreads == 12 * 32, "the router adds twelve warps' shares");
constexpr int kTileRows = 16;
constexpr int kTok = 8;                          // tokens of one expert per pass (N of the MMA)
constexpr int kTerms = 3;                        // bf16 terms of an fp32 value
constexpr int kUnit = 32;                        // contraction values of two MMA steps
constexpr int kBoxK = 224;                       // one TMA load: a tile's rows x 7 units.  Not 256: rows 448 bytes apart
                                                 // let lanes of two neighbouring rows fetch 16 bytes each without a bank
                                                 // conflict (512 apart: two-way, shared memory was the bottleneck)
constexpr int kBoxBytes = kBoxK * kTileRows * 2;
constexpr int kSlice = 2 * kBoxK;                // contraction values per stage
static_assert(kTeams == 2 && kTeamWarps == 4, "the epilogue adds two teams of four");
static_assert(kSlice == kWdSlice, "the workspace is laid out in slices");
constexpr int kStageBytes = 2 * kBoxBytes;       // [column half][16 rows][224 values]
constexpr int kUnits = (kSlice / kUnit + kTeamWarps - 1) / kTeamWarps;  // units of a stage for each warp of a team
constexpr int kTermRun = kWdTermRun;             // values between two terms of a slice: 64 bytes beyond a multiple of 128, so
                                                 // that lanes of two terms meet no bank conflict
constexpr int kVecRun = kTerms * kTermRun;       // values of one token's slice, in memory as in shared memory
constexpr int kTokBytes = kVecRun * 2;
constexpr int kMaxStages = 5;                    // of one team
constexpr int kMaxVecs = 8;
constexpr int kGroupTiles = 4;                   // tiles of 16 rows of a group
constexpr int kPartTok = kTileRows;              // floats between two tokens' partial sums
constexpr int kPartTile = kTok * kPartTok;
constexpr int kPartBytes = kGroupTiles * kConsWarps * kPartTile * 4;  // one of two buffers
constexpr int kMaxSlots = MOE_STREAM_MAX_TOKENS * MOE_MAX_TOPK;
constexpr int kProducts = 4;
// With this many CTAs per active expert or more a CTA's rows are all of one expert: the shares are then up to 1 / 8 uneven,
// which costs less than the partly filled tiles on both sides of an expert boundary (at 6 experts the CTAs with a boundary
// finished a product up to 9 % after the others).
constexpr int kAlignCtas = 8;

struct Product {
  int rows;      // outputs per expert
  int K;         // contraction length
  int nsub;      // 2: an output is made from a (gate, up) pair of rows, each with an input vector of its own
  int n_slices;  // slices of the contraction
};

struct WtParams {
  int T, k, E, d, mode, x_is_bf16, y_rows;
  int n_stages;  // of a team's ring
  const uint16_t* x;  // bf16 rows [T][d], or fp32 rows as terms [T][slice][3][480]
  const uint16_t* w_router;  // set: the router runs in the prologue, CTA 0 writes its products to topk_idx / topk_w
  const float* b_router;
  const void* x_rows;        // the token rows as the caller has them
  int renorm;
  int32_t* topk_idx;
  float* topk_w;
  const int32_t* offsets;
  const int32_t* perm;
  const int32_t* expert_slot;
  uint16_t *t, *h, *v;  // terms of the intermediates: [slot][2][slice][3][480], [slot][slice][3][480] twice
  void* y;
  float* out_slots;
  DeviceState* st;
  Product pr[kProducts];
};
struct WtMaps {
  CUtensorMap m[kProducts];  // [slot][row][sub-row][value] of every product's matrix, boxes of 16 rows x 224 values
};

struct WtSmem {
  // Each team has rings of its own: a waiter must see every phase of a barrier it waits on.
  uint64_t full[kTeams][kMaxStages], freeb[kTeams][kMaxStages];
  uint64_t vfull[kTeams][kMaxVecs], vfree[kTeams][kMaxVecs];
  uint64_t pfull[2], pfree[2];
  uint64_t product_done[kProducts];    // this CTA's outputs of the product are stored (one each: a CTA may have no rows of some)
  int act_e[MOE_MAX_EXPERTS];
  int act_slot[MOE_MAX_EXPERTS];       // packed-array slot of the active expert
  int act_off[MOE_MAX_EXPERTS + 1];    // slot ranges, expert-ascending (same numbering as moe_permute)
  int slot_tok[kMaxSlots];
  float slot_w[kMaxSlots];
  int stage_e[kMaxSlots];              // the routing, before grouping
  float stage_w[kMaxSlots];
  int cursor[MOE_MAX_EXPERTS];
  int n_act;
  int vec_toks, n_vecs;                // token slices of a vector buffer (the most tokens an expert has), buffers of a team
  volatile int abort;
};
constexpr int kHeaderBytes = (sizeof(WtSmem) + 127) / 128 * 128;

struct Ring {
  int slot;
  unsigned par;
  int n;
  __device__ __forceinline__ void advance(int slots) {
    ++n;
    if (++slot == slots) slot = 0, par ^= 1u;
  }
};

__device__ __forceinline__ void swap_rings(Ring& mine, Ring& other, int& team) {
  const Ring t = mine;
  mine = other, other = t, team ^= 1;
}

// One group: rows [row0, row0 + rows) of active expert a for the tokens of its slots slot0 .. slot0 + ns - 1.
struct Group {
  int a, slot0, ns, row0, rows;
  bool last_use;  // no further token group reads these rows
};

// This CTA's rows of a product: [g0, g1) of all active experts' rows in a row, beginning in expert a0 (product 3: of each one's).
struct Share {
  int g0, g1, a0;
};
__device__ __forceinline__ Share share_of(const WtParams& P, const WtSmem& sm, int ph) {
  const int N = P.pr[ph].rows, na = sm.n_act;
  const long long b = blockIdx.x, G = gridDim.x;
  if (ph == kProducts - 1) return Share{(int)(N * b / G), (int)(N * (b + 1) / G), 0};
  if ((int)G >= kAlignCtas * na) {
    // a CTA works for one expert: the first G mod na experts get one CTA more
    const int c = (int)G / na, more = (int)G - c * na, big = more * (c + 1), bi = (int)b;
    const int a0 = bi < big ? bi / (c + 1) : more + (bi - big) / c;
    const int jn = bi < big ? bi - a0 * (c + 1) : bi - big - (a0 - more) * c, cn = bi < big ? c + 1 : c;
    return Share{a0 * N + (int)((long long)N * jn / cn), a0 * N + (int)((long long)N * (jn + 1) / cn), a0};
  }
  const long long tot = (long long)na * N;
  const int g0 = (int)(tot * b / G);
  return Share{g0, (int)(tot * (b + 1) / G), g0 / N};
}
// Every role walks this list of groups: a pure function of (routing, product, CTA).
template <class F>
__device__ __forceinline__ bool walk(const WtParams& P, const WtSmem& sm, int ph, const Share& my, F&& body) {
  const int N = P.pr[ph].rows, na = sm.n_act;
  const bool split_out = ph == kProducts - 1;
  constexpr int per = kGroupTiles * kTileRows;
  if (my.g0 >= my.g1) return true;
  for (int a = my.a0; a < na; ++a) {
    const int lo = split_out ? my.g0 : max(my.g0 - a * N, 0), hi = split_out ? my.g1 : min(my.g1 - a * N, N);
    if (hi <= lo) break;
    const int groups = (hi - lo + per - 1) / per;
    const int step = ((hi - lo + groups - 1) / groups + kTileRows - 1) / kTileRows * kTileRows;
    const int s_lo = sm.act_off[a], s_hi = sm.act_off[a + 1];
    for (int r0 = lo; r0 < hi; r0 += step)
      for (int s0 = s_lo; s0 < s_hi; s0 += kTok)
        if (!body(Group{a, s0, min(kTok, s_hi - s0), r0, min(step, hi - r0), s0 + kTok >= s_hi})) return false;
  }
  return true;
}
template <class F>
__device__ __forceinline__ bool walk(const WtParams& P, const WtSmem& sm, int ph, F&& body) {
  return walk(P, sm, ph, share_of(P, sm, ph), body);
}

// The two consumer teams take the slices of the contraction in turn; in product 3, whose groups are one short tile per
// expert, the groups.
__device__ __forceinline__ bool teams_by_group(int ph) { return ph == kProducts - 1; }

__device__ __forceinline__ void give_up(const WtParams& P, WtSmem& sm, unsigned detail) {
  sm.abort = 1;
  flag_error(P.st, MOE_ERR_TIMEOUT, detail);
}

__device__ __forceinline__ void tma_rows(void* dst, const CUtensorMap* map, int k, int sub, int row, int slot, uint64_t* bar,
                                         uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, "
      "%4, %5}], [%6], %7;" ::"r"(smem_u32(dst)),
      "l"(map), "r"(k), "r"(sub), "r"(row), "r"(slot), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}
__device__ __forceinline__ uint64_t l2_policy_normal() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
// All groups of one product by one consumer warp.  (A lane that gives up a wait says so and leaves the kernel: none waits for it.)
// The loops stay rolled and serve all products (bf16 token rows meet
// zeros as their second and third term): a launch runs each of them a few dozen times only, and code that is fetched
// anew from L2 for every tile costs more than the idle columns.
// The 8 columns of an MMA are two tokens with four columns each: most experts have one or two of the tokens, and one MMA
// then does what three (one per term) did; the columns of a token are added by its two lanes.
// An MMA's sums are cut, not rounded, which pulls every product towards zero by as much as its LARGEST term is long.  So the
// first term has two columns, eight of an MMA's sixteen k-values in either (the second and third terms have one each), every
// MMA starts at zero, and all adding up is done in fp32, in pairs.  Relative error of the layer (d 1600, f 4352, r 800, fp32
// rows) against 64 bits: fp32 multiply-adds 2.7e-7; one column per term and two MMAs in a row 2.9e-7, of which 1.8e-7 is that
// pull; as it is 2.1e-7.  (Eight products per MMA, m16n8k8, instead of the second column: 2.2e-7 and 4 % slower.)
__device__ __forceinline__ bool consume(const WtParams& P, WtSmem& sm, int ph, const unsigned char* stages,
                                        const unsigned char* vecs, float* parts, Ring& rs, Ring& rv, unsigned& turn, Ring& rp,
                                        int warp, int lane) {
  const int K = P.pr[ph].K, nsub = P.pr[ph].nsub;
  const int nt = ph == 0 && P.x_is_bf16 ? 1 : kTerms;
  // The slices of the input vectors are taken by the two teams in turn: a stage is a chain of shared-memory loads, MMAs
  // and additions, and two of them side by side keep up with the stream.
  const unsigned team = warp / kTeamWarps;
  const int tw = warp % kTeamWarps;
  // lane (g, q) = (lane / 4, lane % 4) fetches values 8 q .. 8 q + 7 of a unit, of rows g and g + 8 / of column g; this
  // warp's units are tw, tw + 4, tw + 8, tw + 12 (a column half of a stage holds 7)
  const int g8 = lane >> 2, q4 = lane & 3;
  const uint32_t a_lane = (uint32_t)g8 * (kBoxK * 2) + q4 * 16;
  const int term = g8 & 3, col = tw * kUnit + q4 * 8;
  const bool live = term == 0 || term == 3 || nt == kTerms;
  const uint32_t even = live && term != 3 ? ~0u : 0u, odd = live && term != 0 ? ~0u : 0u;  // of the k-values, in pairs of pairs
  constexpr int kUnitStep = kTeamWarps * kUnit;
  const int n_vecs = sm.n_vecs;
  const bool by_group = teams_by_group(ph);
  return walk(P, sm, ph, [&](const Group& g) -> bool {
    const int tiles = (g.rows + kTileRows - 1) / kTileRows;
    if (rp.n >= 2 && !mbar_wait(&sm.pfree[rp.slot], rp.par ^ 1u)) {
      give_up(P, sm, 0x612u);
      return false;
    }
    if (by_group && turn++ % kTeams != team) {
      if (lane == 0) mbar_arrive(&sm.pfull[rp.slot]);
      rp.advance(2);
      return true;
    }
    // this lane's partial sums, [tile][warp][token][row]: row g8 (even lanes) or g8 + 8 of tokens q4 / 2 + 2 p.  A team's
    // first slice stores, the others add.  Of a (gate, up) pair either team has one; a group with a single slice is
    // one team's alone.
    float* const part = parts + (size_t)rp.slot * (kPartBytes / 4) + warp * kPartTile + (q4 >> 1) * kPartTok + g8 + 8 * (q4 & 1);
    bool first = true;
#pragma unroll 1
    for (int k0 = 0; k0 < K; k0 += kSlice) {
      const int width = min(kSlice, K - k0);
#pragma unroll 1
      for (int sub = 0; sub < nsub; ++sub) {
        if (!by_group && turn++ % kTeams != team) continue;
        if (!mbar_wait(&sm.vfull[team][rv.slot], rv.par)) {
          give_up(P, sm, 0x610u);
          return false;
        }
        const unsigned char* vec = vecs + (team * (uint32_t)kTok + (uint32_t)(rv.slot * sm.vec_toks)) * kTokBytes +
                                   (term < nt ? term : 0) * (kTermRun * 2) + col * 2;  // (column 3: the first term again)
        // (no branches below: what lies past the vector's end is fetched and dropped, and the weights that would meet it
        // are those of unit 0, which are finite, or the zeros TMA puts past the end of a row)
        uint32_t a_off[kUnits];
#pragma unroll
        for (int j = 0; j < kUnits; ++j) {
          const uint32_t n = tw + kTeamWarps * j, hf = n >= kBoxK / kUnit;
          a_off[j] = a_lane + ((int)n * kUnit < width ? hf * kBoxBytes + (n - hf * (kBoxK / kUnit)) * (kUnit * 2) : 0u);
        }
#pragma unroll 1
        for (int u = 0; u < tiles; ++u) {
          if (!mbar_wait(&sm.full[team][rs.slot], rs.par)) {
            give_up(P, sm, 0x611u);
            return false;
          }
          const unsigned char* st = stages + (team * (uint32_t)P.n_stages + (uint32_t)rs.slot) * kStageBytes;
          uint4 lo[kUnits], hi[kUnits];  // rows g8 and g8 + 8
#pragma unroll
          for (int j = 0; j < kUnits; ++j) {
            lo[j] = *reinterpret_cast<const uint4*>(st + a_off[j]);
            hi[j] = *reinterpret_cast<const uint4*>(st + a_off[j] + 8 * kBoxK * 2);
          }
          float* dst = part + u * (kConsWarps * kPartTile);
#pragma unroll 1
          for (int t0 = 0; t0 < g.ns; t0 += 2) {
            const unsigned char* vt = vec + (uint32_t)min(t0 + (g8 >> 2), g.ns - 1) * kTokBytes;
            uint4 b[kUnits];
#pragma unroll
            for (int j = 0; j < kUnits; ++j) {
              b[j] = *reinterpret_cast<const uint4*>(vt + j * (kUnitStep * 2));
              const bool in = col + j * kUnitStep < width;
              b[j].x &= in ? even : 0u, b[j].y &= in ? odd : 0u, b[j].z &= in ? even : 0u, b[j].w &= in ? odd : 0u;
            }
            float m[2 * kUnits][4];
#pragma unroll
            for (int j = 0; j < 2 * kUnits; ++j) m[j][0] = m[j][1] = m[j][2] = m[j][3] = 0.f;
#pragma unroll
            for (int j = 0; j < kUnits; ++j) {
              mma16(m[j], lo[j].x, hi[j].x, lo[j].y, hi[j].y, b[j].x, b[j].y);
              mma16(m[kUnits + j], lo[j].z, hi[j].z, lo[j].w, hi[j].w, b[j].z, b[j].w);
            }
#pragma unroll
            for (int n = kUnits; n > 0; n >>= 1)
#pragma unroll
              for (int j = 0; j < n; ++j) add4(m[j], m[j + n]);
            const float top = m[0][1] + m[0][0], bot = m[0][3] + m[0][2];  // rows g8 and g8 + 8: this lane's two columns
            const float send = (q4 & 1) ? top : bot, keep = (q4 & 1) ? bot : top;
            const float v = keep + __shfl_xor_sync(0xffffffffu, send, 1);
            dst[t0 * kPartTok] = first ? v : dst[t0 * kPartTok] + v;
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(&sm.freeb[team][rs.slot]);
          rs.advance(P.n_stages);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.vfree[team][rv.slot]);
        rv.advance(n_vecs);
        first = false;
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&sm.pfull[rp.slot]);
    rp.advance(2);
    return true;
  });
}

// Router (Eq. 2, Eq. 3) of all T tokens by every CTA, E = 8 or 16.  A thread owns the input features tid, tid + 384, ...:
// their rows of W_r are fetched once and serve every token.
// part: [12 warps][16 tokens][16 experts].
constexpr int kRouteQ = 6;  // features per thread and round: d <= 2304 in one
__device__ __forceinline__ void route_fetch(const WtParams& P, int q0, int e8, int tid, uint4* wr) {
#pragma unroll
  for (int q = 0; q < kRouteQ; ++q)
    wr[q] = ldcg_now(reinterpret_cast<const uint4*>(P.w_router + (size_t)min(tid + (q0 + q) * kThreads, P.d - 1) * P.E + e8));
}
__device__ __forceinline__ void route_tokens(const WtParams& P, WtSmem& sm, float* part, int tid) {
  const int lane = tid & 31, warp = tid >> 5, d = P.d;
  for (int e8 = 0; e8 < P.E; e8 += 8) {
    for (int q0 = 0; q0 * kThreads < d; q0 += kRouteQ) {
      uint4 wr[kRouteQ];
      route_fetch(P, q0, e8, tid, wr);
#pragma unroll 1
      for (int t0 = 0; t0 < P.T; t0 += 4) {
        float xv[4][kRouteQ];  // four tokens' features in one round trip
#pragma unroll
        for (int t = 0; t < 4; ++t)
#pragma unroll
          for (int q = 0; q < kRouteQ; ++q) {
            const int i = tid + (q0 + q) * kThreads;
            const size_t at = (size_t)min(t0 + t, P.T - 1) * d + min(i, d - 1);
            xv[t][q] = P.x_is_bf16 ? bf16_to_float(__ldg((const uint16_t*)P.x_rows + at)) : __ldg((const float*)P.x_rows + at);
            if (i >= d) xv[t][q] = 0.f;
          }
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          float a[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) a[e] = 0.f;
#pragma unroll
          for (int q = 0; q < kRouteQ; ++q) {
            float w[8];
            unpack8(wr[q], w);
#pragma unroll
            for (int e = 0; e < 8; ++e) a[e] = fmaf(xv[t][q], w[e], a[e]);
          }
          const float v = warp_sum8(a, lane);
          if ((lane & 3) == 0 && t0 + t < P.T) {
            float* dst = part + (warp * 16 + t0 + t) * 16 + e8 + (lane >> 2);
            *dst = q0 == 0 ? v : *dst + v;
          }
        }
      }
    }
  }
  __syncthreads();
  for (int t = warp; t < P.T; t += kThreads / 32) {
    float l = 0.f;
    if (lane < P.E) {
      float a[kThreads / 64];  // (in pairs: a serial sum of the warps' shares loses more than all that is in front of it)
#pragma unroll
      for (int w = 0; w < kThreads / 64; ++w) a[w] = part[(2 * w * 16 + t) * 16 + lane] + part[((2 * w + 1) * 16 + t) * 16 + lane];
      l = ((a[0] + a[1]) + (a[2] + a[3])) + (a[4] + a[5]);
      if (P.b_router) l += P.b_router[lane];
    }
    warp_route_finish(l, 0.f, P.E, P.k, P.renorm, lane, sm.stage_e + t * P.k, sm.stage_w + t * P.k, nullptr);
    __syncwarp();
    if (blockIdx.x == 0 && lane < P.k) {
      P.topk_idx[t * P.k + lane] = sm.stage_e[t * P.k + lane];
      P.topk_w[t * P.k + lane] = sm.stage_w[t * P.k + lane];
    }
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kThreads, 1) wd_tokens_kernel(const __grid_constant__ WtParams P, const __grid_constant__ WtMaps M) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  WtSmem& sm = *reinterpret_cast<WtSmem*>(smem_raw);
  unsigned char* const stages = smem_raw + kHeaderBytes;
  unsigned char* const vecs = stages + kTeams * P.n_stages * kStageBytes;
  float* const parts = reinterpret_cast<float*>(vecs + kTeams * kTok * kTokBytes);
  float* const yacc = parts + 2 * (kPartBytes / 4);  // [T][y_rows]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  DeviceState* const st = P.st;

  pdl_launch_dependents();
  if (tid == kWeightWarp * 32) {
    for (int i = 0; i < kProducts; ++i) asm volatile("prefetch.tensormap [%0];" ::"l"(&M.m[i]) : "memory");
    for (int t = 0; t < kTeams; ++t) {
      for (int i = 0; i < P.n_stages; ++i) mbar_init(&sm.full[t][i], 1), mbar_init(&sm.freeb[t][i], kTeamWarps);
      for (int i = 0; i < kMaxVecs; ++i) mbar_init(&sm.vfull[t][i], 1), mbar_init(&sm.vfree[t][i], kTeamWarps);
    }
    for (int i = 0; i < 2; ++i) mbar_init(&sm.pfull[i], kConsWarps), mbar_init(&sm.pfree[i], kEpiWarps);
    for (int i = 0; i < kProducts; ++i) mbar_init(&sm.product_done[i], kEpiWarps);
    fence_mbar_init();
    fence_proxy_async_smem();
    sm.abort = 0;
  }
  if (P.mode == 0)
    for (int i = tid; i < P.T * P.y_rows; i += kThreads) yacc[i] = 0.f;
  if (P.w_router && tid == 0) prefetch_router(P.w_router, P.d, P.E);
  pdl_wait();
  if (P.w_router) route_tokens(P, sm, parts, tid);

  // ---------------------------------------------------------------- routing -> active experts and their slots
  const int n = P.T * P.k;
  if (warp == 0 && P.mode == 0 && n <= 32) {
    const int e = lane < n ? (P.w_router ? sm.stage_e[lane] : P.topk_idx[lane]) : -1;
    const float wt = lane < n ? (P.w_router ? sm.stage_w[lane] : P.topk_w[lane]) : 0.f;
    int pos, rank, bad = lane < n && (e < 0 || e >= P.E);
    bool first;
    const int na = warp_group32(e, n, lane, pos, rank, first);
    if (first && !bad) {
      const int sl = P.expert_slot ? P.expert_slot[e] : e;
      bad = sl < 0;
      sm.act_e[rank] = e, sm.act_off[rank] = pos, sm.act_slot[rank] = sl < 0 ? 0 : sl;
    }
    if (lane < n) sm.slot_tok[pos] = lane / P.k, sm.slot_w[pos] = wt;
    bad = __any_sync(0xffffffffu, bad);
    __syncwarp();
    if (lane == 0) {
      sm.act_off[bad ? 0 : na] = bad ? 0 : n;
      sm.n_act = bad ? 0 : na;  // every CTA takes the same decision from the same data: nobody streams anything
      if (bad) flag_error(st, MOE_ERR_STATE, 0x600u);
    }
  } else if (warp == 0 && P.mode == 0) {
    const unsigned below = (1u << lane) - 1u;
    int bad = 0;
    sm.cursor[lane] = 0, sm.cursor[lane + 32] = 0;
    if (!P.w_router)
      for (int p = lane; p < n; p += 32) sm.stage_e[p] = P.topk_idx[p], sm.stage_w[p] = P.topk_w[p];
    __syncwarp();
    for (int p0 = 0; p0 < n; p0 += 32) {  // counts: the first lane of each group of equal experts adds the group
      const int p = p0 + lane;
      int e = p < n ? sm.stage_e[p] : -1;
      if (p < n && (e < 0 || e >= P.E)) bad = 1, e = -1;
      const unsigned peers = __match_any_sync(0xffffffffu, e);
      if (e >= 0 && (peers & below) == 0u) sm.cursor[e] += __popc(peers);
      __syncwarp();
    }
    const int c[2] = {sm.cursor[lane], sm.cursor[lane + 32]};
    int run = 0, na = 0;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      int s = c[half];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += u;
      }
      const int off = run + s - c[half], e = lane + 32 * half;
      run += __shfl_sync(0xffffffffu, s, 31);
      const unsigned m = __ballot_sync(0xffffffffu, c[half] > 0);
      sm.cursor[e] = off;  // next free slot of every expert
      if (c[half] > 0) {
        const int a = na + __popc(m & below);
        const int sl = P.expert_slot ? P.expert_slot[e] : e;
        bad |= sl < 0;
        sm.act_e[a] = e, sm.act_off[a] = off, sm.act_slot[a] = sl < 0 ? 0 : sl;
      }
      na += __popc(m);
    }
    bad = __any_sync(0xffffffffu, bad);
    __syncwarp();
    for (int p0 = 0; p0 < n && !bad; p0 += 32) {
      const int p = p0 + lane;
      const int e = p < n ? sm.stage_e[p] : -1;
      const unsigned peers = __match_any_sync(0xffffffffu, e);
      const int base = e >= 0 ? sm.cursor[e] : 0;
      __syncwarp();
      if (e >= 0) {
        const int s = base + __popc(peers & below);  // pairs of one expert keep their order
        sm.slot_tok[s] = p / P.k;
        sm.slot_w[s] = sm.stage_w[p];
        if ((peers & below) == 0u) sm.cursor[e] = base + __popc(peers);
      }
      __syncwarp();
    }
    if (lane == 0) {
      sm.act_off[bad ? 0 : na] = bad ? 0 : n;
      sm.n_act = bad ? 0 : na;  // every CTA takes the same decision from the same data: nobody streams anything
      if (bad) flag_error(st, MOE_ERR_STATE, 0x600u);
    }
  } else if (warp == 0) {
    // the caller's grouping (moe_permute's products): lane e works for experts e and e + 32
    int bad = 0, run = 0, na = 0;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int e = lane + 32 * half;
      const int lo = e < P.E ? P.offsets[e] : 0, hi = e < P.E ? P.offsets[e + 1] : 0;
      const int c = hi - lo;
      bad |= lo < 0 || c < 0 || hi > n;
      int end = bad ? 0 : c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, end, o);
        if (lane >= o) end += u;
      }
      const bool any = !bad && c > 0;
      const int off = run + end - c;
      bad |= any && lo != off;
      run += __shfl_sync(0xffffffffu, end, 31);
      const unsigned m = __ballot_sync(0xffffffffu, any);
      if (any) {
        const int a = na + __popc(m & ((1u << lane) - 1u)), sl = P.expert_slot ? P.expert_slot[e] : e;
        bad |= sl < 0;
        sm.act_e[a] = e, sm.act_slot[a] = sl < 0 ? 0 : sl, sm.act_off[a] = off;
      }
      na += __popc(m);
    }
    for (int s = lane; s < n; s += 32) {
      const int p = P.perm[s];
      bad |= p < 0 || p >= n;
      sm.slot_tok[s] = p / P.k, sm.slot_w[s] = 1.0f;
    }
    bad = __any_sync(0xffffffffu, bad || run != n);
    if (lane == 0) {
      sm.act_off[bad ? 0 : na] = bad ? 0 : n;
      sm.n_act = bad ? 0 : na;
      if (bad) flag_error(st, MOE_ERR_STATE, 0x600u);
    }
  }
  if (warp == 0) {
    // the vector buffers are cut to the tokens the busiest expert has: with few, more slices are on their way
    __syncwarp();
    int most = 1;
    for (int a = lane; a < sm.n_act; a += 32) most = max(most, sm.act_off[a + 1] - sm.act_off[a]);
    most = min(__reduce_max_sync(0xffffffffu, most), kTok);
    if (lane == 0) sm.vec_toks = most, sm.n_vecs = min(kMaxVecs, kTok / most);
  }
  __syncthreads();
  // From here on the roles meet at mbarriers only; every wait is bounded.
  const int last = sm.n_act > 0 ? kProducts : 0;  // (nothing to do: no products, no meetings, zeros out)

  if (warp == kWeightWarp) {
    // ================================================================= weight producer
    if (lane != 0) return;
    const uint64_t once = l2_policy_evict_first(), keep = l2_policy_normal();
    Ring rs{0, 0u, 0}, other{0, 0u, 0};  // the ring of the team whose turn it is, the other team's
    int team = 0;
    bool ok = true;
#pragma unroll 1
    for (int ph = 0; ph < last && ok; ++ph) {
      const Product& pr = P.pr[ph];
      const CUtensorMap* map = &M.m[ph];
      const int K = pr.K, nsub = pr.nsub;
      const bool by_group = teams_by_group(ph);
      ok = walk(P, sm, ph, [&](const Group& g) -> bool {
        const int e = sm.act_slot[g.a];
        for (int k0 = 0; k0 < K; k0 += kSlice) {
          const int halves = K - k0 > kBoxK ? 2 : 1;
          for (int sub = 0; sub < nsub; ++sub) {
            for (int u = 0; u < g.rows; u += kTileRows) {
              const int row = g.row0 + u;
              // rows another CTA or another token group reads as well stay in L2
              const uint64_t pol = g.last_use && g.rows - u >= kTileRows ? once : keep;
              uint64_t* bar = &sm.full[team][rs.slot];
              if ((rs.n >= P.n_stages && !mbar_wait(&sm.freeb[team][rs.slot], rs.par ^ 1u)) || sm.abort) {
                give_up(P, sm, 0x620u);
                return false;
              }
              mbar_arrive_expect_tx(bar, (uint32_t)(halves * kBoxBytes));
              unsigned char* dst = stages + (size_t)(team * P.n_stages + rs.slot) * kStageBytes;
              tma_rows(dst, map, k0, sub, row, e, bar, pol);
              if (halves == 2) tma_rows(dst + kBoxBytes, map, k0 + kBoxK, sub, row, e, bar, pol);
              rs.advance(P.n_stages);
            }
            if (!by_group) swap_rings(rs, other, team);
          }
        }
        if (by_group) swap_rings(rs, other, team);
        return true;
      });
    }
    if (!ok)  // copies in flight must land before this CTA's shared memory goes away
      for (int t = 0; t < kTeams; ++t, rs = other, team ^= 1)
        for (int j = max(0, rs.n - P.n_stages); j < rs.n; ++j)
          (void)mbar_wait(&sm.full[team][j % P.n_stages], (unsigned)(j / P.n_stages) & 1u);
    return;
  }

  if (warp == kVectorWarp) {
    // ================================================================= vector producer, meetings
    Ring rv{0, 0u, 0}, other{0, 0u, 0};  // the ring of the team whose turn it is, the other team's
    int team = 0;
    const int n_vecs = sm.n_vecs, vec_bytes = sm.vec_toks * kTokBytes;
    bool ok = true;
#pragma unroll 1
    for (int ph = 0; ph < last && ok; ++ph) {
      const Share my = share_of(P, sm, ph);  // (its divisions are done when the meeting is over)
      if (ph > 0) {  // every CTA has stored its outputs of the product before
        int met = 1;
        if (lane == 0) {
          met = mbar_wait(&sm.product_done[ph - 1], 0u);
          if (met) {
            // (release: the epilogue warps' stores, ordered before this thread by the barrier; acquire: the others')
            const unsigned G = gridDim.x;
            const unsigned long long old = atom_add_acq_rel64(&st->phase_total, 1ull);
            const unsigned long long target = old - old % G + G;
            const long long t0 = clock64();
            while (ld_acquire64(&st->phase_total) < target)
              if (clock64() - t0 > kWaitBudgetCycles || sm.abort) {
                met = 0;
                break;
              }
          }
          if (!met) give_up(P, sm, 0x630u);
        }
        ok = __shfl_sync(0xffffffffu, met, 0) != 0;
        if (!ok) break;
        fence_proxy_async_all();  // the vectors were stored through the generic proxy, the copies below read them
      }
      const Product& pr = P.pr[ph];
      const int K = pr.K;
      const bool by_group = teams_by_group(ph);
      ok = walk(P, sm, ph, my, [&](const Group& g) -> bool {
        // lane = the token whose slices it brings
        const bool mine = lane < g.ns;
        const int s = g.slot0 + min(lane, g.ns - 1);
        const bool plain = ph == 0 && P.x_is_bf16;  // rows of x themselves
        const size_t run = (size_t)pr.n_slices * kVecRun;
        const uint16_t* src = plain     ? P.x + (size_t)sm.slot_tok[s] * K
                              : ph == 0 ? P.x + (size_t)sm.slot_tok[s] * run
                              : ph == 1 ? P.t + (size_t)s * 2 * run
                                        : (ph == 2 ? P.h : P.v) + (size_t)s * run;
        for (int ks = 0; ks < pr.n_slices; ++ks) {
          const uint32_t bytes = plain ? (uint32_t)min(kSlice, K - ks * kSlice) * 2u : (uint32_t)kVecRun * 2u;
          for (int sub = 0; sub < pr.nsub; ++sub) {
            if (!__all_sync(0xffffffffu, (rv.n < n_vecs || mbar_wait(&sm.vfree[team][rv.slot], rv.par ^ 1u)) && !sm.abort)) {
              if (lane == 0) give_up(P, sm, 0x631u);
              return false;
            }
            if (lane == 0) mbar_arrive_expect_tx(&sm.vfull[team][rv.slot], bytes * (uint32_t)g.ns);
            __syncwarp();
            if (mine)
              bulk_g2s(vecs + (size_t)team * kTok * kTokBytes + (size_t)rv.slot * vec_bytes + (size_t)lane * kTokBytes,
                       src + sub * run + (size_t)ks * (plain ? kSlice : kVecRun), bytes, &sm.vfull[team][rv.slot]);
            rv.advance(n_vecs);
            if (!by_group) swap_rings(rv, other, team);
          }
        }
        if (by_group) swap_rings(rv, other, team);
        return true;
      });
    }
    if (!ok)
      for (int t = 0; t < kTeams; ++t, rv = other, team ^= 1)
        for (int j = max(0, rv.n - n_vecs); j < rv.n; ++j) (void)mbar_wait(&sm.vfull[team][j % n_vecs], (unsigned)(j / n_vecs) & 1u);
    return;
  }

  if (warp >= kEpiWarp0) {
    // ================================================================= epilogue
    // Warp ew takes rows 8 ew .. 8 ew + 7 of every tile, a lane one (row, token) pair at a time: in product 3 all
    // experts' contributions to an output meet in one warp, in expert order.
    const int rq = 8 * (warp - kEpiWarp0) + (lane & 7), q0 = lane >> 3;
    const int y0 = (int)((long long)P.d * blockIdx.x / gridDim.x);
    Ring rp{0, 0u, 0};
    unsigned turn = 0;  // as the consumers count their slices
    bool ok = true;
#pragma unroll 1
    for (int ph = 0; ph < last && ok; ++ph) {
      const Product& pr = P.pr[ph];
      const bool by_group = teams_by_group(ph);
      ok = walk(P, sm, ph, [&](const Group& g) -> bool {
        if (!mbar_wait_warp(&sm.pfull[rp.slot], rp.par)) {
          if (lane == 0) give_up(P, sm, 0x640u);
          return false;
        }
        const int items = (g.rows + kTileRows - 1) / kTileRows * g.ns;
        int u = 0, tok = q0;  // item (tile u, token tok) = number q of tiles x tokens
        for (int q = q0; q < items; q += 4, tok += 4) {
          while (tok >= g.ns) tok -= g.ns, ++u;
          const int s = g.slot0 + tok;
          const float* part = parts + (size_t)rp.slot * (kPartBytes / 4) + tok * kPartTok + rq;
          const float* p = part + (size_t)u * kConsWarps * kPartTile;
          float sum[kTeams];
#pragma unroll
          for (int t = 0; t < kTeams; ++t) {
            const float* pt = p + t * kTeamWarps * kPartTile;
            sum[t] = (pt[0] + pt[kPartTile]) + (pt[2 * kPartTile] + pt[3 * kPartTile]);
          }
          const int rl = u * kTileRows + rq, row = g.row0 + rl;
          float v;
          const float mine = sum[turn % kTeams], theirs = sum[(turn + 1) % kTeams];  // the team of the first slice, the other
          if (pr.nsub == 2)
            v = mine / (1.0f + expf(-mine)) * theirs;
          else
            v = pr.n_slices > 1 && !by_group ? sum[0] + sum[1] : mine;
          if (rl >= g.rows) continue;
          if (ph == kProducts - 1) {
            if (P.mode == 1)
              P.out_slots[(size_t)s * P.d + row] = v;
            else
              yacc[sm.slot_tok[s] * P.y_rows + (row - y0)] += sm.slot_w[s] * v;
          } else {
            uint16_t tm[kTerms];
            split3(v, tm);
            // (product 0's rows are (j, gate | up) pairs)
            const int c = ph == 0 ? row >> 1 : row, sl = ph == 0 ? 2 * s + (row & 1) : s;
            uint16_t* dst = (ph == 0 ? P.t : ph == 1 ? P.h : P.v) +
                            ((size_t)sl * P.pr[ph + 1].n_slices + c / kSlice) * kVecRun + c % kSlice;
#pragma unroll
            for (int i = 0; i < kTerms; ++i) dst[i * kTermRun] = tm[i];
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.pfree[rp.slot]);
        rp.advance(2);
        turn += by_group ? 1u : (unsigned)(pr.n_slices * pr.nsub);
        return true;
      });
      ok = __all_sync(0xffffffffu, ok);
      __syncwarp();
      if (ok && lane == 0) mbar_arrive(&sm.product_done[ph]);
    }
    if (ok && P.mode == 0) {
      const int y1 = (int)((long long)P.d * (blockIdx.x + 1) / gridDim.x);
      for (int r0 = 0; r0 < y1 - y0; r0 += kTileRows)
        for (int t = q0; t < P.T; t += 4) {
          const int rl = r0 + rq;
          if (rl >= y1 - y0) continue;
          const float v = yacc[t * P.y_rows + rl];
          if (P.x_is_bf16)
            ((__nv_bfloat16*)P.y)[(size_t)t * P.d + y0 + rl] = __float2bfloat16_rn(v);
          else
            ((float*)P.y)[(size_t)t * P.d + y0 + rl] = v;
        }
    }
    return;
  }

  // ===================================================================== consumers
  Ring rs{0, 0u, 0}, rv{0, 0u, 0}, rp{0, 0u, 0};
  unsigned turn = 0;
  bool ok = true;
#pragma unroll 1
  for (int ph = 0; ph < last && ok; ++ph) ok = consume(P, sm, ph, stages, vecs, parts, rs, rv, turn, rp, warp, lane);
}

// fp32 token rows -> their bf16 terms [T][slice][3][480]
__global__ void split_rows_kernel(const float* __restrict__ x, int d, uint16_t* __restrict__ out) {
  pdl_launch_dependents();
  pdl_wait();
  const float* row = x + (size_t)blockIdx.x * d;
  uint16_t* dst = out + (size_t)blockIdx.x * ((d + kSlice - 1) / kSlice) * kVecRun;
  for (int i = threadIdx.x; i < d; i += blockDim.x) {
    uint16_t tm[kTerms];
    split3(row[i], tm);
#pragma unroll
    for (int j = 0; j < kTerms; ++j) dst[(size_t)(i / kSlice) * kVecRun + j * kTermRun + i % kSlice] = tm[j];
  }
}

}  // namespace

// 8 or 16 experts: the shapes whose partial logits the prologue holds.  (A router launch in front of the kernel instead: 156
// against 133 us for the two layers above.)
bool wd_tokens_fuses_route(const moe_config& c) { return (c.n_experts & 7) == 0 && c.n_experts <= 16; }

int launch_wd_tokens(moe_ctx* ctx, int mode, const void* x, int T, const moe_weights* w, int32_t* topk_idx,
                     float* topk_w, const int32_t* offsets, const int32_t* perm, void* y, float* out_slots, char* ws,
                     const WsLayout& L, cudaStream_t s) {
  const moe_config& c = ctx->cfg;
  if (c.wd_rank == 0) return MOE_ERR_UNSUPPORTED;  // dense experts stream through launch_dense_stream
  const int d = c.d_model, f = c.d_ff, r = c.wd_rank, G = ctx->sm_count;
  WtParams P{};
  P.T = T, P.k = c.top_k, P.E = c.n_experts, P.d = d, P.mode = mode;
  P.x_is_bf16 = c.x_dtype == MOE_BF16;
  P.topk_idx = topk_idx, P.topk_w = topk_w, P.offsets = offsets, P.perm = perm, P.expert_slot = w->expert_slot;
  P.t = (uint16_t*)(ws + L.vec_a), P.h = (uint16_t*)(ws + L.vec_b), P.v = (uint16_t*)(ws + L.vec_c);
  P.renorm = c.renorm, P.x_rows = x;
  if (mode == 0 && wd_tokens_fuses_route(c)) P.w_router = (const uint16_t*)w->w_router, P.b_router = w->b_router;
  P.y = y, P.out_slots = out_slots, P.st = ctx->d_state;
  P.y_rows = (d + G - 1) / G + 1;
  WtMaps M;
  int rc = MOE_OK;
  auto set = [&](int i, const void* mat, int rows, int K, int nsub) {
    P.pr[i] = Product{rows, K, nsub, (K + kSlice - 1) / kSlice};
    // (the slot coordinate never leaves the array: its extent is not needed, only the rows' end inside a slot is)
    if (rc == MOE_OK) rc = make_map_rows(&M.m[i], mat, K, nsub, rows, MOE_MAX_EXPERTS << 10, kBoxK, kTileRows);
  };
  set(0, w->wd_a, 2 * r, d, 1);
  set(1, w->wd_b, f, r, 2);
  set(2, w->wd_c, r, f, 1);
  set(3, w->wd_d, d, r, 1);
  if (rc != MOE_OK) return rc;
  const size_t fixed = kHeaderBytes + (size_t)kTeams * kTok * kTokBytes + 2 * (size_t)kPartBytes +
                       (mode == 0 ? (size_t)T * P.y_rows * 4 : 0);
  P.n_stages = (int)min((long long)kMaxStages, ((long long)ctx->max_smem_optin - (long long)fixed) / (kTeams * kStageBytes));
  if (P.n_stages < 2) return MOE_ERR_UNSUPPORTED;
  const size_t smem = fixed + (size_t)kTeams * P.n_stages * kStageBytes;
  if (P.x_is_bf16) {
    P.x = (const uint16_t*)x;
  } else {
    uint16_t* terms = (uint16_t*)(ws + L.vec_x);
    MOE_CUDA_TRY(launch_pdl(split_rows_kernel, dim3(T), dim3(256), 0, s, (const float*)x, d, terms));
    ctx->launches++;
    P.x = terms;
  }
  MOE_TRY(allow_full_smem<wd_tokens_kernel>(ctx));
  // The CTAs wait for one another, so the launch is cooperative: it starts only when all of them fit on the device.
  cudaLaunchConfig_t lc{};
  lc.gridDim = dim3(G), lc.blockDim = dim3(kThreads), lc.dynamicSmemBytes = smem, lc.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = attr, lc.numAttrs = 2;
  MOE_CUDA_TRY(cudaLaunchKernelEx(&lc, wd_tokens_kernel, P, M));
  ctx->launches++;
  return MOE_OK;
}

}  // namespace cosmoe
