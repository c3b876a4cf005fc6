// Prefill of dense experts: both expert GEMMs of a layer in ONE launch on the 5th-generation tensor cores.
//
//   (1) H = silu(X Wg) * (X Wu)   bf16 [slot][f]        (2) O = H Wd   fp32 [part][slot][d]
//
// The weights are the M side of the products (rows of a tile: features; columns: an expert's tokens), so an expert with few
// tokens costs few columns and every weight passes through shared memory once per 256 tokens of its expert.  Two CTAs on
// neighbouring SMs (a cluster of 2) compute a tile with tcgen05.mma.cta_group::2, M = 256 over the pair: each stages hb (at most
// 128) features of its own and HALF of the tile's tokens.  A tile of (1) has two weight matrices, gate and up, against the same
// tokens.
//   warp 0     loads weights, 64-wide K slices, into a ring of shared-memory slots;
//   warp 2     loads the K step's tokens (both CTAs' copies complete on a barrier of the leader's);
//   warp 1     in the leader, one elected lane issues the MMAs for the pair;
//   warp 3     in the leader, takes the pair's tiles; in the other CTA, writes down where the (token, choice) pairs went;
//   warps 4-19 epilogue: one tensor-memory lane = one feature per thread.
// Tiles of (1), then of (2), are numbered through, and a pair takes the next number from a counter when it is about to run out of
// loads.  A tile of (2) waits for its expert's tiles of (1) at a counter of theirs; there is no barrier over the grid and no second
// launch.  Because the numbers are taken in order and by pairs that run, a wait is always for tiles that a running pair has in
// hand, and those of (1) wait for nobody: the launch ends however few of its CTAs find room at a time, beside whatever else the
// GPU runs.  (With the tiles dealt out by block number it did not: a pair without an SM held tiles that others waited for.)
//
// Why so: with the tokens on the M side, an expert's last 256-row tile cost what a full one does, and 128 weight rows were loaded
// for every 128 token rows.  Here a K step of a pair is 48 KB per CTA for 2 x 256 features x 256 tokens instead of 64 KB, an
// expert's last tile costs what its tokens cost, and the tiles of (2) fill what the last round of (1) leaves idle.
// What bounds it: with 256 tokens per expert and more, the tensor cores (a tile of phase 1 with 224 columns and 32 K steps takes 17
// us, 28.7 k cycles of them) and the special-function unit, which the epilogue's exponentials and reciprocals keep busy for 2 us per
// tile, in the open when a tile takes all 512 columns; with fewer, HBM and the round trip of 1.5 us through the ring.
// Before (five launches, tokens on the M side) and now, whole layer, graphs of 20 calls on one GPU: d 1024, f 2816, 512 tokens 53.6 ->
// 51.1 us; d 1440, f 3840, 333 tokens 81.2 -> 66.7; d 2048, f 5632, 2048 tokens 296 -> 256 (for seconds on end, under the power cap, 301).
// Tried: weights asked into L2 ahead of their loads, from the router's launch or from here (less than 1 us for 30 MB, 2 lost for 92);
// the first K steps loaded in front of the dependency wait (about half a us); eight epilogue warps that keep a tile's gate sums in 128
// registers, to free half of the accumulators early (registers spill to L2: +100 us).
// All waits are bounded; an expired wait sets the ctx's status word.  Every CTA fetches what it needs with its own loads (no
// multicast).
#include "tcgen.cuh"

namespace cosmoe {

namespace {

constexpr int kEpiWarpsDP = 16;  // four per quarter of the tensor-memory lanes
constexpr int kThreadsDP = (4 + kEpiWarpsDP) * 32;
constexpr int kSteps = 16;  // K steps in the ring at most (a power of two)
constexpr int kEpiBytesDP = kEpiWarpsDP * 1024;
constexpr int kAhead = 4;   // K steps in front of a tile's end at which the next tile is taken: a microsecond or two
constexpr int kQueue = 4;   // tiles on their way to the roles (a power of two)

struct DPPhase {
  int K, num_kb;    // contraction length, its K steps
  int m_total;      // output features of a weight matrix
  int hb;           // features of a tile per CTA and weight matrix (a pair's tile: 2 hb)
  int ksplit;       // parts the contraction is cut into, each a tile of its own
  int per_tok;      // tiles per token tile: feature tiles x ksplit
};

struct DPParams {
  const unsigned* counts;  // [E] tokens of each expert, or null: ...
  const int32_t* offsets;  // ... [E+1] slot ranges
  int E, n_pairs_tk;       // experts, (token, choice) pairs
  int cap;                 // > 0: the rows of x are grouped at [e * cap ...] and not by slot
  const int32_t *topk_idx, *pos;  // with counts: the pairs' experts and places among their expert's tokens ...
  int32_t* inv;                   // ... from which their slots are worked out
  int w_max, tb;           // tokens of a tile at most (a multiple of 32, <= 256), token rows per box
  DPPhase ph[2];
  __nv_bfloat16* hidden;
  float* out;
  long long plane_elems;
  int ring_slots, slot_bytes;  // the ring: slots of one operand's K step each
  int likely;  // tokens per expert under even routing
  DeviceState* st;
};

// The experts' slots and token tiles, a column of the table per lane (lane l: experts l and l + 32).
struct TokenMap {
  int n[2][32];   // tokens
  int lo[2][32];  // first slot
  int w[2][32];   // width of the expert's tiles: its tokens dealt out evenly, rounded up to 32
  int p[2][32];   // token tiles of the experts up to and including this one
};

struct SmemDP {
  uint64_t full[kSteps];    // leader's: both CTAs' operands of the K step have landed (weights' and tokens' producer arrive)
  uint64_t empty[kSteps];   // own: the MMAs have finished reading this CTA's operands of the K step
  uint64_t accum_full[2];        // own: all MMAs of the tile have completed
  uint64_t accum_empty[2];       // leader's: columns [256 b, 256 b + 256) have been read out of both CTAs' tensor memory
  uint64_t tile_full[kQueue];    // own: the pair's next tile is there
  uint64_t tile_empty[kQueue];   // leader's: all roles of both CTAs have read it (the epilogue, which comes last, arrives)
  uint64_t tile_ask;             // leader's: the loads of the tokens of the tile in hand are about to end
  int first_no;
  int4 tile[kQueue][2];
  TokenMap map;
  uint32_t tmem_base;
};

// The table from the lane's n0 and n1.  Every warp writes it (the same values) and reads what its own lanes wrote: it is in
// shared memory to be out of the registers.
__device__ __forceinline__ void token_map(TokenMap& m, int lane, int w_max, int n0, int n1, int& total, int& widest) {
  const int t0 = (n0 + w_max - 1) / w_max, t1 = (n1 + w_max - 1) / w_max;
  const int w0 = t0 ? ((n0 + t0 - 1) / t0 + 31) & ~31 : 0, w1 = t1 ? ((n1 + t1 - 1) / t1 + 31) & ~31 : 0;
  widest = (int)__reduce_max_sync(0xffffffffu, (unsigned)max(w0, w1));
  int p0 = t0, p1 = t1, s0 = n0, s1 = n1;
#pragma unroll 1
  for (int o = 1; o < 32; o <<= 1) {
    const int a = __shfl_up_sync(0xffffffffu, p0, o), b = __shfl_up_sync(0xffffffffu, p1, o);
    const int c = __shfl_up_sync(0xffffffffu, s0, o), d = __shfl_up_sync(0xffffffffu, s1, o);
    if (lane >= o) p0 += a, p1 += b, s0 += c, s1 += d;
  }
  p1 += __shfl_sync(0xffffffffu, p0, 31), s1 += __shfl_sync(0xffffffffu, s0, 31);
  total = __shfl_sync(0xffffffffu, p1, 31);
  volatile TokenMap& v = m;
  v.n[0][lane] = n0, v.n[1][lane] = n1, v.lo[0][lane] = s0 - n0, v.lo[1][lane] = s1 - n1;
  v.w[0][lane] = w0, v.w[1][lane] = w1, v.p[0][lane] = p0, v.p[1][lane] = p1;
}

struct TokTile {
  int e, s0, x0, toks, n, f0, ks;  // expert; first slot, first row of x; tokens, width; first feature; part of the contraction
  int tiles;                       // token tiles of the expert
};
// idx-th tile of a phase: expert major, then feature tile, then part of the contraction, then token tile (pairs that run side by
// side share the weights).  By a whole warp.
__device__ __forceinline__ TokTile decode_tile(const DPPhase& H, int cap, int w_max, const volatile TokenMap& m, int lane, int idx) {
  TokTile t;
  const int mt = idx / H.per_tok;
  // the first expert whose tiles reach past mt (mt < total: there is one)
  const int e = __popc(__ballot_sync(0xffffffffu, m.p[0][lane] <= mt)) + __popc(__ballot_sync(0xffffffffu, m.p[1][lane] <= mt));
  const int h = e >> 5, l = e & 31;
  const int p = __shfl_sync(0xffffffffu, m.p[h][lane], l), n = __shfl_sync(0xffffffffu, m.n[h][lane], l);
  const int lo = __shfl_sync(0xffffffffu, m.lo[h][lane], l);
  t.n = __shfl_sync(0xffffffffu, m.w[h][lane], l);
  t.tiles = (n + w_max - 1) / w_max;
  const int local = idx - (p - t.tiles) * H.per_tok;
  const int rest = local / t.tiles, ft = rest / H.ksplit, tok = (local - rest * t.tiles) * t.n;
  t.e = e;
  t.s0 = lo + tok, t.x0 = cap > 0 ? e * cap + tok : t.s0;
  t.toks = min(t.n, n - tok);
  t.ks = rest - ft * H.ksplit;
  t.f0 = ft * 2 * H.hb;
  return t;
}

// 16 tokens (registers) x 32 features (lanes) as bf16 to rows of tokens, through 1 KB of shared memory: two tokens of the lane's
// feature at a time ...
__device__ __forceinline__ void put_tokens(unsigned char* ebuf, int lane, int j, float v0, float v1) {
  const uint32_t o = pack_bf16x2(v0, v1);
  *reinterpret_cast<uint16_t*>(ebuf + j * 64 + lane * 2) = (uint16_t)o;
  *reinterpret_cast<uint16_t*>(ebuf + (j + 1) * 64 + lane * 2) = (uint16_t)(o >> 16);
}
// ... and then eight tokens' 64 bytes per instruction.  toks, feats: how many of them exist (feats a multiple of 8).
__device__ __forceinline__ void send_tokens(const unsigned char* ebuf, int lane, __nv_bfloat16* out, long long ld, int toks, int feats) {
  const int piece = lane & 3;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int r = (lane >> 2) + 8 * i;
    if (r < toks && piece * 8 < feats)
      *reinterpret_cast<uint4*>(out + (size_t)r * ld + piece * 8) = *reinterpret_cast<const uint4*>(ebuf + r * 64 + piece * 16);
  }
}

// A K step's weights into their slots; the leader's lane announces both CTAs' bytes.  By a whole warp.
__device__ __forceinline__ void load_gate_up(const CUtensorMap* map, uint64_t* full, uint32_t rank, uint32_t gate, uint32_t up, uint32_t bytes,
                                             int k, int f, int e, uint32_t bar) {
  if (elect_one()) {
    if (rank == 0) mbar_arrive_expect_tx(full, 4u * bytes);
    tma_load_4d(gate, map, k, 0, f, e, bar);
    tma_load_4d(up, map, k, 1, f, e, bar);
  }
  __syncwarp();
}
__device__ __forceinline__ void load_down(const CUtensorMap* map, uint64_t* full, uint32_t rank, uint32_t dst, uint32_t bytes, int k,
                                          int f, int e, uint32_t bar) {
  constexpr uint32_t block = 64 * kBK * 2;
  if (elect_one()) {
    if (rank == 0) mbar_arrive_expect_tx(full, 2u * bytes);
    tma_load_4d(dst, map, f, 2, k, e, bar);
    if (bytes > block) tma_load_4d(dst + block, map, f + 64, 2, k, e, bar);
  }
  __syncwarp();
}

// A role's place in the ring: K step, and the slot that its first operand takes.  A K step of phase 1 takes three slots (gate,
// up, tokens), one of phase 2 two (down, tokens), so that phase 2 has more K steps on their way.
struct RingPos {
  int step, slot;
  __device__ __forceinline__ int at(int i, int ns) const { return slot + i < ns ? slot + i : slot + i - ns; }
  __device__ __forceinline__ void next(int slots, int ns) { ++step, slot = at(slots, ns); }
};
// A producer's: what is free, and the oldest K step that has not been handed back.
struct Room {
  int free, oldest;
};
// steps1: the pair's K steps of phase 1, as far as they are known.
__device__ __forceinline__ bool make_room(SmemDP& sm, Room& r, int step, int need, int steps1) {
  while (r.free < need || step - r.oldest >= kSteps) {
    if (!mbar_wait_warp(&sm.empty[r.oldest & (kSteps - 1)], (r.oldest / kSteps) & 1)) return false;
    r.free += r.oldest < steps1 ? 3 : 2;
    ++r.oldest;
  }
  r.free -= need;
  return true;
}

// The pair's tiles after the first go to both CTAs as a whole, so that no role but one works them out.  idx >= the number of
// tiles: there is none.  By one thread of the leader.
__device__ __forceinline__ void hand_out(SmemDP& sm, int b, int idx, const TokTile& t) {
#pragma unroll
  for (uint32_t r = 0; r < 2; ++r) {
    const uint32_t dst = map_to_rank(&sm.tile[b][0], r), bar = map_to_rank(&sm.tile_full[b], r);
    st_async4(dst, make_int4(idx, t.e, t.s0, t.x0), bar);
    st_async4(dst + 16, make_int4(t.toks | t.n << 16, t.f0, t.ks, t.tiles), bar);
  }
}

__global__ void __launch_bounds__(kThreadsDP, 1)
    dense_prefill_kernel(const __grid_constant__ CUtensorMap map_w1, const __grid_constant__ CUtensorMap map_x1,
                         const __grid_constant__ CUtensorMap map_w2, const __grid_constant__ CUtensorMap map_x2,
                         const __grid_constant__ DPParams P) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  // the ring's slots are identical in both CTAs, because the MMA addresses the pair's operands by one shared-memory offset
  const uint32_t a1_bytes = (uint32_t)P.ph[0].hb * kBK * 2, a2_bytes = (uint32_t)P.ph[1].hb * kBK * 2;
  unsigned char* slots = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char* const epi_bufs = slots + (size_t)P.ring_slots * P.slot_bytes;
  SmemDP& sm = *reinterpret_cast<SmemDP*>(epi_bufs + kEpiBytesDP);
  const int tid = threadIdx.x, lane = tid & 31, warp = lane0(tid >> 5);
  const int NS = P.ring_slots;
  const uint32_t rank = (uint32_t)lane0((int)cluster_ctarank());
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;

  // The pair's first number is taken in front of the dependency wait, and lies there when the counts are known.  That is safe
  // because this kernel does not let its successors start early: they find the counter set back.  (Started early, they would
  // only hold places: letting them in at the start of the launch costs a microsecond, d 1024, f 2816, 512 tokens 51.7 and 50.5 us.)
  cluster_arrive();
  int first_no = 0;
  const bool takes = rank == 0 && tid == 3 * 32;
  if (takes) first_no = (int)atomicAdd(&P.st->ffn_next, 1u);
  if (tid == 0) {
    for (int i = 0; i < kSteps; ++i) {
      mbar_init(&sm.full[i], 2);
      mbar_init(&sm.empty[i], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&sm.accum_full[b], 1);
      mbar_init(&sm.accum_empty[b], 2 * kEpiWarpsDP);
    }
    for (int i = 0; i < kQueue; ++i) {
      mbar_init(&sm.tile_full[i], 1);
      mbar_init(&sm.tile_empty[i], 2 * kEpiWarpsDP);
      mbar_arrive_expect_tx(&sm.tile_full[i], 32);
    }
    mbar_init(&sm.tile_ask, 1);
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_w1) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_x1) : "memory");
    fence_mbar_init();
    fence_proxy_async_smem();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sm.tmem_base)),
                 "n"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  cluster_wait();  // (the other CTA has started: its shared memory may be written)
  if (takes) sm.first_no = first_no, st_cluster(map_to_rank(&sm.first_no, 1u), (uint32_t)first_no);
  __syncthreads();
  __syncwarp();
  cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem = (uint32_t)lane0((int)sm.tmem_base);
  const uint32_t full0 = (uint32_t)lane0((int)map_to_rank(&sm.full[0], 0u)), st0 = (uint32_t)lane0((int)smem_u32(slots)), slot_bytes = (uint32_t)P.slot_bytes;
  // The experts' slots and the pair's first tile are worked out twice: in front of the dependency wait as if every expert had
  // the same number of tokens, and from the counts behind it.  The first pass only brings in the code of the second, which
  // stands in front of the first loads.
  TokTile t{};
  int total = 0, widest = 0, n_work1 = 0, n_work = 0, idx = lane0(sm.first_no);
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    const int e1 = lane + 32;
    int n0 = lane < P.E ? P.likely : 0, n1 = e1 < P.E ? P.likely : 0;
    if (pass == 1) {
      pdl_wait();
      if (P.counts) {
        n0 = lane < P.E ? (int)__ldcg(P.counts + lane) : 0, n1 = e1 < P.E ? (int)__ldcg(P.counts + e1) : 0;
      } else {
        const int a = min(lane, P.E), b = min(e1, P.E);
        n0 = max(P.offsets[min(a + 1, P.E)] - P.offsets[a], 0), n1 = max(P.offsets[min(b + 1, P.E)] - P.offsets[b], 0);
      }
    }
    __syncthreads();  // (no warp still reads the first pass's table)
    token_map(sm.map, lane, P.w_max, n0, n1, total, widest);
    n_work1 = total * P.ph[0].per_tok, n_work = n_work1 + total * P.ph[1].per_tok;
    t.e = -1;
    if (idx < n_work) {  // (with few tiles a pair's first one may be of phase 2)
      const int ph = idx >= n_work1;
      t = decode_tile(P.ph[ph], ph ? 0 : P.cap, P.w_max, sm.map, lane, idx - (ph ? n_work1 : 0));
    }
  }
  // accumulators: two buffers of 256 columns, or, for two matrices and more than 128 tokens, a single one of 512
  const bool two = widest <= 128;
  const uint32_t acc1 = two ? 128u : 256u;  // the up products' columns behind the gate's
  // the pair's seq-th tile to idx and t (the first one is there); false: there is none
  auto next_tile = [&](int seq) {
    if (seq > 0) {
      const int b = (seq - 1) & (kQueue - 1);
      if (!mbar_wait_warp(&sm.tile_full[b], ((seq - 1) / kQueue) & 1)) {
        if (lane == 0) flag_error(P.st, MOE_ERR_TIMEOUT, 0x416u);
        return false;
      }
      const int4 u = sm.tile[b][0], v = sm.tile[b][1];
      if (tid == 0) mbar_arrive_expect_tx(&sm.tile_full[b], 32);  // (for the tile kQueue further on)
      idx = lane0(u.x);
      t.e = lane0(u.y), t.s0 = lane0(u.z), t.x0 = lane0(u.w);
      t.toks = lane0(v.x) & 0xffff, t.n = lane0(v.x) >> 16, t.f0 = lane0(v.y), t.ks = lane0(v.z), t.tiles = lane0(v.w);
    }
    return idx < n_work;
  };

  if (warp == 0) {
    // ================================================================= weights (both CTAs)
    RingPos at{0, 0};
    Room room{NS, 0};
    int steps1 = 0x7fffffff;
    bool ok = true;
    for (int seq = 0; ok && next_tile(seq); ++seq) {
      const int ph = idx >= n_work1;
      const DPPhase& H = P.ph[ph];
      if (ph) steps1 = min(steps1, at.step);
      const int kb0 = t.ks * H.num_kb / H.ksplit, kb1 = (t.ks + 1) * H.num_kb / H.ksplit, f = t.f0 + (int)rank * H.hb;
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!(ok = make_room(sm, room, at.step, 3 - ph, steps1))) {
          if (lane == 0) flag_error(P.st, MOE_ERR_TIMEOUT, 0x410u);
          break;
        }
        const int b = at.step & (kSteps - 1);
        const uint32_t dst = st0 + (uint32_t)at.slot * slot_bytes, bar = full0 + 8u * (uint32_t)b;
        if (ph == 0)
          load_gate_up(&map_w1, &sm.full[b], rank, dst, st0 + (uint32_t)at.at(1, NS) * slot_bytes, a1_bytes, kb * kBK, f, t.e, bar);
        else
          load_down(&map_w2, &sm.full[b], rank, dst, a2_bytes, kb * kBK, f, t.e, bar);
        at.next(3 - ph, NS);
      }
    }
    if (!ok && rank == 0) {  // copies in flight (both CTAs' complete on these barriers) must land before the pair goes away
      for (int j = max(0, at.step - kSteps); j < at.step; ++j) (void)mbar_wait(&sm.full[j & (kSteps - 1)], (j / kSteps) & 1);
    }
  } else if (warp == 2) {
    // ================================================================= tokens (both CTAs)
    RingPos at{0, 0};
    Room room{NS, 0};
    int steps1 = 0x7fffffff;
    bool ok = true;
    for (int seq = 0; ok && next_tile(seq); ++seq) {
      const int ph = idx >= n_work1;
      const DPPhase& H = P.ph[ph];
      if (ph) steps1 = min(steps1, at.step);
      if (ph == 1) {  // the expert's hidden activations: all of its tiles of phase 1 have been stored
        const unsigned want = (unsigned)(t.tiles * P.ph[0].per_tok * 2 * kEpiWarpsDP);
        const long long c0 = clock64();
        while (ok && ld_acquire(&P.st->ffn_done[t.e]) < want) ok = clock64() - c0 <= kWaitBudgetCycles;
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) {
          if (lane == 0) flag_error(P.st, MOE_ERR_TIMEOUT, 0x414u);
          break;
        }
        fence_proxy_async_all();  // (they were written by ordinary stores and are read by the copy engine)
      }
      const int boxes = (t.n / 2 + P.tb - 1) / P.tb, box_bytes = P.tb * kBK * 2;
      const int row = (ph ? t.s0 : t.x0) + (int)rank * (t.n / 2);
      const int kb0 = t.ks * H.num_kb / H.ksplit, kb1 = (t.ks + 1) * H.num_kb / H.ksplit, ask = max(kb0, kb1 - kAhead);
      for (int kb = kb0; kb < kb1; ++kb) {
        // (here and not where the weights are loaded: a pair that waits for hidden activations takes no further tiles meanwhile)
        if (kb == ask && rank == 0 && lane == 0) mbar_arrive(&sm.tile_ask);
        if (!(ok = make_room(sm, room, at.step, 3 - ph, steps1))) {
          if (lane == 0) flag_error(P.st, MOE_ERR_TIMEOUT, 0x415u);
          break;
        }
        const int b = at.step & (kSteps - 1);
        uint32_t dst = st0 + (uint32_t)at.at(2 - ph, NS) * slot_bytes;
        const uint32_t bar = full0 + 8u * (uint32_t)b;
        if (elect_one()) {
          if (rank == 0) mbar_arrive_expect_tx(&sm.full[b], (uint32_t)(2 * boxes * box_bytes));
          int r = row;
          if (ph == 0)
            for (int i = 0; i < boxes; ++i, r += P.tb, dst += box_bytes) tma_load_2d(dst, &map_x1, kb * kBK, r, bar);
          else
            for (int i = 0; i < boxes; ++i, r += P.tb, dst += box_bytes) tma_load_2d(dst, &map_x2, kb * kBK, r, bar);
        }
        __syncwarp();
        at.next(3 - ph, NS);
      }
    }
    if (!ok && rank == 0) {
      for (int j = max(0, at.step - kSteps); j < at.step; ++j) (void)mbar_wait(&sm.full[j & (kSteps - 1)], (j / kSteps) & 1);
    }
  } else if (warp == 1) {
    // ================================================================= MMA issuer (leader CTA only)
    if (rank == 0) {
      const uint64_t hi_k = smem_desc(0, 16, 1024) & 0xffffffff00000000ull;                  // K-major: gate, up, tokens
      const uint64_t hi_m = smem_desc(0, 64 * kBK * 2, 1024) & 0xffffffff00000000ull;        // [k][feature]: down
      const uint32_t lbo_k = 1u << 16, lbo_m = (uint32_t)(64 * kBK * 2 >> 4) << 16;
      const uint32_t slot0 = st0 >> 4, slot_step = slot_bytes >> 4;
      RingPos at{0, 0};
      int used0 = 0, used1 = 0;  // tiles that have gone through either half of the accumulators
      bool ok = true;
      auto operands = [&]() {  // of the ring's current K step
        if (mbar_wait_warp(&sm.full[at.step & (kSteps - 1)], (at.step / kSteps) & 1)) {
          tc_fence_after();
          return true;
        }
        if (lane == 0) flag_error(P.st, MOE_ERR_TIMEOUT, 0x411u);
        return false;
      };
      auto drained = [&](int b, int used) {  // what was there before has left, in both CTAs
        if (used == 0) return true;
        if (mbar_wait_warp(&sm.accum_empty[b], (used - 1) & 1)) {
          tc_fence_after();
          return true;
        }
        if (lane == 0) flag_error(P.st, MOE_ERR_TIMEOUT, 0x413u);
        return false;
      };
      for (int seq = 0; ok && next_tile(seq); ++seq) {
        const int ph = idx >= n_work1;
        const DPPhase& H = P.ph[ph];
        const int buf = ph == 0 && !two ? 0 : seq & 1;
        const bool both = ph == 0 && !two;
        if (!(ok = drained(buf, buf ? used1 : used0) && (!both || drained(1, used1)))) break;
        const uint32_t idesc = instr_desc(t.n, ph == 1), d_tmem = tmem + (uint32_t)(buf * kAccCols);
        int kb = t.ks * H.num_kb / H.ksplit;
        const int kb1 = (t.ks + 1) * H.num_kb / H.ksplit;
        uint32_t acc = 0;
        auto release = [&]() {  // both CTAs' producers may refill the slots once the MMAs issued so far have read them
          tc_commit_pair(&sm.empty[at.step & (kSteps - 1)]);
          if (kb + 1 == kb1) tc_commit_pair(&sm.accum_full[buf]);
        };
        for (; kb < kb1; ++kb) {
          if (!(ok = operands())) break;
          const uint32_t lo = slot0 + (uint32_t)at.slot * slot_step, lo_b = slot0 + (uint32_t)at.at(2 - ph, NS) * slot_step;
          const uint64_t db = hi_k | (uint64_t)(lo_b | lbo_k);
          if (ph == 0) {
            const uint64_t da = hi_k | (uint64_t)(lo | lbo_k), da1 = hi_k | (uint64_t)((slot0 + (uint32_t)at.at(1, NS) * slot_step) | lbo_k);
            if (elect_one()) {
#pragma unroll
              for (uint32_t kk = 0; kk < kBK / 16; ++kk) {
                tc_mma_bf16(d_tmem, da + 2u * kk, db + 2u * kk, idesc, acc | kk);
                tc_mma_bf16(d_tmem + acc1, da1 + 2u * kk, db + 2u * kk, idesc, acc | kk);
              }
              release();
            }
          } else {
            const uint64_t da = hi_m | (uint64_t)(lo | lbo_m);
            if (elect_one()) {
#pragma unroll
              for (uint32_t kk = 0; kk < kBK / 16; ++kk) tc_mma_bf16(d_tmem, da + 128u * kk, db + 2u * kk, idesc, acc | kk);
              release();
            }
          }
          __syncwarp();
          acc = 1;
          at.next(3 - ph, NS);
        }
        if (both || buf == 0) ++used0;
        if (both || buf == 1) ++used1;
      }
    }
  } else if (warp == 3) {
    if (rank == 0) {
      // =============================================================== takes the pair's tiles
      // Every pair takes one number that is past the last tile, so the launch takes n_work + n_pairs of them; who has the
      // highest sets the counter back.
      // (The fence: it is zero before this CTA ends, so before any successor starts.)
      auto set_back = [&]() {
        if (idx == n_work + n_pairs - 1) {
          atomicExch(&P.st->ffn_next, 0u);
          __threadfence();
        }
      };
      if (lane == 0) set_back();
      for (int q = 0; idx < n_work; ++q) {
        const int b = q & (kQueue - 1);
        if (!mbar_wait_warp(&sm.tile_ask, q & 1) || (q >= kQueue && !mbar_wait_warp(&sm.tile_empty[b], (q / kQueue - 1) & 1))) {
          if (lane == 0) flag_error(P.st, MOE_ERR_TIMEOUT, 0x417u);
          break;
        }
        if (lane == 0) idx = (int)atomicAdd(&P.st->ffn_next, 1u);
        idx = lane0(idx);
        if (idx < n_work) {
          const int ph = idx >= n_work1;
          t = decode_tile(P.ph[ph], ph ? 0 : P.cap, P.w_max, sm.map, lane, idx - (ph ? n_work1 : 0));
        }
        if (lane == 0) {
          hand_out(sm, b, idx, t);
          set_back();
        }
      }
    } else if (P.counts) {
      // =============================================================== slots of the (token, choice) pairs, for the combine
      __syncwarp();
      for (int p = pair * 32 + lane; p < P.n_pairs_tk; p += n_pairs * 32) {
        const int e = P.topk_idx[p];
        P.inv[p] = sm.map.lo[e >> 5][e & 31] + P.pos[p];
      }
    }
  } else {
    // ================================================================= epilogue (warps 4..19, both CTAs)
    const int q = warp & 3, part = (warp - 4) >> 2;  // quarter of the lanes it may read; every fourth 16-column chunk
    const uint32_t acce_bar[2] = {map_to_rank(&sm.accum_empty[0], 0u), map_to_rank(&sm.accum_empty[1], 0u)};
    unsigned char* const ebuf = epi_bufs + (warp - 4) * (kEpiBytesDP / kEpiWarpsDP);
    const uint32_t tile_bar = map_to_rank(&sm.tile_empty[0], 0u);
    int seen0 = 0, seen1 = 0;
    for (int seq = 0; next_tile(seq); ++seq) {
      const int ph = idx >= n_work1;
      const bool both = ph == 0 && !two;
      const int buf = both ? 0 : seq & 1, hb = P.ph[ph].hb, m_total = P.ph[ph].m_total;
      if (!mbar_wait_warp(&sm.accum_full[buf], (buf ? seen1 : seen0) & 1)) {
        if (lane == 0) flag_error(P.st, MOE_ERR_TIMEOUT, 0x412u);
        break;
      }
      if (buf) ++seen1; else ++seen0;
      // (the tile is in the lanes' registers; the producers and the issuer have had it before any of the tile's products)
      if (lane == 0 && seq > 0) mbar_arrive_cluster(tile_bar + 8u * (uint32_t)((seq - 1) & (kQueue - 1)));
      tc_fence_after();
      const int fb = t.f0 + (int)rank * hb + 32 * q;              // this warp's first feature,
      const int feats = min(min(hb - 32 * q, 32), m_total - fb);  // how many it has (a multiple of 8; <= 0: none)
      const int toks = feats > 0 ? t.toks : 0;
      const uint32_t tbase = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(buf * kAccCols);
      if (ph == 0) {
        __nv_bfloat16* out = P.hidden + (size_t)(t.s0 + 16 * part) * m_total + fb;
#pragma unroll 1
        for (int c = 16 * part; c < toks; c += 64, out += 64ll * m_total) {
          uint32_t g[16], u[16];
          tc_ld16(tbase + c, g);
          tc_ld16(tbase + acc1 + c, u);
          tc_wait_ld16(g, u);
          __syncwarp();  // (the buffer's last contents have been read)
#pragma unroll
          for (int j = 0; j < 8; ++j)
            put_tokens(ebuf, lane, 2 * j, silu_mul(__uint_as_float(g[2 * j]), __uint_as_float(u[2 * j])),
                       silu_mul(__uint_as_float(g[2 * j + 1]), __uint_as_float(u[2 * j + 1])));
          __syncwarp();
          send_tokens(ebuf, lane, out, m_total, toks - c, feats);
        }
      } else {
        // lane = feature: a token's 32 features leave as one line
        float* out = P.out + (size_t)t.ks * P.plane_elems + (size_t)(t.s0 + 16 * part) * m_total + fb + lane;
#pragma unroll 1
        for (int c = 16 * part; c < toks; c += 64, out += 64ll * m_total) {
          uint32_t a[16];
          tc_ld16(tbase + c, a);
          tc_wait_ld16(a);
          if (lane < feats) {
            float* dst = out;
#pragma unroll
            for (int j = 0; j < 16; ++j, dst += m_total)
              if (c + j < toks) *dst = __uint_as_float(a[j]);
          }
        }
      }
      // the accumulators are in registers / memory now: hand them back to the leader's MMA warp
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive_cluster(acce_bar[buf]);
        if (both) mbar_arrive_cluster(acce_bar[1]);
      }
      if (ph == 0) {
        fence_proxy_async_all();
        __syncwarp();
        if (lane == 0) red_add_release(&P.st->ffn_done[t.e], 1u);
      }
    }
  }
  // ---- teardown: every role gets here in bounded time; neither CTA leaves while the other may still count on
  // its barriers or read its operands
  tc_fence_before();
  __syncthreads();
  __syncwarp();
  cluster_sync_all();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kTmemCols) : "memory");
  }
  // the last CTA leaves the counters as the next call expects them
  if (warp == 0) {
    unsigned old = 0;
    if (lane == 0) old = atom_add_acq_rel(&P.st->ffn_exit, 1u);
    old = __shfl_sync(0xffffffffu, old, 0);
    if (old == gridDim.x - 1u) {
      for (int e = lane; e < MOE_MAX_EXPERTS; e += 32) P.st->ffn_done[e] = 0u, P.st->route_count[e] = 0u;
      if (lane == 0) P.st->ffn_exit = 0u;
    }
  }
}

// Token tiles of at most w tokens the routing will give, on average.
int token_tiles_expected(int n_slots, int E, int w) {
  return std::max((n_slots + w - 1) / w + (n_slots > E * w * 3 / 4 ? E / 2 : 0), std::min(E, n_slots));
}

// Cycles of one K step of a pair's tile of na matrices, hb features per CTA and n tokens: the tensor cores; shared memory (what
// is loaded, and what the MMAs read: 128 rows of weights and half of the tokens each); a round trip through the ring (about
// 2800 cycles from a slot's release to the use of its next contents), shared by the K steps it holds.
double step_cycles(int na, int hb, int n, int steps_in_ring) {
  const double mma = na * 2.0 * n, smem = (na * hb * 128.0 + n * 64.0 + na * 4.0 * (4096 + n * 16.0)) / 128.0;
  return std::max(std::max(mma, smem), 2800.0 / std::min(steps_in_ring, kSteps));
}
// ... and if every SM loads weights at the same time: its share of HBM (25.5 bytes per clock).
double hbm_cycles(int na, int hb, double tiles_per_weight) { return na * hb * 128.0 / 25.5 / tiles_per_weight; }

}  // namespace

// Decomposed experts with few pairs gain too little by it for E / k times the scratch.  Grouped and gathered -> placed, graph of 20
// calls, us: d 2048, r 128, 8 experts, 512 pairs 57.4 -> 57.5, 768 60.2 -> 60.2, 1024 62.9 -> 62.4, 2048 77.8 -> 77.0, 4096 101.8 -> 97.4;
// d 440, r 216: 384 45.6 -> 44.8, 1024 50.9 -> 49.4, 4096 63.9 -> 59.2; d 512, r 64, 16 experts: 512 40.8 -> 40.3, 1024 42.9 -> 41.3,
// 4096 53.9 -> 48.6.
int prefill_placed_tokens(const moe_config& c, int T) {
  const int t = (int)std::min<size_t>(T, kScatterBytesMax / ((size_t)c.n_experts * c.d_model * 2));
  return route_tile_applies(c, t) && (c.wd_rank == 0 || (long long)t * c.top_k >= 1024) ? t : 0;
}

int launch_dense_prefill(moe_ctx* ctx, int T, const moe_weights* w, const PrefillRows& rows, void* hidden, float* out_slots,
                         float* planes, int* out_planes, cudaStream_t s) {
  const moe_config& c = ctx->cfg;
  const int d = c.d_model, f = c.d_ff, E = c.n_experts, n_slots = T * c.top_k, pairs_all = ctx->sm_count / 2;
  const int active = std::min(E, n_slots), m = std::max(1, n_slots / E);
  DPParams P{};
  P.counts = rows.counts, P.offsets = rows.offsets, P.E = E, P.n_pairs_tk = n_slots, P.cap = rows.counts ? T : 0;
  P.topk_idx = rows.topk_idx, P.pos = rows.pos, P.inv = rows.inv;
  P.tb = m + m / 4 + 16 <= 192 ? 32 : 64;  // (32 rows: less read past an expert's tokens; 64: fewer loads to issue)
  P.likely = m, P.st = ctx->d_state;
  P.hidden = (__nv_bfloat16*)hidden, P.plane_elems = (long long)n_slots * d;
  // how the work is cut: the fewest cycles for the pair with the most, tiles of both phases being dealt out in turn
  // (a slot has 128 rows: an MMA reads as many of the weights, whatever hb is, and half of a tile's tokens are no more)
  const size_t fixed = kEpiBytesDP + sizeof(SmemDP) + 1024 + 128;
  const auto ring_slots = [&](int h) { return (int)((ctx->max_smem_optin - fixed) / ((size_t)h * kBK * 2)); };
  const int kb1 = (d + kBK - 1) / kBK, kb2 = (f + kBK - 1) / kBK;
  int hb1 = 0, ks2 = 1;
  const int hb2 = d > 128 ? 128 : 64;
  int last_nt = 0;
  double best = 0;
  // Tiles of up to 256 tokens: an expert with more than its share needs no further pass over its weights (512 tokens, d 1024, f 2816,
  // all at the same two of 8 experts: tiles as wide as an even share, 192, 45.6 us, 256 41.7; 1000 tokens, d 2048, f 5632, 2 of 16:
  // 133.9, 122.9).  Up to 128 where the contractions are short and the epilogue of a wide tile, in the open, weighs more (1900
  // tokens, d 304, f 904, 2 experts: 256 30.2 us, 128 27.4).
  for (const int w_max : {256, 128}) {
    const int nt = token_tiles_expected(n_slots, E, w_max), n = std::min(w_max, (n_slots / nt + 31) / 32 * 32), ns = ring_slots(128);
    if (nt == last_nt) break;  // (an even share fits into either: the same tiles)
    last_nt = nt;
    const double tpw = (double)nt / active;
    for (int h1 = 128; h1 >= 32; h1 -= 8) {
      const int n1 = nt * ((f + 2 * h1 - 1) / (2 * h1));
      // (a pair whose loads take longer than its neighbours' gets more of HBM: half of that term)
      const double c1 = kb1 * (step_cycles(2, h1, n, ns / 3) + 0.5 * hbm_cycles(2, h1, tpw)) + (n > 128 ? 4000 : 1500);
      for (int ks = 1; ks <= (n_slots <= kKSplitMaxSlots ? std::min(kKSplitMax, kb2) : 1); ++ks) {
        const int n2 = nt * ((d + 2 * hb2 - 1) / (2 * hb2)) * ks;
        const double c2 = (kb2 + ks - 1) / ks * (step_cycles(1, hb2, n, ns / 2) + 0.5 * hbm_cycles(1, hb2, tpw)) + 1500;
        const int q1 = n1 / pairs_all, r1 = n1 % pairs_all, q = (n1 + n2) / pairs_all, r = (n1 + n2) % pairs_all;
        const auto load = [&](int a, int all) { return a * c1 + (all - a) * c2; };
        double worst = std::max(load(q1, q), std::min(r1, r) > 0 ? load(q1 + 1, q + 1) : 0.0);
        if (r > r1) worst = std::max(worst, load(q1, q + 1));
        if (r1 > r) worst = std::max(worst, load(q1 + 1, q));
        worst = std::max(worst, (q1 + (r1 > 0)) * c1 + c2);  // (the last experts' second product starts when all of phase 1 is done)
        // a further plane of partial sums, written and read, in the epilogue and in the combine (wearable, 512 tokens: one plane 56.9
        // us, two 52.8, four 54.7; paper, 333 tokens: 74.7, 69.6, 74.8)
        worst += (ks - 1) * 16.0 * n_slots * d / 3800.0;
        if (hb1 == 0 || worst < 0.98 * best) best = worst, hb1 = h1, ks2 = ks, P.w_max = w_max;
      }
    }
  }
  P.ph[0] = DPPhase{d, kb1, f, hb1, 1, (f + 2 * hb1 - 1) / (2 * hb1)};
  P.ph[1] = DPPhase{f, kb2, d, hb2, ks2, (d + 2 * hb2 - 1) / (2 * hb2) * ks2};
  // the parts' planes are summed by the caller, or here (in the same order: the layer and its four calls give the same bits)
  P.out = ks2 > 1 && !out_planes ? planes : out_slots;
  CUtensorMap w1, x1, w2, x2;
  MOE_TRY(make_map_b(&w1, w->gud, d, 3, f, E, kBK, hb1));
  MOE_TRY(make_map_a(&x1, rows.x, P.cap ? (long long)E * T : n_slots, d, d, P.tb));
  MOE_TRY(make_map_b(&w2, w->gud, d, 3, f, E, 64, kBK));
  MOE_TRY(make_map_a(&x2, hidden, n_slots, f, f, P.tb));
  P.slot_bytes = 128 * kBK * 2;
  P.ring_slots = ring_slots(128);
  if (P.ring_slots < 6) return MOE_ERR_UNSUPPORTED;
  const size_t smem = (size_t)P.ring_slots * P.slot_bytes + fixed;
  MOE_TRY(allow_full_smem<dense_prefill_kernel>(ctx));
  const long long most = ((long long)(n_slots + P.w_max - 1) / P.w_max + E) * (P.ph[0].per_tok + P.ph[1].per_tok);
  const int pairs = (int)std::min<long long>(most, max_pairs<dense_prefill_kernel>(ctx, kThreadsDP, smem));
  cudaLaunchConfig_t lc;
  cudaLaunchAttribute attr[2];
  pair_launch_config(lc, attr, 2 * pairs, kThreadsDP, smem, s);
  MOE_CUDA_TRY(cudaLaunchKernelEx(&lc, dense_prefill_kernel, w1, x1, w2, x2, P));
  ctx->launches++;
  if (out_planes)
    *out_planes = ks2;
  else if (ks2 > 1)
    return launch_sum_planes(ctx, planes, P.plane_elems, ks2, out_slots, s);
  return MOE_OK;
}

}  // namespace cosmoe
