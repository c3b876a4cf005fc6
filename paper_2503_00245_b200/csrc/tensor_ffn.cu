// Prefill of weight-decomposed experts: grouped GEMMs on the 5th-generation tensor cores (dense experts: csrc/dense_prefill.cu).
//
// Tokens are grouped by expert (moe_permute), their rows gathered into a bf16 operand, and every expert's
// FFN becomes dense contractions  C[m, n] = sum_k A[m, k] * B_e[n, k]  over that expert's rows:
//
//   (1) T = X [gL | uL]   (2) H = silu(Tg gR) * (Tu uR)   (3) V = H dL   (4) O = V dR
//
// Two CTAs on neighbouring SMs (a cluster of 2) compute one tile of 256 rows x up to 256 columns with
// tcgen05.mma.cta_group::2: each CTA stages its own 128 rows of A and HALF of the tile's B rows, the tensor
// cores of the pair exchange the B halves, and each CTA ends up with the accumulators of its 128 rows
// (128 TMEM lanes x N columns).  Per flop a CTA moves half the B bytes into shared memory and reads a third
// fewer operand bytes out of it than a single CTA computing 256 x 256 on its own, and the tile takes 256 of the
// 512 TMEM columns, so the accumulators are double-buffered: the epilogue of tile i runs under the MMAs of
// tile i + 1.  Roles in each CTA:
//   warp 0     TMA producer: 64-wide K slices of A and B into a ring of shared-memory stages (128-byte swizzle);
//              both CTAs' copies complete on the LEADER's (rank 0) stage barrier;
//   warp 1     allocates tensor memory (both CTAs); in the leader one elected lane issues the MMAs for the pair
//              (M = 256, N <= 256, K = 16 per instruction) and commits to both CTAs' barriers;
//   warps 2-9  epilogue: tcgen05.ld the accumulators (one TMEM lane = one output row per thread), apply
//              SiLU * mul or nothing, convert, store the rows that belong to the expert.
// Tiles are handed out statically (pair p takes tiles p, p + pairs, ...): both CTAs of a pair derive the same
// sequence without talking to each other.
// Ragged groups: a tile may read rows of the next expert (or zeros past the end); they are never stored.
// K and N tails are zero-filled by TMA.  All waits are bounded; an expired wait sets the ctx's status word.
// No copy in this file uses cluster multicast: every CTA fetches what it needs with its own loads.
#include "tcgen.cuh"

namespace cosmoe {

namespace {

constexpr int kThreadsGG = (2 + kEpiWarps) * 32;
constexpr int kMaxStagesGG = 6;
constexpr int kEpiBuf = 4096;
constexpr int kPairRows = 2 * kBM;  // rows of a pair's tile

enum Epi { EPI_SWIGLU = 0, EPI_BF16_PAIR = 1, EPI_BF16 = 2, EPI_F32 = 3 };
// How the B operand of a tile is laid out and shared between the two CTAs of a pair (rank 0 / rank 1):
enum BMode {
  B_PAIR = 0,    // interleaved matrix, columns [0, bn) = sub-row 0 (rank 0 loads them), [bn, 2 bn) = sub-row 1 (rank 1)
  B_DUAL = 1,    // the same columns, but sub-row 1 meets a second A operand: two MMAs of N = bn, each rank loads half of both
  B_SINGLE = 2   // one sub-row: rank r loads rows [n0 + r bn/2, n0 + (r+1) bn/2)
};

struct GGParams {
  const unsigned* counts;  // [E] tokens of each expert, or null: ...
  const int32_t* offsets;  // ... [E+1] slot ranges
  int cap;                 // > 0: the rows of A are grouped at [e * cap ...] and not by slot
  const int32_t *topk_idx, *pos;  // with inv: the (token, choice) pairs' experts and places among their expert's tokens ...
  int32_t* inv;                   // ... from which their slots are worked out, by this launch
  int n_pairs_tk;
  int clear;                      // the last CTA clears the counts
  int E;
  int K;         // contraction length
  int n_total;   // output columns (per sub-row in B_PAIR / B_DUAL)
  int n_store;   // columns stored, >= n_total: the columns between are written as zeros (accumulators of B rows that do
                 // not exist), so that a consumer may read the padded width
  int bn;        // output columns per tile (per sub-row in B_PAIR / B_DUAL: <= 128; else <= 256)
  int bmode;
  int k_wrap;    // > 0: the B operand's k coordinate wraps at k_wrap (A = [hi | lo] halves of a split operand)
  int split;     // bf16 epilogues also store the rounding remainder: value = hi + lo, lo at column offset out_off_lo
  int epi;
  void* out;
  long long ld_out;    // elements
  long long out_off2;  // EPI_BF16_PAIR: column offset of the second half
  long long out_off_lo;  // split: column offset of the remainders
  int ksplit;             // the contraction is cut into this many parts, each a work item of its own ...
  long long plane_elems;  // ... writing its partial sums plane_elems further on in `out` (EPI_F32 only)
  int n_stages;
  DeviceState* st;
};

struct SmemGG {
  uint64_t full[kMaxStagesGG];   // leader's: both CTAs' operands of the stage have landed
  uint64_t empty[kMaxStagesGG];  // own: the MMAs have finished reading this CTA's stage
  uint64_t accum_full[2];        // own: all MMAs of the tile in accumulator buffer b have completed
  uint64_t accum_empty[2];       // leader's: the epilogue warps of both CTAs have read buffer b out of TMEM
  uint32_t tmem_base;
};

struct Tile {
  int e, m0, m_end, n0, ks;
  int a0;  // first row of A
};

// The experts' slot ranges and tiles, spread over a warp's lanes (lane l: experts l and l + 32).  Every warp keeps its own:
// nothing has to be published to the CTA between the dependency wait and the first load.
struct TileMap {
  int lo0, lo1, hi0, hi1;  // slots [lo, hi)
  int p0, p1;              // 256-row tiles of the experts up to and including this one
  int total;
};
__device__ __forceinline__ TileMap read_tile_map(const GGParams& P, int lane) {
  TileMap m;
  if (P.counts) {
    const int n0 = lane < P.E ? (int)__ldcg(P.counts + lane) : 0, n1 = lane + 32 < P.E ? (int)__ldcg(P.counts + lane + 32) : 0;
    m.hi0 = n0, m.hi1 = n1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v0 = __shfl_up_sync(0xffffffffu, m.hi0, o), v1 = __shfl_up_sync(0xffffffffu, m.hi1, o);
      if (lane >= o) m.hi0 += v0, m.hi1 += v1;
    }
    m.hi1 += __shfl_sync(0xffffffffu, m.hi0, 31);
    m.lo0 = m.hi0 - n0, m.lo1 = m.hi1 - n1;
  } else {
    const int e0 = min(lane, P.E), e1 = min(lane + 32, P.E);
    m.lo0 = P.offsets[e0], m.hi0 = P.offsets[min(e0 + 1, P.E)];
    m.lo1 = P.offsets[e1], m.hi1 = P.offsets[min(e1 + 1, P.E)];
  }
  m.p0 = (max(m.hi0 - m.lo0, 0) + kPairRows - 1) / kPairRows;
  m.p1 = (max(m.hi1 - m.lo1, 0) + kPairRows - 1) / kPairRows;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v0 = __shfl_up_sync(0xffffffffu, m.p0, o), v1 = __shfl_up_sync(0xffffffffu, m.p1, o);
    if (lane >= o) m.p0 += v0, m.p1 += v1;
  }
  m.p1 += __shfl_sync(0xffffffffu, m.p0, 31);
  m.total = __shfl_sync(0xffffffffu, m.p1, 31);
  return m;
}

// idx-th tile of this launch: row-tile major, column tile minor (pairs that run side by side share the A rows
// and sweep the expert's B columns, which then sit in L2 for the expert's other row tiles).  By a whole warp.
__device__ __forceinline__ Tile decode_tile(const GGParams& P, const TileMap& m, int idx, int n_tiles) {
  Tile t;
  const int per_row = n_tiles * P.ksplit;
  const int mt = idx / per_row, rem = idx - mt * per_row;
  const int nt = rem / P.ksplit;
  t.ks = rem - nt * P.ksplit;
  t.n0 = nt * P.bn;
  // the first expert whose tiles reach past mt (mt < total: there is one)
  const int e = __popc(__ballot_sync(0xffffffffu, m.p0 <= mt)) + __popc(__ballot_sync(0xffffffffu, m.p1 <= mt));
  const int before0 = __shfl_sync(0xffffffffu, m.p0, (e - 1) & 31), before1 = __shfl_sync(0xffffffffu, m.p1, (e - 1) & 31);
  const int lo0 = __shfl_sync(0xffffffffu, m.lo0, e & 31), lo1 = __shfl_sync(0xffffffffu, m.lo1, e & 31);
  const int hi0 = __shfl_sync(0xffffffffu, m.hi0, e & 31), hi1 = __shfl_sync(0xffffffffu, m.hi1, e & 31);
  const int before = e == 0 ? 0 : e <= 32 ? before0 : before1;
  t.e = e;
  t.m0 = (e < 32 ? lo0 : lo1) + (mt - before) * kPairRows;
  t.m_end = e < 32 ? hi0 : hi1;
  t.a0 = P.cap > 0 ? e * P.cap + (mt - before) * kPairRows : t.m0;
  return t;
}


// 64 bytes of each of 32 rows from a warp's registers (lane = row) to memory, through 2 KB of shared memory: a store of
// the accumulator layout as it is touches 32 lines with 16 bytes each; this one writes 8 rows' 64 bytes per instruction.
// (16-byte pieces are swapped by row pair, so that neither side meets a bank conflict.)  rows: valid rows; pieces: valid
// 16-byte pieces of a row.
__device__ __forceinline__ void store_rows(unsigned char* buf, int lane, const uint32_t* v, void* dst, long long ld_bytes,
                                           int rows, int pieces) {
  __syncwarp();  // (the buffer's last contents have been read)
#pragma unroll
  for (int i = 0; i < 4; ++i)
    *reinterpret_cast<uint4*>(buf + lane * 64 + ((i ^ ((lane >> 1) & 3)) << 4)) =
        make_uint4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
  __syncwarp();
  const int piece = lane & 3;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = (lane >> 2) + 8 * i;
    if (r < rows && piece < pieces)
      *reinterpret_cast<uint4*>((unsigned char*)dst + (long long)r * ld_bytes + piece * 16) =
          *reinterpret_cast<const uint4*>(buf + r * 64 + ((piece ^ ((r >> 1) & 3)) << 4));
  }
}
// (phone WD r = 128, T = 2048: the layer 163.7 -> 151.2 us; wearable T = 512: 61.6 -> 60.3.)
// The same for 128 bytes of each row: 4 whole lines per instruction.
__device__ __forceinline__ void store_rows128(unsigned char* buf, int lane, const uint32_t* v, void* dst, long long ld_bytes,
                                              int rows, int pieces) {
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 8; ++i)
    *reinterpret_cast<uint4*>(buf + lane * 128 + ((i ^ (lane & 7)) << 4)) =
        make_uint4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
  __syncwarp();
  const int piece = lane & 7;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = (lane >> 3) + 4 * i;
    if (r < rows && piece < pieces)
      *reinterpret_cast<uint4*>((unsigned char*)dst + (long long)r * ld_bytes + piece * 16) =
          *reinterpret_cast<const uint4*>(buf + r * 128 + ((piece ^ (r & 7)) << 4));
  }
}
// 32 fp32 columns rounded to bf16; lo_off > 0: the rounding remainders too, lo_off columns further on
__device__ __forceinline__ void store_bf16(unsigned char* buf, int lane, const uint32_t* a, __nv_bfloat16* dst, long long ld_bytes,
                                           int rows, int pieces, long long lo_off) {
  uint32_t o[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) o[j] = pack_bf16x2(__uint_as_float(a[2 * j]), __uint_as_float(a[2 * j + 1]));
  store_rows(buf, lane, o, dst, ld_bytes, rows, pieces);
  if (lo_off > 0) {
    uint32_t l[16];
#pragma unroll
    for (int j = 0; j < 16; ++j)
      l[j] = pack_bf16x2(__uint_as_float(a[2 * j]) - __uint_as_float(o[j] << 16),
                         __uint_as_float(a[2 * j + 1]) - __uint_as_float(o[j] & 0xffff0000u));
    store_rows(buf, lane, l, dst + lo_off, ld_bytes, rows, pieces);
  }
}

__global__ void __launch_bounds__(kThreadsGG, 1)
    grouped_gemm_kernel(const __grid_constant__ CUtensorMap map_a0, const __grid_constant__ CUtensorMap map_a1,
                        const __grid_constant__ CUtensorMap map_b, const GGParams P) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  // stage layout: [A 16 KB][A' 16 KB, B_DUAL only][B <= 16 KB], all 1024-byte aligned (swizzle atoms); identical
  // in both CTAs, because the MMA addresses the pair's operands by one shared-memory offset
  const uint32_t a_bytes = kBM * kBK * 2;
  const uint32_t n_a = P.bmode == B_DUAL ? 2u : 1u;
  const uint32_t b_rows = (P.bmode == B_PAIR || P.bmode == B_DUAL) ? (uint32_t)P.bn : (uint32_t)P.bn / 2u;  // per CTA
  const uint32_t b_bytes = b_rows * kBK * 2;
  const uint32_t stage_bytes = n_a * a_bytes + 128u * kBK * 2u;
  unsigned char* stages = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char* const epi_bufs = stages + (size_t)P.n_stages * stage_bytes;  // kEpiBuf per epilogue warp
  SmemGG& sm = *reinterpret_cast<SmemGG*>(epi_bufs + kEpiWarps * kEpiBuf);
  const int tid = threadIdx.x, lane = tid & 31, warp = lane0(tid >> 5);
  const int NS = P.n_stages;
  const int num_kb = (P.K + kBK - 1) / kBK;
  const int n_tiles = (P.n_total + P.bn - 1) / P.bn;
  const uint32_t rank = (uint32_t)lane0((int)cluster_ctarank());
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;

  pdl_launch_dependents();
  if (tid == 0) {
    for (int i = 0; i < NS; ++i) {
      mbar_init(&sm.full[i], 1);
      mbar_init(&sm.empty[i], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&sm.accum_full[b], 1);
      mbar_init(&sm.accum_empty[b], 2 * kEpiWarps);
    }
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_a0) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_b) : "memory");
    fence_mbar_init();
    fence_proxy_async_smem();
  }
  if (warp == 1) {  // one warp of each CTA of the pair
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sm.tmem_base)),
                 "n"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  __syncwarp();
  cluster_sync_all();  // the other CTA's barriers are initialised before anything is counted on them
  tc_fence_after();
  const uint32_t tmem = (uint32_t)lane0((int)sm.tmem_base);
  // everything above touches only this CTA's shared memory and TMEM; the expert offsets and the operands may
  // come from the kernel before
  pdl_wait();
  const TileMap tm = read_tile_map(P, lane);
  const int n_work = tm.total * n_tiles * P.ksplit;

  if (warp == 0) {
    // ================================================================= TMA producer (both CTAs)
    int it = 0;                  // k-blocks issued so far, over all tiles
    uint32_t slot = 0, par = 1;  // ring position; parity of the `empty` phase the slot's next fill waits for
    bool ok = true;
    const uint32_t tx_pair = 2u * (n_a * a_bytes + b_bytes);  // bytes both CTAs bring in per stage
    const uint32_t full0 = (uint32_t)lane0((int)map_to_rank(&sm.full[0], 0u));  // the leader's stage barriers, 8 bytes apart
    const int half_bn = P.bn / 2;
    const uint32_t st0 = (uint32_t)lane0((int)smem_u32(stages));
    for (int idx = pair; ok && idx < n_work; idx += n_pairs) {
      const Tile t = decode_tile(P, tm, idx, n_tiles);
      const int n0 = t.n0;
      const int kb0 = t.ks * num_kb / P.ksplit, kb1 = (t.ks + 1) * num_kb / P.ksplit;
      const int a_row = t.a0 + (int)rank * kBM;
      int k0 = kb0 * kBK;
      int kB = P.k_wrap > 0 ? k0 % P.k_wrap : k0;
      for (int kb = kb0; kb < kb1; ++kb, ++it) {
        if (it >= NS && !mbar_wait_warp(&sm.empty[slot], par)) {
          if (lane == 0) flag_error(P.st, MOE_ERR_TIMEOUT, 0x400u);
          ok = false;
          break;
        }
        const uint32_t st_a0 = st0 + slot * stage_bytes, st_b = st_a0 + n_a * a_bytes;
        const uint32_t bar = full0 + 8u * slot;
        if (elect_one()) {
          if (rank == 0) mbar_arrive_expect_tx(&sm.full[slot], tx_pair);
          tma_load_2d(st_a0, &map_a0, k0, a_row, bar);
          if (P.bmode == B_PAIR) {
            tma_load_4d(st_b, &map_b, kB, (int)rank, n0, t.e, bar);
          } else if (P.bmode == B_DUAL) {
            const int nr = n0 + (int)rank * half_bn;
            tma_load_2d(st_a0 + a_bytes, &map_a1, k0, a_row, bar);
            tma_load_4d(st_b, &map_b, kB, 0, nr, t.e, bar);
            tma_load_4d(st_b + (uint32_t)half_bn * kBK * 2, &map_b, kB, 1, nr, t.e, bar);
          } else {
            tma_load_4d(st_b, &map_b, kB, 0, n0 + (int)rank * half_bn, t.e, bar);
          }
        }
        __syncwarp();
        k0 += kBK, kB += kBK;
        if (P.k_wrap > 0 && kB >= P.k_wrap) kB -= P.k_wrap;
        if (++slot == (uint32_t)NS) slot = 0, par ^= 1u;
      }
    }
    if (!ok && rank == 0) {  // copies in flight (both CTAs' complete on these barriers) must land before the pair goes away
      for (int j = max(0, it - NS); j < it; ++j) (void)mbar_wait(&sm.full[j % NS], (j / NS) & 1);
    }
  } else if (warp == 1) {
    // ================================================================= MMA issuer (leader CTA only)
    if (rank == 0) {
      // One warp feeds the tensor cores of both SMs, so its instruction stream is kept short: the ring position
      // is a counter, not a division, and the operand descriptors are a constant high word plus a low word that
      // steps through the stage (32 bytes per 16 k-values).
      const int n_mma = P.bmode == B_PAIR ? 2 * P.bn : P.bn;
      const uint32_t idesc = instr_desc(n_mma, false);
      const uint64_t hi_k = smem_desc(0, 16, 1024) & 0xffffffff00000000ull;
      const uint32_t stage0 = (uint32_t)lane0((int)(smem_u32(stages) >> 4)), stage_step = stage_bytes >> 4;
      const uint32_t b_off = (n_a * a_bytes) >> 4, a1_off = a_bytes >> 4, b1_off = ((uint32_t)(P.bn / 2) * kBK * 2) >> 4;
      uint32_t slot = 0, par = 0, st_lo = stage0;
      int tile_i = 0;
      bool ok = true;
      for (int idx = pair; ok && idx < n_work; idx += n_pairs, ++tile_i) {
        const int buf = tile_i & 1;
        if (tile_i >= 2) {  // the accumulators two tiles back must have left this buffer, in both CTAs
          if (!mbar_wait_warp(&sm.accum_empty[buf], ((tile_i >> 1) - 1) & 1)) {
            if (lane == 0) flag_error(P.st, MOE_ERR_TIMEOUT, 0x403u);
            break;
          }
          tc_fence_after();
        }
        const uint32_t d_tmem = tmem + (uint32_t)(buf * kAccCols);
        const int ks = idx % P.ksplit;
        const int kb0 = ks * num_kb / P.ksplit, kb1 = (ks + 1) * num_kb / P.ksplit;
        uint32_t acc = 0;
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait_warp(&sm.full[slot], par)) {
            if (lane == 0) flag_error(P.st, MOE_ERR_TIMEOUT, 0x401u);
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t da = hi_k | (uint64_t)(st_lo | (1u << 16));
          const uint64_t db = hi_k | (uint64_t)((st_lo + b_off) | (1u << 16));
          if (elect_one()) {
            if (P.bmode == B_DUAL) {
              const uint64_t da1 = da + a1_off, db1 = db + b1_off;
#pragma unroll
              for (uint32_t kk = 0; kk < kBK / 16; ++kk) {
                tc_mma_bf16(d_tmem, da + 2u * kk, db + 2u * kk, idesc, acc | kk);
                tc_mma_bf16(d_tmem + (uint32_t)P.bn, da1 + 2u * kk, db1 + 2u * kk, idesc, acc | kk);
              }
            } else {
#pragma unroll
              for (uint32_t kk = 0; kk < kBK / 16; ++kk) tc_mma_bf16(d_tmem, da + 2u * kk, db + 2u * kk, idesc, acc | kk);
            }
            tc_commit_pair(&sm.empty[slot]);  // both CTAs' producers may refill the stage once these MMAs have read it
            if (kb + 1 == kb1) tc_commit_pair(&sm.accum_full[buf]);
          }
          __syncwarp();
          acc = 1;
          st_lo += stage_step;
          if (++slot == (uint32_t)NS) slot = 0, par ^= 1u, st_lo = stage0;
        }
      }
    } else if (P.inv) {  // slots of the (token, choice) pairs, for the combine
      for (int p0 = pair * 32; p0 < P.n_pairs_tk; p0 += n_pairs * 32) {
        const int p = min(p0 + lane, P.n_pairs_tk - 1), e = P.topk_idx[p];
        const int a = __shfl_sync(0xffffffffu, tm.lo0, e & 31), b = __shfl_sync(0xffffffffu, tm.lo1, e & 31);
        P.inv[p] = (e < 32 ? a : b) + P.pos[p];
      }
    }
  } else {
    // ================================================================= epilogue (warps 2..9, both CTAs)
    const int q = warp & 3;  // TMEM lanes 32q .. 32q+31 are the only ones this warp may read
    const int cpar = (warp - 2) >> 2;  // which of the two warps of this quarter: it takes every other 32-column chunk
    const uint32_t acce_bar[2] = {map_to_rank(&sm.accum_empty[0], 0u), map_to_rank(&sm.accum_empty[1], 0u)};
    unsigned char* const ebuf = epi_bufs + (warp - 2) * kEpiBuf;
    int tile_i = 0;
    for (int idx = pair; idx < n_work; idx += n_pairs, ++tile_i) {
      const Tile t = decode_tile(P, tm, idx, n_tiles);
      const int buf = tile_i & 1;
      if (!mbar_wait_warp(&sm.accum_full[buf], (tile_i >> 1) & 1)) {
        if (lane == 0) flag_error(P.st, MOE_ERR_TIMEOUT, 0x402u);
        break;
      }
      tc_fence_after();
      const int ncols = min(P.bn, P.n_store - t.n0);  // columns of this tile to store (multiple of 8)
      const int row = t.m0 + (int)rank * kBM + 32 * q + lane;
      const int rows = t.m_end - (row - lane);  // rows of this warp's 32 that belong to the expert (<= 0: none)
      const uint32_t tbase = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(buf * kAccCols);
      const size_t row0 = (size_t)(row - lane);
      if (P.epi == EPI_SWIGLU || P.epi == EPI_BF16_PAIR) {
        __nv_bfloat16* out = (__nv_bfloat16*)P.out + row0 * P.ld_out + t.n0;
        for (int c = 32 * cpar; c < P.bn; c += 64) {
          uint32_t g[32], u[32];
          tc_ld32(tbase + c, g);
          tc_ld32(tbase + P.bn + c, u);
          tc_wait_ld(g, u);
          const int pieces = (ncols - c) / 8;  // of 16 bytes
          uint32_t o[16];
          if (P.epi == EPI_SWIGLU) {
#pragma unroll
            for (int j = 0; j < 16; ++j)
              o[j] = pack_bf16x2(silu_mul(__uint_as_float(g[2 * j]), __uint_as_float(u[2 * j])),
                                 silu_mul(__uint_as_float(g[2 * j + 1]), __uint_as_float(u[2 * j + 1])));
            store_rows(ebuf, lane, o, out + c, P.ld_out * 2, rows, pieces);
          } else {
            store_bf16(ebuf, lane, g, out + c, P.ld_out * 2, rows, pieces, P.split ? P.out_off_lo : 0);
            store_bf16(ebuf, lane, u, out + P.out_off2 + c, P.ld_out * 2, rows, pieces, P.split ? P.out_off_lo : 0);
          }
        }
      } else {
        if (P.epi == EPI_F32) {
          float* out = (float*)P.out + (size_t)t.ks * P.plane_elems + row0 * P.ld_out + t.n0;
          uint32_t a[2][32];  // the next chunk's columns are fetched while this one's leave
          if (32 * cpar < P.bn) tc_ld32(tbase + 32 * cpar, a[0]);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int c = 32 * cpar + 64 * i;
            if (c < P.bn) {
              tc_wait_ld(a[i & 1]);
              if (c + 64 < P.bn) tc_ld32(tbase + c + 64, a[(i + 1) & 1]);
              store_rows128(ebuf, lane, a[i & 1], out + c, P.ld_out * 4, rows, (ncols - c) / 4);
            }
          }
        } else {
          for (int c = 32 * cpar; c < P.bn; c += 64) {
            uint32_t a[32];
            tc_ld32(tbase + c, a);
            tc_wait_ld(a);
            store_bf16(ebuf, lane, a, (__nv_bfloat16*)P.out + row0 * P.ld_out + t.n0 + c, P.ld_out * 2, rows, (ncols - c) / 8,
                       P.split ? P.out_off_lo : 0);
          }
        }
      }
      // the accumulators are in registers / memory now: hand the buffer back to the leader's MMA thread
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(acce_bar[buf]);
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
  if (P.clear && warp == 0) {  // the last CTA leaves the counts as the next call's router expects them
    unsigned old = 0;
    if (lane == 0) old = atom_add_acq_rel(&P.st->ffn_exit, 1u);
    old = __shfl_sync(0xffffffffu, old, 0);
    if (old == gridDim.x - 1u) {
      for (int e = lane; e < MOE_MAX_EXPERTS; e += 32) P.st->route_count[e] = 0u;
      if (lane == 0) P.st->ffn_exit = 0u;
    }
  }
}

int launch_gg(moe_ctx* ctx, const CUtensorMap& a0, const CUtensorMap& a1, const CUtensorMap& b, GGParams P,
              int n_slots, cudaStream_t s) {
  const moe_config& c = ctx->cfg;
  P.E = c.n_experts;
  P.st = ctx->d_state;
  if (P.n_store < P.n_total) P.n_store = P.n_total;
  if (P.ksplit < 1) P.ksplit = 1;
  const int n_tiles = (P.n_total + P.bn - 1) / P.bn;
  const size_t stage_bytes = (size_t)kBM * kBK * 2 * (P.bmode == B_DUAL ? 2 : 1) + 128 * kBK * 2;
  P.n_stages = P.bmode == B_DUAL ? 4 : kMaxStagesGG;
  const size_t smem = P.n_stages * stage_bytes + kEpiWarps * kEpiBuf + sizeof(SmemGG) + 1024 + 128;
  if ((long long)smem > ctx->max_smem_optin) return MOE_ERR_UNSUPPORTED;
  MOE_TRY(allow_full_smem<grouped_gemm_kernel>(ctx));
  const long long m_tiles = (n_slots + kPairRows - 1) / kPairRows + c.n_experts;  // upper bound
  const int pairs = (int)std::min<long long>(m_tiles * n_tiles * P.ksplit, max_pairs<grouped_gemm_kernel>(ctx, kThreadsGG, smem));
  cudaLaunchConfig_t lc;
  cudaLaunchAttribute attr[2];
  pair_launch_config(lc, attr, 2 * pairs, kThreadsGG, smem, s);
  MOE_CUDA_TRY(cudaLaunchKernelEx(&lc, grouped_gemm_kernel, a0, a1, b, P));
  ctx->launches++;
  return MOE_OK;
}

// Output columns per tile: the largest of 64, 128, ... `cap` that is not mostly padding.
int pick_bn(int n_total, int cap) {
  int bn = cap;
  while (bn > 64 && bn / 2 >= n_total) bn /= 2;
  return bn;
}

// 256-row tiles the routing will give, on average: every expert's last one is half full, and no expert has less than one.
int row_tiles(int n_slots, int E) {
  return std::max((n_slots + kPairRows - 1) / kPairRows + E / 2, std::min(E, n_slots));
}
// Parts to cut a contraction of num_kb K steps into, for the fewest rounds of steps over the pairs; a further part (a
// plane of partial sums, written and read once more) has to save 1/8.
int pick_ksplit(long long tiles, int num_kb, int pairs, int most) {
  int ks = 1;
  long long best = (tiles + pairs - 1) / pairs * num_kb;
  for (int c = 2; c <= std::min(most, num_kb); ++c) {
    const long long steps = (tiles * c + pairs - 1) / pairs * ((num_kb + c - 1) / c);
    if (8 * steps <= 7 * best) best = steps, ks = c;
  }
  return ks;
}

}  // namespace

int make_map_rows(CUtensorMap* m, const void* base, long long inner, int nsub, long long rows, int slots, int box_inner,
                  int box_rows) {
  return make_map_b(m, base, inner, nsub, rows, slots, box_inner, box_rows, CU_TENSOR_MAP_SWIZZLE_NONE);
}

int launch_prefill_ffn(moe_ctx* ctx, int T, const moe_weights* w, const PrefillRows& rows, char* ws, const WsLayout& L,
                       float* out_slots, int* out_planes, cudaStream_t s) {
  const moe_config& c = ctx->cfg;
  if (w->expert_slot) return MOE_ERR_UNSUPPORTED;  // the tensor path reads experts in place (slot == expert)
  const int d = c.d_model, f = c.d_ff, r = c.wd_rank, E = c.n_experts;
  const int n_slots = T * c.top_k;
  if (out_planes) *out_planes = 1;
  if (r == 0) return launch_dense_prefill(ctx, T, w, rows, ws + L.hidden, out_slots, (float*)(ws + L.out_slots), out_planes, s);
  void* xperm = ws + L.xperm;
  void* hidden = ws + L.hidden;
  int rc;
  CUtensorMap ma, ma1, mb;
  GGParams P{};
  P.counts = rows.counts, P.offsets = rows.offsets;
  // The rank-r intermediates t and v are kept as hi + lo pairs of bf16 (value = hi + lo): the GEMMs that
  // consume them run over K = 2 * rp with the weight slices repeated, so the intermediates carry ~16 mantissa
  // bits and the chain's only bf16 roundings are those of the dense path (hidden activations, output).
  // rp = r rounded up to the K step: the columns [r, rp) of an intermediate are stored as zeros and meet
  // weight rows past the end of the matrix (zero-filled by the loads), so any rank that is a multiple of 8 works.
  const int rp = (r + kBK - 1) / kBK * kBK;
  const int tw = 2 * rp;  // stored width of one intermediate: hi | lo
  void* mid_a = ws + L.mid_a;  // [n_slots][2*tw]: t_g (hi | lo) | t_u (hi | lo)
  void* mid_b = ws + L.mid_b;  // [n_slots][tw]:   v (hi | lo)
  // (1) T = X [gL | uL]
  if ((rc = make_map_a(&ma, rows.x, rows.counts ? (long long)E * T : n_slots, d, d)) != MOE_OK) return rc;
  const int pairs = ctx->sm_count / 2, m_tiles = row_tiles(n_slots, E);
  P.bn = pick_bn(r, 128);
  while (P.bn > 64 && 2 * m_tiles * ((r + P.bn - 1) / P.bn) <= pairs) P.bn /= 2;  // a small rank leaves pairs idle: narrower tiles
  if ((rc = make_map_b(&mb, w->wd_a, d, 2, r, E, kBK, P.bn)) != MOE_OK) return rc;
  P.K = d, P.n_total = r, P.bmode = B_PAIR, P.epi = EPI_BF16_PAIR;
  P.k_wrap = 0, P.split = 1, P.out = mid_a, P.ld_out = 2 * tw, P.out_off2 = tw, P.out_off_lo = rp, P.n_store = rp;
  if (rows.counts) P.cap = T, P.topk_idx = rows.topk_idx, P.pos = rows.pos, P.inv = rows.inv, P.n_pairs_tk = n_slots;
  if ((rc = launch_gg(ctx, ma, ma, mb, P, n_slots, s)) != MOE_OK) return rc;
  P.cap = 0, P.inv = nullptr;
  // (2) hidden = silu(Tg gR) * (Tu uR): two A operands, each CTA brings half of the gate and half of the up rows
  if ((rc = make_map_a(&ma, mid_a, n_slots, tw, 2 * tw)) != MOE_OK) return rc;
  if ((rc = make_map_a(&ma1, (const __nv_bfloat16*)mid_a + tw, n_slots, tw, 2 * tw)) != MOE_OK) return rc;
  if ((rc = make_map_b(&mb, w->wd_b, r, 2, f, E, kBK, 64)) != MOE_OK) return rc;
  P.K = tw, P.n_total = f, P.bn = 128, P.bmode = B_DUAL, P.epi = EPI_SWIGLU;
  P.k_wrap = rp, P.split = 0, P.out = hidden, P.ld_out = f, P.out_off2 = 0, P.out_off_lo = 0, P.n_store = 0;
  if ((rc = launch_gg(ctx, ma, ma1, mb, P, n_slots, s)) != MOE_OK) return rc;
  // (3) V = hidden dL
  if ((rc = make_map_a(&ma, hidden, n_slots, f, f)) != MOE_OK) return rc;
  P.bn = pick_bn(r, 256);
  if ((rc = make_map_b(&mb, w->wd_c, f, 1, r, E, kBK, P.bn / 2)) != MOE_OK) return rc;
  P.K = f, P.n_total = r, P.bmode = B_SINGLE, P.epi = EPI_BF16;
  P.k_wrap = 0, P.split = 1, P.out = mid_b, P.ld_out = tw, P.out_off2 = 0, P.out_off_lo = rp, P.n_store = rp;
  // few tiles of a long contraction: cut into parts whose fp32 sums (in the gathered rows' place, which are not needed any
  // more) are added, in order, and split by a kernel of their own.  r 128, 2048 tokens: 20 tiles on 74 pairs, 37 us.
  const int planes_fit = d / (2 * rp);
  const int ks = pick_ksplit((long long)m_tiles * ((r + P.bn - 1) / P.bn), (f + kBK - 1) / kBK, pairs, std::min(kKSplitMax, planes_fit));
  if (ks > 1) {
    P.epi = EPI_F32, P.split = 0, P.out = xperm, P.ld_out = rp, P.ksplit = ks, P.plane_elems = (long long)n_slots * rp;
    if ((rc = launch_gg(ctx, ma, ma, mb, P, n_slots, s)) != MOE_OK) return rc;
    P.ksplit = 1, P.plane_elems = 0;
    if ((rc = launch_split_planes(ctx, (const float*)xperm, n_slots, rp, ks, mid_b, s)) != MOE_OK) return rc;
  } else if ((rc = launch_gg(ctx, ma, ma, mb, P, n_slots, s)) != MOE_OK) {
    return rc;
  }
  // (4) out_slots = V dR
  if ((rc = make_map_a(&ma, mid_b, n_slots, tw, tw)) != MOE_OK) return rc;
  P.bn = pick_bn(d, 256);
  if ((rc = make_map_b(&mb, w->wd_d, r, 1, d, E, kBK, P.bn / 2)) != MOE_OK) return rc;
  P.K = tw, P.n_total = d, P.bmode = B_SINGLE, P.epi = EPI_F32;
  P.k_wrap = rp, P.split = 0, P.out = out_slots, P.ld_out = d, P.out_off2 = 0, P.out_off_lo = 0, P.n_store = 0;
  P.clear = rows.counts != nullptr;
  return launch_gg(ctx, ma, ma, mb, P, n_slots, s);
}

}  // namespace cosmoe
