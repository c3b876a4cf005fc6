// Tensor-core (prefill) path of the expert FFN: grouped GEMMs on the 5th-generation tensor cores.
//
// Tokens are grouped by expert (moe_permute), their rows gathered into a bf16 operand, and every expert's
// FFN becomes dense contractions  C[m, n] = sum_k A[m, k] * B_e[n, k]  over that expert's rows:
//
//   dense experts  (1) H = silu(X Wg) * (X Wu)   A = gathered x,  B = gate / up rows of gud   -> bf16 hidden
//                  (2) O = H Wd                  A = H,           B = down rows of gud (N-major) -> fp32 slots
//   Eq. 1 factors  (1) T = X [gL | uL]   (2) H = silu(Tg gR) * (Tu uR)   (3) V = H dL   (4) O = V dR
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
#include <cuda.h>

#include <algorithm>

#include "common.cuh"

namespace cosmoe {

namespace {

constexpr int kBM = 128;  // rows per CTA and tile (TMEM lanes)
constexpr int kBK = 64;   // K elements per stage (128 bytes of bf16 = one swizzle row)
constexpr int kEpiWarps = 8;  // two per quarter of the TMEM lanes, splitting the columns
constexpr int kThreadsGG = (2 + kEpiWarps) * 32;
constexpr int kTmemCols = 512;  // two accumulator buffers of 256 columns
constexpr int kAccCols = 256;
constexpr int kMaxStagesGG = 6;
constexpr int kEpiBuf = 4096;
constexpr int kPairRows = 2 * kBM;  // rows of a pair's tile

enum Epi { EPI_SWIGLU = 0, EPI_BF16_PAIR = 1, EPI_BF16 = 2, EPI_F32 = 3 };
// How the B operand of a tile is laid out and shared between the two CTAs of a pair (rank 0 / rank 1):
enum BMode {
  B_PAIR = 0,    // interleaved matrix, columns [0, bn) = sub-row 0 (rank 0 loads them), [bn, 2 bn) = sub-row 1 (rank 1)
  B_DUAL = 1,    // the same columns, but sub-row 1 meets a second A operand: two MMAs of N = bn, each rank loads half of both
  B_SINGLE = 2,  // one sub-row, K-major: rank r loads rows [n0 + r bn/2, n0 + (r+1) bn/2)
  B_NMAJOR = 3   // one sub-row stored [k][n] (the down rows of gud): rank r loads its bn/2 columns in 64-column boxes
};

struct GGParams {
  const int32_t* offsets;  // [E+1] slot ranges per expert
  int E;
  int K;         // contraction length
  int n_total;   // output columns (per sub-row in B_PAIR / B_DUAL)
  int n_store;   // columns stored, >= n_total: the columns between are written as zeros (accumulators of B rows that do
                 // not exist), so that a consumer may read the padded width
  int bn;        // output columns per tile (per sub-row in B_PAIR / B_DUAL: <= 128; else <= 256)
  int bmode;
  int b_sub;     // sub-row of the interleaved matrix that B_SINGLE / B_NMAJOR tiles read
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

// ---- PTX wrappers ------------------------------------------------------------------------------------
// Tiled loads whose completion may be counted on a barrier of the other CTA of the pair (cta_group::2); the
// data always lands in the issuing CTA's own shared memory.
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int c0, int c1, uint32_t bar_cluster) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
      "[%4];" ::"r"(smem_u32(dst)),
      "l"(map), "r"(c0), "r"(c1), "r"(bar_cluster)
      : "memory");
}
__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                            uint32_t bar_cluster) {
  asm volatile(
      "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
      "%5}], [%6];" ::"r"(smem_u32(dst)),
      "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar_cluster)
      : "memory");
}
// One lane of a converged warp.  The loops that issue loads and MMAs are run by the whole warp, with loop bounds and
// coordinates taken from lane 0, and only the issuing itself is one lane's: the operands of these instructions live in
// registers that a warp shares, and inside a branch that one lane takes every operand of every instruction has to be
// moved there first -- about 100 cycles for each load and MMA.
// (A K step of the phone-shape GEMM: 720 -> 630 cycles, of which the tensor pipe needs 512; the layer 365 -> 349 us.)
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ int lane0(int v) { return __shfl_sync(0xffffffffu, v, 0); }
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// address of the same shared-memory object in CTA `rank` of this cluster
__device__ __forceinline__ uint32_t map_to_rank(const void* smem_ptr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(smem_ptr)), "r"(rank));
  return r;
}
// (Release at CTA scope: what the arrival hands over are tensor-memory columns, ordered by tcgen05.wait::ld and the tcgen05
// fence.  A release at cluster scope also waits for the warp's stores to memory, about a microsecond per tile.)
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar_cluster) {
  asm volatile("mbarrier.arrive.release.cta.shared::cluster.b64 _, [%0];" ::"r"(bar_cluster) : "memory");
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// The barrier at this shared-memory offset gets one arrival IN BOTH CTAs of the pair when every MMA this thread
// has issued so far has completed.  (A multicast of barrier arrivals, not of data: no copy in this file is multicast.)
__device__ __forceinline__ void tc_commit_pair(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
                   smem_u32(bar)),
               "h"((unsigned short)3)
               : "memory");
}
// `acc` == 0: the product overwrites the accumulator; otherwise it is added.
__device__ __forceinline__ void tc_mma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void tc_ld32(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
        "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr)
      : "memory");
}
// A load's registers may be read behind the wait only; going through it ties every use and copy of them to that place.
__device__ __forceinline__ void tc_wait_ld(uint32_t* v) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
      : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
        "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]),
        "+r"(v[16]), "+r"(v[17]), "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]), "+r"(v[22]), "+r"(v[23]),
        "+r"(v[24]), "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]), "+r"(v[29]), "+r"(v[30]), "+r"(v[31])
      :
      : "memory");
}
__device__ __forceinline__ void tc_wait_ld(uint32_t* a, uint32_t* v) {  // two loads, one wait
  tc_wait_ld(a);
  asm volatile(""
      : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
        "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]),
        "+r"(v[16]), "+r"(v[17]), "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]), "+r"(v[22]), "+r"(v[23]),
        "+r"(v[24]), "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]), "+r"(v[29]), "+r"(v[30]), "+r"(v[31]));
}

// Shared-memory operand descriptor (128-byte swizzle).  K-major tiles: rows of 128 bytes, 8-row groups 1024
// bytes apart (stride byte offset), the leading offset is not used.  N-major tiles: 64 columns (128 bytes) per
// k-row, 8-k-row groups 1024 bytes apart (stride), 64-column blocks `lbo` bytes apart (leading).
// The start address sits in the low 14 bits (in units of 16 bytes), so stepping through a stage or through the
// ring is an addition to the low word.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3ffffu) >> 4);
  d |= (uint64_t)((lbo_bytes >> 4) & 0x3fffu) << 16;
  d |= (uint64_t)((sbo_bytes >> 4) & 0x3fffu) << 32;
  d |= 1ull << 46;  // descriptor version of this architecture
  d |= 2ull << 61;  // 128-byte swizzle
  return d;
}
// Instruction descriptor: bf16 x bf16 -> fp32, A K-major, B K- or N-major, M = 256 over the pair, N = n.
__device__ __forceinline__ uint32_t instr_desc(int n, bool b_nmajor) {
  uint32_t d = 0;
  d |= 1u << 4;   // accumulator format: fp32
  d |= 1u << 7;   // A: bf16
  d |= 1u << 10;  // B: bf16
  d |= (b_nmajor ? 1u : 0u) << 16;
  d |= (uint32_t)(n >> 3) << 17;
  d |= (uint32_t)(kPairRows >> 4) << 24;
  return d;
}

struct SmemGG {
  uint64_t full[kMaxStagesGG];   // leader's: both CTAs' operands of the stage have landed
  uint64_t empty[kMaxStagesGG];  // own: the MMAs have finished reading this CTA's stage
  uint64_t accum_full[2];        // own: all MMAs of the tile in accumulator buffer b have completed
  uint64_t accum_empty[2];       // leader's: the epilogue warps of both CTAs have read buffer b out of TMEM
  uint32_t tmem_base;
};

struct Tile {
  int e, m0, m_end, n0, ks;
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
  const int e0 = min(lane, P.E), e1 = min(lane + 32, P.E);
  m.lo0 = P.offsets[e0], m.hi0 = P.offsets[min(e0 + 1, P.E)];
  m.lo1 = P.offsets[e1], m.hi1 = P.offsets[min(e1 + 1, P.E)];
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
  return t;
}

__device__ __forceinline__ float silu_mul(float g, float u) { return __fdividef(g, 1.0f + __expf(-g)) * u; }

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
    for (int idx = pair; ok && idx < n_work; idx += n_pairs) {
      const Tile t = decode_tile(P, tm, idx, n_tiles);
      const int n0 = t.n0;
      const int kb0 = t.ks * num_kb / P.ksplit, kb1 = (t.ks + 1) * num_kb / P.ksplit;
      const int a_row = t.m0 + (int)rank * kBM;
      int k0 = kb0 * kBK;
      int kB = P.k_wrap > 0 ? k0 % P.k_wrap : k0;
      for (int kb = kb0; kb < kb1; ++kb, ++it) {
        if (it >= NS && !mbar_wait_warp(&sm.empty[slot], par)) {
          if (lane == 0) flag_error(P.st, MOE_ERR_TIMEOUT, 0x400u);
          ok = false;
          break;
        }
        unsigned char* st_a0 = stages + (size_t)slot * stage_bytes;
        unsigned char* st_b = st_a0 + n_a * a_bytes;
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
            tma_load_4d(st_b + (size_t)half_bn * kBK * 2, &map_b, kB, 1, nr, t.e, bar);
          } else if (P.bmode == B_SINGLE) {
            tma_load_4d(st_b, &map_b, kB, P.b_sub, n0 + (int)rank * half_bn, t.e, bar);
          } else {
            const int nc = n0 + (int)rank * half_bn;
            tma_load_4d(st_b, &map_b, nc, P.b_sub, kB, t.e, bar);
            if (P.bn > 128) tma_load_4d(st_b + (size_t)64 * kBK * 2, &map_b, nc + 64, P.b_sub, kB, t.e, bar);
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
      // steps through the stage (K-major operands: 32 bytes per 16 k-values; N-major: 16 k-rows of 128 bytes).
      const int n_mma = P.bmode == B_PAIR ? 2 * P.bn : P.bn;
      const uint32_t idesc = instr_desc(n_mma, P.bmode == B_NMAJOR);
      const uint64_t hi_k = smem_desc(0, 16, 1024) & 0xffffffff00000000ull;
      const uint64_t hi_b = (P.bmode == B_NMAJOR ? smem_desc(0, 64 * kBK * 2, 1024) : smem_desc(0, 16, 1024)) & 0xffffffff00000000ull;
      const uint32_t lo_b_lbo = (P.bmode == B_NMAJOR ? (uint32_t)(64 * kBK * 2 >> 4) : 1u) << 16;
      const uint32_t b_step = P.bmode == B_NMAJOR ? (2048u >> 4) : (32u >> 4);
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
          const uint64_t db = hi_b | (uint64_t)((st_lo + b_off) | lo_b_lbo);
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
              for (uint32_t kk = 0; kk < kBK / 16; ++kk) tc_mma_bf16(d_tmem, da + 2u * kk, db + b_step * kk, idesc, acc | kk);
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
}

// ---- host: tensor maps --------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess) {
      (void)cudaGetLastError();
      return nullptr;
    }
    fn = (EncodeTiledFn)p;
  }
  return fn;
}

// rank-2 map over a row-major bf16 matrix [rows][ld], columns [0, cols): box 64 x 128
int make_map_a(CUtensorMap* m, const void* base, long long rows, long long cols, long long ld) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return MOE_ERR_CUDA;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  const cuuint32_t box[2] = {kBK, kBM};
  const cuuint32_t es[2] = {1, 1};
  const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? MOE_OK : MOE_ERR_CUDA;
}
// rank-4 map over an interleaved matrix [S][rows][nsub][inner]: coordinates (inner, sub, row, slot)
int make_map_b(CUtensorMap* m, const void* base, long long inner, int nsub, long long rows, int slots, int box_inner,
               int box_rows, CUtensorMapSwizzle swizzle = CU_TENSOR_MAP_SWIZZLE_128B) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return MOE_ERR_CUDA;
  const cuuint64_t dims[4] = {(cuuint64_t)inner, (cuuint64_t)nsub, (cuuint64_t)rows, (cuuint64_t)slots};
  const cuuint64_t strides[3] = {(cuuint64_t)inner * 2, (cuuint64_t)inner * nsub * 2,
                                 (cuuint64_t)inner * nsub * rows * 2};
  const cuuint32_t box[4] = {(cuuint32_t)box_inner, 1, (cuuint32_t)box_rows, 1};
  const cuuint32_t es[4] = {1, 1, 1, 1};
  const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, es,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? MOE_OK : MOE_ERR_CUDA;
}

void pair_launch_config(cudaLaunchConfig_t& lc, cudaLaunchAttribute* attr, int ctas, size_t smem, cudaStream_t s) {
  lc = cudaLaunchConfig_t{};
  lc.gridDim = dim3(ctas), lc.blockDim = dim3(kThreadsGG), lc.dynamicSmemBytes = smem, lc.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2, attr[0].val.clusterDim.y = 1, attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = attr, lc.numAttrs = 2;
}

// Pairs of CTAs the device can hold at once (one CTA per SM; a pair sits on two SMs of one cluster).
// Every launch of the kernel takes more than half of an SM's shared memory, so the number does not depend on the
// launch: the driver is asked once per device (the query costs more than a launch).
int max_pairs(const moe_ctx* ctx, size_t smem) {
  static std::atomic<int> known[kMaxDevices];
  const bool tracked = ctx->device >= 0 && ctx->device < kMaxDevices;
  if (tracked && known[ctx->device].load(std::memory_order_relaxed) > 0)
    return known[ctx->device].load(std::memory_order_relaxed);
  cudaLaunchConfig_t lc;
  cudaLaunchAttribute attr[2];
  pair_launch_config(lc, attr, ctx->sm_count & ~1, smem, nullptr);
  lc.numAttrs = 1;  // the cluster shape alone decides the occupancy
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, grouped_gemm_kernel, &lc) != cudaSuccess || n < 1) {
    (void)cudaGetLastError();
    n = ctx->sm_count / 2;
  }
  n = std::max(1, std::min(n, ctx->sm_count / 2));
  if (tracked) known[ctx->device].store(n, std::memory_order_relaxed);
  return n;
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
  const int pairs = (int)std::min<long long>(m_tiles * n_tiles * P.ksplit, max_pairs(ctx, smem));
  cudaLaunchConfig_t lc;
  cudaLaunchAttribute attr[2];
  pair_launch_config(lc, attr, 2 * pairs, smem, s);
  MOE_CUDA_TRY(cudaLaunchKernelEx(&lc, grouped_gemm_kernel, a0, a1, b, P));
  ctx->launches++;
  return MOE_OK;
}

// Output columns per tile: the largest of 64, 128, ... `cap` that is not mostly padding.
int pick_bn(int n_total, int cap, int floor_bn = 64) {
  int bn = cap;
  while (bn > floor_bn && bn / 2 >= n_total) bn /= 2;
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

int launch_tensor_ffn(moe_ctx* ctx, const void* x, int T, const moe_weights* w, const int32_t* offsets,
                      const int32_t* perm, char* ws, const WsLayout& L, float* out_slots, int* out_planes,
                      cudaStream_t s) {
  const moe_config& c = ctx->cfg;
  if (w->expert_slot) return MOE_ERR_UNSUPPORTED;  // the tensor path reads experts in place (slot == expert)
  const int d = c.d_model, f = c.d_ff, r = c.wd_rank, E = c.n_experts;
  const int n_slots = T * c.top_k;
  if (out_planes) *out_planes = 1;
  void* xperm = ws + L.xperm;
  void* hidden = ws + L.hidden;
  int rc = launch_gather_rows(ctx, x, perm, n_slots, xperm, s);
  if (rc != MOE_OK) return rc;
  CUtensorMap ma, ma1, mb;
  GGParams P{};
  P.offsets = offsets;
  if (r == 0) {
    // (1) hidden = silu(X Wg) * (X Wu): the tile's 128 gate rows come in through one CTA, its 128 up rows through the other
    if ((rc = make_map_a(&ma, xperm, n_slots, d, d)) != MOE_OK) return rc;
    if ((rc = make_map_b(&mb, w->gud, d, 3, f, E, kBK, 128)) != MOE_OK) return rc;
    P.K = d, P.n_total = f, P.bn = 128, P.bmode = B_PAIR, P.b_sub = 0, P.epi = EPI_SWIGLU;
    P.out = hidden, P.ld_out = f, P.out_off2 = 0;
    if ((rc = launch_gg(ctx, ma, ma, mb, P, n_slots, s)) != MOE_OK) return rc;
    // (2) out_slots = hidden Wd   (B = down rows of gud: [k = hidden unit][n = model column], n contiguous)
    if ((rc = make_map_a(&ma, hidden, n_slots, f, f)) != MOE_OK) return rc;
    if ((rc = make_map_b(&mb, w->gud, d, 3, f, E, 64, kBK)) != MOE_OK) return rc;
    P.K = f, P.n_total = d, P.bn = pick_bn(d, 256, 128), P.bmode = B_NMAJOR, P.b_sub = 2;
    P.epi = EPI_F32, P.out = out_slots, P.ld_out = d, P.out_off2 = 0;
    if (n_slots <= kKSplitMaxSlots) {
      // short prefill: too few tiles for the SMs, and every tile streams a long run of weights.  Cut the contraction so
      // that every pair streams a part, each part into its own plane; the caller sums the planes, or they are summed
      // here (in the same order: the layer and its four calls give the same bits).
      const long long tiles = (long long)row_tiles(n_slots, E) * ((d + P.bn - 1) / P.bn);
      const int ks = pick_ksplit(tiles, (f + kBK - 1) / kBK, ctx->sm_count / 2, kKSplitMax);
      if (ks > 1) {
        P.ksplit = ks, P.plane_elems = (long long)n_slots * d;
        if (!out_planes) {
          P.out = ws + L.out_slots;
          if ((rc = launch_gg(ctx, ma, ma, mb, P, n_slots, s)) != MOE_OK) return rc;
          return launch_sum_planes(ctx, (const float*)P.out, P.plane_elems, ks, out_slots, s);
        }
        *out_planes = ks;
      }
    }
    return launch_gg(ctx, ma, ma, mb, P, n_slots, s);
  }
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
  if ((rc = make_map_a(&ma, xperm, n_slots, d, d)) != MOE_OK) return rc;
  const int pairs = ctx->sm_count / 2, m_tiles = row_tiles(n_slots, E);
  P.bn = pick_bn(r, 128);
  while (P.bn > 64 && 2 * m_tiles * ((r + P.bn - 1) / P.bn) <= pairs) P.bn /= 2;  // a small rank leaves pairs idle: narrower tiles
  if ((rc = make_map_b(&mb, w->wd_a, d, 2, r, E, kBK, P.bn)) != MOE_OK) return rc;
  P.K = d, P.n_total = r, P.bmode = B_PAIR, P.b_sub = 0, P.epi = EPI_BF16_PAIR;
  P.k_wrap = 0, P.split = 1, P.out = mid_a, P.ld_out = 2 * tw, P.out_off2 = tw, P.out_off_lo = rp, P.n_store = rp;
  if ((rc = launch_gg(ctx, ma, ma, mb, P, n_slots, s)) != MOE_OK) return rc;
  // (2) hidden = silu(Tg gR) * (Tu uR): two A operands, each CTA brings half of the gate and half of the up rows
  if ((rc = make_map_a(&ma, mid_a, n_slots, tw, 2 * tw)) != MOE_OK) return rc;
  if ((rc = make_map_a(&ma1, (const __nv_bfloat16*)mid_a + tw, n_slots, tw, 2 * tw)) != MOE_OK) return rc;
  if ((rc = make_map_b(&mb, w->wd_b, r, 2, f, E, kBK, 64)) != MOE_OK) return rc;
  P.K = tw, P.n_total = f, P.bn = 128, P.bmode = B_DUAL, P.b_sub = 0, P.epi = EPI_SWIGLU;
  P.k_wrap = rp, P.split = 0, P.out = hidden, P.ld_out = f, P.out_off2 = 0, P.out_off_lo = 0, P.n_store = 0;
  if ((rc = launch_gg(ctx, ma, ma1, mb, P, n_slots, s)) != MOE_OK) return rc;
  // (3) V = hidden dL
  if ((rc = make_map_a(&ma, hidden, n_slots, f, f)) != MOE_OK) return rc;
  P.bn = pick_bn(r, 256);
  if ((rc = make_map_b(&mb, w->wd_c, f, 1, r, E, kBK, P.bn / 2)) != MOE_OK) return rc;
  P.K = f, P.n_total = r, P.bmode = B_SINGLE, P.b_sub = 0, P.epi = EPI_BF16;
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
  P.K = tw, P.n_total = d, P.bmode = B_SINGLE, P.b_sub = 0, P.epi = EPI_F32;
  P.k_wrap = rp, P.split = 0, P.out = out_slots, P.ld_out = d, P.out_off2 = 0, P.out_off_lo = 0, P.n_store = 0;
  return launch_gg(ctx, ma, ma, mb, P, n_slots, s);
}

}  // namespace cosmoe
