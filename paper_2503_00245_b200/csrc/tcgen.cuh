// PTX wrappers and host helpers of the kernels that run on the 5th-generation tensor cores (csrc/tensor_ffn.cu, csrc/dense_prefill.cu).
#pragma once

#include <cuda.h>

#include <algorithm>

#include "common.cuh"

namespace cosmoe {

namespace {

constexpr int kBM = 128;  // rows per CTA and tile (TMEM lanes)
constexpr int kBK = 64;   // K elements per stage (128 bytes of bf16 = one swizzle row)
constexpr int kEpiWarps = 8;  // two per quarter of the TMEM lanes, splitting the columns
constexpr int kTmemCols = 512;  // two accumulator buffers of 256 columns
constexpr int kAccCols = 256;

// ---- PTX wrappers ------------------------------------------------------------------------------------
// Tiled loads whose completion may be counted on a barrier of the other CTA of the pair (cta_group::2); the
// data always lands in the issuing CTA's own shared memory.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar_cluster) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
      "[%4];" ::"r"(dst),
      "l"(map), "r"(c0), "r"(c1), "r"(bar_cluster)
      : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                            uint32_t bar_cluster) {
  asm volatile(
      "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
      "%5}], [%6];" ::"r"(dst),
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
// A word to the shared memory of another CTA of the cluster (ordered by a barrier of the cluster) ...
__device__ __forceinline__ void st_cluster(uint32_t dst_cluster, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(dst_cluster), "r"(v) : "memory");
}
// ... and 16 bytes that the barrier there counts when they have arrived.
__device__ __forceinline__ void st_async4(uint32_t dst_cluster, int4 v, uint32_t bar_cluster) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.u32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(dst_cluster),
               "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar_cluster)
               : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
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
__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tc_wait_ld16(uint32_t* v) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
      : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
        "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15])
      :
      : "memory");
}
__device__ __forceinline__ void tc_wait_ld16(uint32_t* a, uint32_t* v) {  // two loads, one wait
  tc_wait_ld16(a);
  asm volatile(""
      : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
        "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]));
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
// Instruction descriptor: bf16 x bf16 -> fp32, M = 256 over the pair, N = n; B K-major, A K-major or stored [k][m].
__device__ __forceinline__ uint32_t instr_desc(int n, bool a_mmajor) {
  uint32_t d = 0;
  d |= 1u << 4;   // accumulator format: fp32
  d |= 1u << 7;   // A: bf16
  d |= 1u << 10;  // B: bf16
  d |= (a_mmajor ? 1u : 0u) << 15;
  d |= (uint32_t)(n >> 3) << 17;
  d |= (uint32_t)(2 * kBM >> 4) << 24;
  return d;
}

// silu(g) u = g u / (1 + e^-g), with e^-g = 2^(-g log2(e)): one power of two and one reciprocal on the special-function unit, whose
// rate bounds the epilogue.  The PTX manual gives their relative errors, 2^-22 and 2^-23.  The exponent is rounded to fp32 (its
// factor too), 1.25 2^-24 of itself, which is |g| 1.25 2^-24 of e^-g; the sum and the two products round at 2^-24.  With
// p = e^-g / (1 + e^-g), at most 1: the relative error is at most p (|g| 1.25 2^-24 + 2^-22) + 5 2^-24.  Below g = -87 the
// reciprocal would be smaller than 2^-126 and is zero, as is the result then: |g| 2^-126 is lost.  The bf16 that the value is
// stored as is 2^-9 wide.
// (One reciprocal for two values' denominators would save a quarter of these instructions; but a value would then depend on its
// neighbour, which is another token.)
__device__ __forceinline__ float silu_mul(float g, float u) {
  float e, r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(g * -1.4426950408889634f));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(1.0f + e));
  return g * r * u;
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

// rank-2 map over a row-major bf16 matrix [rows][ld], columns [0, cols): box 64 x box_rows
int make_map_a(CUtensorMap* m, const void* base, long long rows, long long cols, long long ld, int box_rows = kBM) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return MOE_ERR_CUDA;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  const cuuint32_t box[2] = {kBK, (cuuint32_t)box_rows};
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

void pair_launch_config(cudaLaunchConfig_t& lc, cudaLaunchAttribute* attr, int ctas, int threads, size_t smem, cudaStream_t s) {
  lc = cudaLaunchConfig_t{};
  lc.gridDim = dim3(ctas), lc.blockDim = dim3(threads), lc.dynamicSmemBytes = smem, lc.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2, attr[0].val.clusterDim.y = 1, attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = attr, lc.numAttrs = 2;
}

// Pairs of CTAs the device can hold at once (one CTA per SM; a pair sits on two SMs of one cluster).
// Every launch of the kernel takes more than half of an SM's shared memory, so the number does not depend on the
// launch: the driver is asked once per device (the query costs more than a launch).
template <auto Kernel>
int max_pairs(const moe_ctx* ctx, int threads, size_t smem) {
  static std::atomic<int> known[kMaxDevices];
  const bool tracked = ctx->device >= 0 && ctx->device < kMaxDevices;
  if (tracked && known[ctx->device].load(std::memory_order_relaxed) > 0)
    return known[ctx->device].load(std::memory_order_relaxed);
  cudaLaunchConfig_t lc;
  cudaLaunchAttribute attr[2];
  pair_launch_config(lc, attr, ctx->sm_count & ~1, threads, smem, nullptr);
  lc.numAttrs = 1;  // the cluster shape alone decides the occupancy
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, Kernel, &lc) != cudaSuccess || n < 1) {
    (void)cudaGetLastError();
    n = ctx->sm_count / 2;
  }
  n = std::max(1, std::min(n, ctx->sm_count / 2));
  if (tracked) known[ctx->device].store(n, std::memory_order_relaxed);
  return n;
}

}  // namespace
}  // namespace cosmoe
