// tcgen05 (5th-generation tensor core) and TMA helpers shared by the
// tensor-core kernels of the library: the dense refresh (did_refresh_tc.cu)
// and the batched order of Algorithm 3 (did_batched.cu).
//
// Conventions used throughout:
//   - Shared-memory operands are in the no-swizzle K-major core-matrix layout:
//     a core matrix is 8 rows x 16 bytes; core matrices adjacent along K are
//     128 bytes apart (LBO), adjacent along M/N are Kp*E*8 bytes apart (SBO)
//     for a contraction length Kp of E-byte elements.  One bfloat16 MMA
//     (kind::f16) consumes 16 elements of K, 32 bytes (two core matrices), so
//     its start address advances by 256 bytes per K step.
//   - An A operand held in tensor memory (TMEM) has row i in lane i and two
//     bfloat16 elements per 32-bit column (the even K index in the low half);
//     one MMA reads 8 consecutive columns.
//   - A warp reads or writes only its own quarter of the 128 TMEM lanes
//     (lanes 32 (warp % 4) ..), addressed as (lane << 16) | column.
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>

#include <mutex>

#include "did_internal.cuh"

namespace did {
namespace tc {

// Shared-memory matrix descriptor (no swizzle, K-major): start address >> 4
// in bits 0-13, leading (K-direction) byte offset >> 4 in bits 16-29, stride
// (M/N-direction) byte offset >> 4 in bits 32-45, descriptor version 1 in
// bits 46-47, base offset 0, swizzle mode 0.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// Instruction descriptor of tcgen05.mma kind::f16: dense, D float32 (bits
// 4-5 = 1), A and B bfloat16 (bits 7-9 = 1, bits 10-12 = 1), both K-major
// (bits 15, 16 = 0), N >> 3 in bits 17-22, M >> 4 in bits 24-28.
__host__ __device__ constexpr uint32_t instr_desc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void tmem_alloc(uint32_t* dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// True in one thread of a converged warp (elect.sync; the same thread each
// time).  MMA issue must sit under this predicate, not under `lane == 0`: with
// an elected thread the compiler knows that one thread is active, so an MMA's
// descriptors stay in uniform registers.  Measured back to back on one
// SM (M = 128, K = 16, A in TMEM): 16 / 32 / 48 / 64 / 128 cycles an MMA at
// N = 32 / 64 / 96 / 128 / 256 -- N / 2, the tensor rate -- against 45 / 45 /
// 48 / 64 / 128 under `lane == 0`, and about 114 at every N up to 128 there
// once the descriptors come out of the pipeline loops of the real kernels.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(p));
  return p != 0;
}

// D (TMEM) (+)= A (shared memory) x B (shared memory).
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrive once on an mbarrier when every MMA this thread issued so far is done.
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// N consecutive float32 columns of this thread's TMEM lane (warp-collective).
template <int N>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, float* v);
template <>
__device__ __forceinline__ void tmem_ld<8>(uint32_t taddr, float* v) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}
template <>
__device__ __forceinline__ void tmem_ld<16>(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Three loads of 16 columns in flight at once, one wait: the registers are
// tied to the wait through empty asm statements, so no use of them can be
// scheduled before it.
__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void regs_after_wait16(uint32_t* r) {
  asm volatile(""
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                 "+r"(r[15])
               :
               : "memory");
}
__device__ __forceinline__ void tmem_ld3x16(uint32_t t0, uint32_t t1, uint32_t t2, float* v0, float* v1, float* v2) {
  uint32_t a[16], b[16], c[16];
  tmem_ld16_nowait(t0, a);
  tmem_ld16_nowait(t1, b);
  tmem_ld16_nowait(t2, c);
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
  regs_after_wait16(a);
  regs_after_wait16(b);
  regs_after_wait16(c);
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    v0[i] = __uint_as_float(a[i]);
    v1[i] = __uint_as_float(b[i]);
    v2[i] = __uint_as_float(c[i]);
  }
}

__device__ __forceinline__ void tmem_ld2x16(uint32_t t0, uint32_t t1, float* v0, float* v1) {
  uint32_t a[16], b[16];
  tmem_ld16_nowait(t0, a);
  tmem_ld16_nowait(t1, b);
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
  regs_after_wait16(a);
  regs_after_wait16(b);
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    v0[i] = __uint_as_float(a[i]);
    v1[i] = __uint_as_float(b[i]);
  }
}

// TMEM stores are asynchronous: tmem_st_wait() completes them, and a
// following fence_before + mbarrier arrive publishes the values to the MMA
// thread.
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Bounded mbarrier wait used by every role.  A phase that has completed
// returns at once, without touching global memory (the pipelines wait several
// times per tile, and a load of the error word costs a trip to L2 each time).
// While spinning, the error word and the %globaltimer limit are checked every
// 256 polls; returns false once the error word is set (by this wait running
// out, or by another role whose wait ran out).
__device__ __forceinline__ bool wait(uint64_t* bar, uint32_t parity, int* err, uint64_t timeout_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  for (uint32_t it = 1;; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 255u) == 0) {
      if (ld_volatile(err) != 0) return false;
      if (globaltimer_ns() - t0 > timeout_ns || it > (1u << 28)) {
        atomicCAS(err, 0, kDevErrTimeout);
        return false;
      }
    }
  }
}

// 2-D tensor copy global -> shared of the box at (x, y), completing on an
// mbarrier (x: innermost coordinate in elements; x * element bytes must be a
// multiple of 16).
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
          "r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}
// 2-D tensor copy shared -> global of the box at (x, y) (x >= 0; elements
// outside the tensor are not written).  Committed as a bulk group.
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, int x, int y, const void* src) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(x), "r"(y), "r"(smem_u32(src))
               : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// Wait until the shared-memory sources of this thread's bulk groups have been read.
__device__ __forceinline__ void bulk_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
// Wait until this thread's bulk groups are complete (writes visible).
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Split of a float32 value into three bfloat16 terms, each the round-to-
// nearest of what the previous ones left (the remainders are exact in
// float32): v = p0 + p1 + p2 + r with |r| <= 2^-27 |v| (three 8-bit
// significands).  The six products p_i q_j with i + j <= 2 of two such splits
// carry every term down to 2^-18 of the leading one; the three dropped terms
// are below 2^-26 relative, so BF16x6 products match float32 arithmetic.
__device__ __forceinline__ void split_bf16x3(float v, __nv_bfloat16& p0, __nv_bfloat16& p1, __nv_bfloat16& p2) {
  p0 = __float2bfloat16_rn(v);
  const float r1 = v - __bfloat162float(p0);
  p1 = __float2bfloat16_rn(r1);
  const float r2 = r1 - __bfloat162float(p1);
  p2 = __float2bfloat16_rn(r2);
}

// 8 or 16 32-bit words into this thread's TMEM lane (warp-collective).
__device__ __forceinline__ void tmem_st_u8(uint32_t taddr, const uint32_t* v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(v[0]),
               "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}
__device__ __forceinline__ void tmem_st_u16(uint32_t taddr, const uint32_t* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
          taddr),
      "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
      "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
      : "memory");
}
// D (TMEM) (+)= A (TMEM, 128 lanes x 16 bfloat16 in 8 columns from a_tmem) x B (shared memory), kind::f16.
__device__ __forceinline__ void mma_bf16_tmem_a(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                                uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

}  // namespace tc

// cuTensorMapEncodeTiled from the driver, through the runtime's entry-point query.
inline PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// A float32 column-major matrix (rows contiguous, `ld` elements between
// columns) as a 2-D tensor map with a box of box_rows x box_cols.
inline bool encode_f32_colmajor(CUtensorMap* map, const void* base, int64_t rows, int64_t cols, int64_t ld,
                                int box_rows, int box_cols, CUtensorMapSwizzle swizzle) {
  PFN_cuTensorMapEncodeTiled_v12000 encode = tensor_map_encoder();
  if (!encode) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)rows, (cuuint64_t)cols};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * sizeof(float)};
  const cuuint32_t box[2] = {(cuuint32_t)box_rows, (cuuint32_t)box_cols};
  const cuuint32_t estr[2] = {1, 1};
  return encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(base), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace did
