// nep_tc.cuh -- 5th-generation tensor-core (tcgen05 / UMMA) helpers for sm_103a: shared-memory matrix
// descriptors, the f16-kind instruction descriptor, tensor-memory (TMEM) allocation and loads, and
// mbarrier completion with a bounded wait.
//
// Operand layout used here: K-major, no swizzle, built from "core matrices" of 8 rows x 16 bytes
// (8 x 8 16-bit elements, rows contiguous).  Core matrices are stored [row group][k group]: the byte
// step between core matrices along K is 128 (the descriptor's leading-dimension offset) and along
// M/N is KG * 128 (its stride-dimension offset), KG = K / 8.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "nep_common.cuh"

namespace nep {

constexpr int ST_TIMEOUT = 4;          // status bit: a bounded wait on the tensor core ran out

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Element offset of (row, k) in a K-major no-swizzle tile with KG core matrices along K.
__host__ __device__ constexpr int tile_off(int row, int k, int KG) {
  return ((row >> 3) * KG + (k >> 3)) * 64 + (row & 7) * 8 + (k & 7);
}

// Shared-memory matrix descriptor (sm_100 family): start address, leading- and stride-dimension
// byte offsets (all >> 4), descriptor version 1, no swizzle.
__device__ __forceinline__ uint64_t umma_smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// Instruction descriptor of tcgen05.mma .kind::f16: f32 accumulator, A and B both f16 (0) or both
// bf16 (1), both K-major, N >> 3 at bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t umma_idesc_f16(int M, int N, int bf16) {
  return (1u << 4) | ((uint32_t)bf16 << 7) | ((uint32_t)bf16 << 10) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

template <class T>
__device__ __forceinline__ T to_mma_type(float x);
template <>
__device__ __forceinline__ __nv_bfloat16 to_mma_type<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }
template <>
__device__ __forceinline__ __half to_mma_type<__half>(float x) { return __float2half_rn(x); }
template <class T>
struct MmaKind;
template <>
struct MmaKind<__nv_bfloat16> {
  static constexpr int bf16 = 1;
};
template <>
struct MmaKind<__half> {
  static constexpr int bf16 = 0;
};

template <class MT>
__device__ __forceinline__ float round_to(float x) {
  if constexpr (std::is_same<MT, float>::value) return x;
  else if constexpr (std::is_same<MT, __half>::value) return __half2float(__float2half_rn(x));
  else return __bfloat162float(__float2bfloat16_rn(x));
}


// tanh of the hardware's special-function unit (PTX tanh.approx.f32: relative error about 2^-11, the unit
// roundoff of the 16-bit operands it feeds in the mixed-precision network).
__device__ __forceinline__ float tanh_sfu(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void mbar_init(uint64_t *mbar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(mbar)), "r"(count) : "memory");
}

// Wait for phase `parity` of the mbarrier, giving up after `limit` polls; returns false on time-out.
__device__ __forceinline__ bool mbar_wait(uint64_t *mbar, uint32_t parity, long limit) {
  uint32_t done = 0;
  for (long it = 0; it < limit && !done; ++it) {
    asm volatile(
        "{\n\t.reg .pred P;\n\tmbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n\tselp.b32 %0, 1, 0, P;\n\t}"
        : "=r"(done)
        : "r"(smem_addr(mbar)), "r"(parity)
        : "memory");
  }
  return done != 0;
}

__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Warp-wide TMEM allocation of ncols columns (power of two >= 32); the base address goes to *dst.
__device__ __forceinline__ void tmem_alloc(uint32_t *dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(dst)), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// D[tmem] (+)= A * B^T, issued by one thread.
__device__ __forceinline__ void umma_f16(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, int accumulate) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(
                   tmem_d),
               "l"(da), "l"(db), "r"(idesc), "r"(accumulate)
               : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t *mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(mbar))
               : "memory");
}

// 32 consecutive f32 columns of this thread's TMEM lane (warp w reads lanes 32w..32w+31).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int k = 0; k < 32; ++k) v[k] = __uint_as_float(r[k]);
}

// TMEM as per-thread storage (no tensor-core instruction involved): with the 32x32b shape, thread t
// of warp w owns lane 32 (w mod 4) + t, and a thread's values occupy consecutive columns of its lane.
// All of these are warp-collective (.sync.aligned): the whole warp executes them together.

// Columns [taddr, taddr + 4), and [taddr, taddr + 16), of this thread's lane <- v.
__device__ __forceinline__ void tmem_st(uint32_t taddr, const float (&v)[4]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(__float_as_uint(v[0])),
               "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])));
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16};" ::"r"(taddr),
      "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])),
      "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])),
      "r"(__float_as_uint(v[8])), "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])),
      "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])), "r"(__float_as_uint(v[15])));
}
// Wait until this thread's TMEM stores have completed.
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Per-thread rows of 5 channels x NLM components in TMEM ("chunked" layout): chunk k holds the
// components lm = 4k..4k+3; channels 0..3 of chunk k sit in the 16 columns 16k + 4a + (lm mod 4)
// (one x16 access at a 16-aligned column) and channel 4 in the 4 columns 16 NC + lm (one x4 access at a
// 4-aligned column), NC = NLM / 4 chunks.  With NLM = 24: 96 + 24 = 120 columns.  Every access is aligned to its own width.
__host__ __device__ constexpr uint32_t tm_col(int a, int lm, int nlm) {
  return a < 4 ? (uint32_t)((lm >> 2) * 16 + a * 4 + (lm & 3)) : (uint32_t)((nlm >> 2) * 16 + lm);
}

// Chunk k of the five channels, loaded and waited for in one statement.
template <int NLM>
__device__ __forceinline__ void tmem_ld_chunk(uint32_t trow, int k, float (&v)[5][4]) {
  uint32_t r[20];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
      "[%20];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%16, %17, %18, %19}, [%21];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19])
      : "r"(trow + tm_col(0, 4 * k, NLM)), "r"(trow + tm_col(4, 4 * k, NLM)));
#pragma unroll
  for (int a = 0; a < 5; ++a)
#pragma unroll
    for (int c = 0; c < 4; ++c) v[a][c] = __uint_as_float(r[4 * a + c]);
}
// Chunk k of the five channels <- v (not waited for: tmem_wait_st before the columns are read again).
template <int NLM>
__device__ __forceinline__ void tmem_st_chunk(uint32_t trow, int k, const float (&v)[5][4]) {
  float w[16];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int c = 0; c < 4; ++c) w[4 * a + c] = v[a][c];
  tmem_st16(trow + tm_col(0, 4 * k, NLM), w);
  tmem_st(trow + tm_col(4, 4 * k, NLM), v[4]);
}

}  // namespace nep
