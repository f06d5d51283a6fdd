// Device helpers shared by the tcgen05 kernels: mbarriers with %globaltimer-bounded
// waits, 3-D TMA loads, shared-memory matrix descriptors (K-major, 64-byte rows, 64-byte
// swizzle), TF32 MMA issue / commit, TMEM loads, and the TF32 hi/lo split.
#pragma once

#include <cstdint>

#include "f32conv.cuh"

namespace tnt {
namespace tc {

constexpr uint64_t WAIT_NS = 2000000000ull;  // 2 s per wait

__device__ __forceinline__ uint32_t su32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint64_t gtimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(b)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(b)) : "memory");
}
__device__ __forceinline__ uint32_t mbar_try(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(su32(b)), "r"(parity)
      : "memory");
  return ok;
}
// bounded wait; false (and the status bit set) if the phase never completed
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, int* status) {
  if (mbar_try(b, parity)) return true;
  const uint64_t t0 = gtimer();
  while (!mbar_try(b, parity)) {
    if (gtimer() - t0 > WAIT_NS) {
      atomicOr(status, 1);
      return false;
    }
  }
  return true;
}
__device__ __forceinline__ void tma_load3(void* dst, const CUtensorMap* tm, uint64_t* bar, int c0,
                                          int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(su32(dst)),
      "l"((uint64_t)tm), "r"(su32(bar)), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}
// K-major operand tile, 64-byte rows, 64-byte swizzle: 8-row atoms of 512 bytes.  The low word of
// the descriptor is the shared-memory address / 16 with the (here unused) leading byte offset
// 1 above it, the high word constant: the stride byte offset to the next 8-row atom, the
// descriptor version and the 64-byte swizzle.  The issuing thread adds to low words only: with
// 64-bit descriptors built per MMA it took longer than the MMAs.
constexpr uint32_t DESC_SW64_HI = (512u >> 4) | (1u << 14) | (4u << 29);
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr) { return (saddr >> 4) | (1u << 16); }
// instruction descriptor: D = F32, A = B = TF32, both K-major, M = 128, N = n
__host__ __device__ constexpr uint32_t idesc_tf32_n(int n) {
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
__device__ __forceinline__ void mma_tf32(uint32_t tmem, uint32_t alo, uint32_t blo, uint32_t id,
                                         uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "mov.b64 a, {%1, %5};\n\t"
      "mov.b64 b, {%2, %5};\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], a, b, %3, p;\n\t}\n" ::"r"(tmem),
      "r"(alo), "r"(blo), "r"(id), "r"(acc), "r"(DESC_SW64_HI)
      : "memory");
}
// The split-TF32 complex products of one stage (16 of K: two MMA steps) at shared address
// `base`: A planes re_hi, re_lo, im_hi, im_lo of TA bytes each, then B's of TB bytes.  re-re
// products into t_re, im-im into t_rn (subtracted by the epilogue), the cross terms into
// t_im; first: the accumulators start here.
template <int TA, int TB>
__device__ __forceinline__ void mma_cplx_tf32x3(uint32_t base, uint32_t t_re, uint32_t t_im, uint32_t t_rn,
                                                uint32_t id, bool first) {
  const uint32_t a0 = desc_lo(base), b0 = a0 + (4 * TA >> 4);
#pragma unroll
  for (int ks = 0; ks < 2; ++ks) {  // K = 8 per tf32 MMA: 32 bytes along the row
    const uint32_t a_rh = a0 + 2 * ks, a_rl = a_rh + (TA >> 4), a_ih = a_rl + (TA >> 4), a_il = a_ih + (TA >> 4);
    const uint32_t b_rh = b0 + 2 * ks, b_rl = b_rh + (TB >> 4), b_ih = b_rl + (TB >> 4), b_il = b_ih + (TB >> 4);
    const uint32_t acc = (ks == 0 && first) ? 0u : 1u;
    mma_tf32(t_re, a_rh, b_rh, id, acc);
    mma_tf32(t_re, a_rh, b_rl, id, 1);
    mma_tf32(t_re, a_rl, b_rh, id, 1);
    mma_tf32(t_rn, a_ih, b_ih, id, acc);
    mma_tf32(t_rn, a_ih, b_il, id, 1);
    mma_tf32(t_rn, a_il, b_ih, id, 1);
    mma_tf32(t_im, a_rh, b_ih, id, acc);
    mma_tf32(t_im, a_rh, b_il, id, 1);
    mma_tf32(t_im, a_rl, b_ih, id, 1);
    mma_tf32(t_im, a_ih, b_rh, id, 1);
    mma_tf32(t_im, a_ih, b_rl, id, 1);
    mma_tf32(t_im, a_il, b_rh, id, 1);
  }
}
// 32 values of one row to memory (nc of them exist): 16 bytes per store where p allows it (one
// float per store put each of a warp's 32 rows into its own sector, 32 times over)
__device__ __forceinline__ void store_row32(float* p, const uint32_t* v, int nc) {
  if (nc >= 32 && ((uintptr_t)p & 15) == 0) {
#pragma unroll
    for (int j = 0; j < 32; j += 4) *(uint4*)(p + j) = make_uint4(v[j], v[j + 1], v[j + 2], v[j + 3]);
    return;
  }
#pragma unroll
  for (int j = 0; j < 32; ++j)
    if (j < nc) p[j] = __uint_as_float(v[j]);
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          su32(bar))
      : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
      "%11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, "
      "%28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
        "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
        "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
      "%11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ float tf32_rna(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}
__device__ __forceinline__ void split_tf32(float x, float* hi, float* lo) {
  const float h = tf32_rna(x);
  *hi = h;
  *lo = tf32_rna(x - h);
}
// An FP64 value is first truncated to FP32 by integer operations (f32conv.cuh; 2^-23
// relative), then split: hi + lo is within ~1.5 2^-22 of x, the split-TF32 products' own
// error, and no FP64-pipe conversion or subtraction enters the operand conversion kernels
__device__ __forceinline__ void split_tf32(double x, float* hi, float* lo) {
  split_tf32(f32_of(x), hi, lo);
}


}  // namespace tc
}  // namespace tnt
