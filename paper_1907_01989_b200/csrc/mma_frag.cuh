// What the kernels on the warp-level matrix instruction share: mma.sync fragments, shared-memory accesses, the banded operand of
// a depthwise convolution.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "gi_internal.h"
#include "sm100_ptx.cuh"

namespace gi {
namespace frag {

constexpr int kTableBytes = 1024;  // banded depthwise operands of 4 slices: [slice][16 lanes][3 window rows + pad] x 4 bytes
constexpr int kBiasBytes = 64;     // 16 floats
constexpr int kDwBiasBytes = 256;  // bias of 16 channels, each four times: the start value of a fragment of sums

// The largest finite fp16 value, twice.  A tensor that stays on the SM and is multiplied by structural zeros - the banded operand of
// a depthwise convolution, a 1x1 evaluated as a window - holds it in the place of infinity: 0 x infinity would reach pixels and
// channels that the value has nothing to do with.
constexpr unsigned kMaxFinite = 0x7bff7bffu;

__device__ __forceinline__ void ldsm4(unsigned addr, unsigned (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm2(unsigned addr, unsigned& a, unsigned& b) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];" : "=r"(a), "=r"(b) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma16816(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// the same with the sum started from zero
__device__ __forceinline__ void mma16816z(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %10, %10, %10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.0f));
}
// the same with the sum started from c0..c3 (a bias).  The compiler copies them into the accumulators: four moves, where the
// values are used again
__device__ __forceinline__ void mma16816c(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1, float c0, float c1, float c2,
                                          float c3) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %11, %12, %13};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(c0), "f"(c1), "f"(c2), "f"(c3));
}
__device__ __forceinline__ void mma1688(float (&d)[4], unsigned a0, unsigned a1, unsigned b0) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5}, {%6}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(b0));
}
// the same with the sum started from zero
__device__ __forceinline__ void mma1688z(float (&d)[4], unsigned a0, unsigned a1, unsigned b0) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5}, {%6}, {%7, %7, %7, %7};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a0), "r"(a1), "r"(b0), "f"(0.0f));
}
// a += c, b += d in one instruction
__device__ __forceinline__ void add2(float& a, float& b, float c, float d) {
  asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%0, %1};\n\tmov.b64 y, {%2, %3};\n\tadd.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}"
      : "+f"(a), "+f"(b)
      : "f"(c), "f"(d));
}
__device__ __forceinline__ uint4 lds128(unsigned addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ uint2 lds64(unsigned addr) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ unsigned lds32(unsigned addr) {
  unsigned v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void sts32(unsigned addr, unsigned a) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(a) : "memory"); }
__device__ __forceinline__ void sts64(unsigned addr, unsigned a, unsigned b) {
  asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ void sts128(unsigned addr, unsigned a, unsigned b, unsigned c, unsigned d) {
  asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ unsigned min_f16x2(unsigned a, unsigned b) {
  unsigned d;
  asm("min.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
// both halves between the largest finite values; NaN stays NaN
__device__ __forceinline__ unsigned finite_f16x2(unsigned a) {
  unsigned d;
  asm("min.NaN.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(kMaxFinite));
  asm("max.NaN.f16x2 %0, %1, %2;" : "=r"(d) : "r"(d), "r"(kMaxFinite | 0x80008000u));
  return d;
}
__device__ __forceinline__ unsigned prmt(unsigned a, unsigned sel) { return __byte_perm(a, 0u, sel); }

__device__ __forceinline__ float act_f(float v, int act) {
  if (act != GI_ACT_NONE) v = fmaxf(v, 0.0f);
  if (act == GI_ACT_RELU6) v = fminf(v, 6.0f);
  return v;
}

__host__ __device__ __forceinline__ int div_by(int i, unsigned mul) {
#ifdef __CUDA_ARCH__
  return static_cast<int>(__umulhi(static_cast<unsigned>(i), mul));
#else
  return static_cast<int>((static_cast<uint64_t>(i) * mul) >> 32);
#endif
}

// division of a small number by d > 1 is one high multiplication (div_by)
inline unsigned magic(uint64_t d) { return static_cast<unsigned>(std::min<uint64_t>(0xffffffffull, (0xffffffffull + d) / d)); }

// The A operand that a bias in four parts (bias_split.h) is multiplied by: what lane t of a quad holds, two halves.
__host__ __device__ constexpr unsigned ones_word(int t) { return t == 0 ? 0x10003c00u : t == 1 ? 0x78000004u : 0u; }  // 1, 2^-11; 2^-22, 2^15

// channel of column n of fragment f in 16-channel block j: lane t of a quad holds the 4 channels of slice 4 j + t
inline int channel_of(int j, int f, int n) { return 16 * j + 4 * (n >> 1) + 2 * f + (n & 1); }

}  // namespace frag
}  // namespace gi
