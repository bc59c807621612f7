// Exact split products on the bf16 tensor cores (Ozaki's scheme) for the
// double-float kernels: a scaled double-float value in (-1, 1) is written as
// six bf16 slices on the grids 2^(-7-8k); products of slices are exact in
// bf16 x bf16 -> FP32, and the products whose slice indices sum to u share
// one power-of-two grid, so their FP32 sum is exact while it stays below
// 2^24 units.  Used by the block updates of the double-float and FP32 kinds
// (blas_rows.cu) and by their Grams (blas_tc.cu).
#pragma once
#include "common.cuh"

namespace bcg {
namespace ozaki {

__device__ __forceinline__ float rnd_grid(float x, float c) {  // x to the grid ulp(c)
  return __fsub_rn(__fadd_rn(x, c), c);
}

// six bf16-exact slices of a scaled double-float value h + l, |h + l| < 1:
// slice k on the grid 2^(-7-8k) (rounding to nearest by adding and removing
// c_k = 1.5 * 2^(16-8k)); every step but the (hi remainder + lo) sum is exact
__device__ __forceinline__ void split6(float h, float l, float (&s)[6]) {
  s[0] = rnd_grid(h, 98304.f);  // 1.5 * 2^16
  float r = __fsub_rn(h, s[0]);
  s[1] = rnd_grid(r, 384.f);  // 1.5 * 2^8
  r = __fsub_rn(r, s[1]);
  s[2] = rnd_grid(r, 1.5f);
  r = __fsub_rn(r, s[2]);
  r = __fadd_rn(r, l);
  s[3] = rnd_grid(r, 0.005859375f);  // 1.5 * 2^-8
  r = __fsub_rn(r, s[3]);
  s[4] = rnd_grid(r, 2.288818359375e-05f);  // 1.5 * 2^-16
  r = __fsub_rn(r, s[4]);
  s[5] = rnd_grid(r, 8.940696716308594e-08f);  // 1.5 * 2^-24
}

// seven slices (56 bits): as split6, with the remainder behind the fourth slice
// kept exact, so that a value far below its scale keeps all its 48 bits
__device__ __forceinline__ void split7(float h, float l, float (&s)[7]) {
  s[0] = rnd_grid(h, 98304.f);
  float r = __fsub_rn(h, s[0]);
  s[1] = rnd_grid(r, 384.f);
  r = __fsub_rn(r, s[1]);
  s[2] = rnd_grid(r, 1.5f);
  r = __fsub_rn(r, s[2]);
  s[3] = rnd_grid(__fadd_rn(r, l), 0.005859375f);
  r = __fadd_rn(__fsub_rn(r, s[3]), l);
  s[4] = rnd_grid(r, 2.288818359375e-05f);
  r = __fsub_rn(r, s[4]);
  s[5] = rnd_grid(r, 8.940696716308594e-08f);
  s[6] = rnd_grid(__fsub_rn(r, s[5]), 3.4924596548080444e-10f);  // 1.5 * 2^-32
}

// four slices (32 bits) of a scaled FP32 value, on the first four grids
__device__ __forceinline__ void split4(float h, float (&s)[4]) {
  s[0] = rnd_grid(h, 98304.f);
  h = __fsub_rn(h, s[0]);
  s[1] = rnd_grid(h, 384.f);
  h = __fsub_rn(h, s[1]);
  s[2] = rnd_grid(h, 1.5f);
  s[3] = rnd_grid(__fsub_rn(h, s[2]), 0.005859375f);
}

// (lo, hi) -> one register of two bf16 (lo in the low half: the element
// with the smaller k of an MMA fragment pair); exact for slice values
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

// the slices of a stored complex number v times the scale sc, slice s as one
// register (re, im); mag: its largest component, which the scale follows
template <class S>
struct SliceKind;
template <>
struct SliceKind<StoreDF> {
  static constexpr int NSL = 6;
  static __device__ __forceinline__ float4 zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
  static __device__ __forceinline__ float mag(float4 v) { return fmaxf(fabsf(v.x), fabsf(v.y)); }
  static __device__ __forceinline__ void slices(float4 v, float sc, uint32_t (&w)[NSL]) {
    float re[6], im[6];
    split6(__fmul_rn(v.x, sc), __fmul_rn(v.z, sc), re);
    split6(__fmul_rn(v.y, sc), __fmul_rn(v.w, sc), im);
#pragma unroll
    for (int s = 0; s < NSL; ++s) w[s] = pack_bf16(re[s], im[s]);
  }
};
template <>
struct SliceKind<StoreF32> {
  static constexpr int NSL = 4;
  static __device__ __forceinline__ float2 zero() { return make_float2(0.f, 0.f); }
  static __device__ __forceinline__ float mag(float2 v) { return fmaxf(fabsf(v.x), fabsf(v.y)); }
  static __device__ __forceinline__ void slices(float2 v, float sc, uint32_t (&w)[NSL]) {
    float re[4], im[4];
    split4(__fmul_rn(v.x, sc), re);
    split4(__fmul_rn(v.y, sc), im);
#pragma unroll
    for (int s = 0; s < NSL; ++s) w[s] = pack_bf16(re[s], im[s]);
  }
};

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// smallest e with |v| < 2^e for the non-negative float with bit pattern b,
// clamped to [-120, 120] (0 and denormals give -126 -> -120; inf/NaN 120,
// which keeps them non-finite after scaling)
__device__ __forceinline__ int pow2_above(unsigned b) {
  const int e = (int)((b >> 23) & 0xffu) - 126;
  return e < -120 ? -120 : e > 120 ? 120 : e;
}
__device__ __forceinline__ float exp2i(int e) { return __int_as_float((e + 127) << 23); }

// h + l += d
__device__ __forceinline__ void exact_add(float& h, float& l, float d) {
  float s, e;
  two_sum(h, d, s, e);
  h = s;
  l = __fadd_rn(l, e);
}

// D = sum_u D_u in double-float.  The leading slices are short (a value is some
// 2^-3 of its scale) and the others are not, so D_3 is still about 2^-20 of the
// sum: D_0 .. D_3 are added exactly, the rest fits one FP32 number.
__device__ __forceinline__ dfacc combine6(float d0, float d1, float d2, float d3, float d4,
                                          float d5) {
  float h = d0, l = __fadd_rn(d5, d4);
  exact_add(h, l, d1);
  exact_add(h, l, d2);
  exact_add(h, l, d3);
  const float s = __fadd_rn(h, l);  // fast two-sum: |h| >= |l|
  return {s, __fsub_rn(l, __fsub_rn(s, h))};
}

}  // namespace ozaki
}  // namespace bcg
