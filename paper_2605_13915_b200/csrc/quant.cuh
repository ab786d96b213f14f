// Element-wise INT8 quantisation shared by the decomposition kernel and the attention kernels' query set-up.
#pragma once
#include <cuda_runtime.h>

namespace msd {

// clamp(rne(fl(v / scale)), -128, 127), bit for bit, without paying for an IEEE division per element:
// c = rne(v * (1/scale)) can differ from the rounded true quotient only when the quotient sits within a few ulps of a
// half-integer: |v*inv - v/scale| <= 127 * 2^-23 < 2^-16, so whenever the exact remainder v - scale*c is further than
// 2^-14 * scale from +-scale/2, c is the nearest integer of the true quotient with a margin that the quotient's own
// FP32 rounding (< 2^-17) cannot cross.  The rare elements inside that band take the true division.
__device__ __forceinline__ int quant_i8(float v, float scale, float inv_scale) {
  const float c = rintf(v * inv_scale);
  const float rem = __fmaf_rn(-scale, c, v);                  // exact for |c| <= 2^7 and BF16-derived inputs
  const float dist = fabsf(fabsf(rem) - 0.5f * scale);
  int q;
  if (dist > scale * 6.103515625e-05f && fabsf(c) <= 127.0f) q = __float2int_rn(c);
  else q = __float2int_rn(__fdiv_rn(v, scale));               // true division, round-half-to-even
  return max(-128, min(127, q));
}

// ---- 8 BF16 values (a 128-bit word) at a time: the unit of the row decomposition (Alg. 1 lines 1-5) ----
__device__ __forceinline__ float bf16lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

__device__ __forceinline__ float unit_absmax(const uint4& a) {
  // |x| as BF16 bits is monotone in the value: both halves of a word are compared at once
  const uint32_t m2 = __vmaxu2(__vmaxu2(a.x & 0x7FFF7FFFu, a.y & 0x7FFF7FFFu), __vmaxu2(a.z & 0x7FFF7FFFu, a.w & 0x7FFF7FFFu));
  return __uint_as_float(max(m2 & 0xFFFFu, m2 >> 16) << 16);
}

// rint(fl(v / scale)) when the quotient lies within 2^-14 of a half-integer: `c` is the integer our estimate rounded to.
// h is that half-integer and d = v - scale * h its exact distance (in units of the scale).  The IEEE quotient rounds to h
// itself - a tie, which goes to the even neighbour - when |d / scale| is at most half a unit in the last place of h;
// otherwise the sign of d says on which side it stays.
__device__ __forceinline__ float resolve_near_tie(float v, float scale, float c, float rem) {
  const float half = copysignf(0.5f, rem);
  const float h = c + half;
  const float d = __fmaf_rn(-scale, h, v);
  const float half_ulp = __uint_as_float(__float_as_uint(h) & 0x7F800000u) * 5.9604644775390625e-08f * scale;   // 2^(e-24) * scale
  const bool tie = fabsf(d) <= half_ulp;
  const bool odd = (__float2int_rn(c) & 1) != 0;
  const bool beyond = (d > 0.0f) == (half > 0.0f);
  return (tie ? odd : beyond) ? c + 2.0f * half : c;
}

// Scales for which the bounds below hold (no denormals, nothing infinite); others go through quant_i8's division.
__device__ __forceinline__ bool unit_scales_ok(float alpha, float beta) { return beta > 1e-30f && alpha < 1e30f; }

// Two FP32 values per instruction (sm_100): halves the issue slots of the quantisation, which are what it is made of.
__device__ __forceinline__ uint64_t pack_f32x2(float lo, float hi) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ float2 unpack_f32x2(uint64_t v) {
  float2 f;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
  return f;
}
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add_f32x2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// Two-pass quantisation of 4 values; returns the packed codes of both passes (Eqs. x1, residual, x2).
// About 9 instructions per value: adding 1.5 * 2^23 inside the FMA that multiplies by the reciprocal rounds the quotient
// half-to-even and leaves the code in the low byte of the sum, and the exact residual of a pass (which the second pass
// needs anyway) also says whether the code can be trusted.  The product v * inv (exact inside the FMA, inv within 2^-24
// of 1/scale) is within 2^-17 of the true quotient, and the IEEE quotient rounds by at most 2^-18 more, so unless a
// residual lies within 2^-16 * scale of scale/2 the code equals that of the true division; one look at the largest
// residuals decides for all 4 values.  BF16 rows whose maximum has a small odd part hit exact ties often (v and the
// maximum are short integers; one warp in six has such a value among its 128), so the other case must not be slow either:
// it settles every value without a division.
__device__ __forceinline__ void quad_quantize(uint32_t w0, uint32_t w1, float alpha, float beta, float inv_alpha, float inv_beta,
                                              uint32_t& p1, uint32_t& p2) {
  constexpr float kMagic = 12582912.0f;                 // 1.5 * 2^23
  constexpr float kHalf = 0.5f - 1.52587890625e-05f;    // 1/2 - 2^-16
  const uint64_t magic2 = pack_f32x2(kMagic, kMagic), minus2 = pack_f32x2(-kMagic, -kMagic);
  const uint64_t ia2 = pack_f32x2(inv_alpha, inv_alpha), ib2 = pack_f32x2(inv_beta, inv_beta);
  const uint64_t na2 = pack_f32x2(-alpha, -alpha), nb2 = pack_f32x2(-beta, -beta);
  float m1[4], m2[4];
  float far1 = 0.0f, far2 = 0.0f;
#pragma unroll
  for (int e = 0; e < 4; e += 2) {
    const uint32_t w = e == 0 ? w0 : w1;
    const uint64_t v = pack_f32x2(bf16lo(w), bf16hi(w));
    const uint64_t q1 = fma_f32x2(v, ia2, magic2);
    const uint64_t r = fma_f32x2(na2, add_f32x2(q1, minus2), v);
    const uint64_t q2 = fma_f32x2(r, ib2, magic2);
    const uint64_t t = fma_f32x2(nb2, add_f32x2(q2, minus2), r);
    const float2 rf = unpack_f32x2(r), tf = unpack_f32x2(t), q1f = unpack_f32x2(q1), q2f = unpack_f32x2(q2);
    far1 = fmaxf(far1, fmaxf(fabsf(rf.x), fabsf(rf.y)));
    far2 = fmaxf(far2, fmaxf(fabsf(tf.x), fabsf(tf.y)));
    m1[e] = q1f.x; m1[e + 1] = q1f.y;
    m2[e] = q2f.x; m2[e + 1] = q2f.y;
  }
  if (!(far1 < kHalf * alpha && far2 < kHalf * beta)) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const uint32_t w = e < 2 ? w0 : w1;
      const float v = (e & 1) ? bf16hi(w) : bf16lo(w);
      float c = m1[e] - kMagic;
      float r = __fmaf_rn(-alpha, c, v);
      if (fabsf(r) >= kHalf * alpha) c = resolve_near_tie(v, alpha, c, r);
      m1[e] = c + kMagic;
      r = __fmaf_rn(-alpha, c, v);
      c = __fmaf_rn(r, inv_beta, kMagic) - kMagic;
      const float t = __fmaf_rn(-beta, c, r);
      if (fabsf(t) >= kHalf * beta) c = resolve_near_tie(r, beta, c, t);
      m2[e] = c + kMagic;
    }
  }
  p1 = __byte_perm(__byte_perm(__float_as_uint(m1[0]), __float_as_uint(m1[1]), 0x0040),
                   __byte_perm(__float_as_uint(m1[2]), __float_as_uint(m1[3]), 0x0040), 0x5410);
  p2 = __byte_perm(__byte_perm(__float_as_uint(m2[0]), __float_as_uint(m2[1]), 0x0040),
                   __byte_perm(__float_as_uint(m2[2]), __float_as_uint(m2[3]), 0x0040), 0x5410);
}

__device__ __forceinline__ void unit_quantize(const uint4& a, float alpha, float beta, float inv_alpha, float inv_beta, uint2& o1,
                                              uint2& o2) {
  quad_quantize(a.x, a.y, alpha, beta, inv_alpha, inv_beta, o1.x, o2.x);
  quad_quantize(a.z, a.w, alpha, beta, inv_alpha, inv_beta, o1.y, o2.y);
}

// The same for any scales, a zero row included: what does not fit the fast path goes value by value with true divisions.
__device__ __forceinline__ void unit_quantize_any(const uint4& a, float alpha, float beta, float inv_alpha, float inv_beta, uint2& o1,
                                                  uint2& o2) {
  if (unit_scales_ok(alpha, beta)) {
    unit_quantize(a, alpha, beta, inv_alpha, inv_beta, o1, o2);
    return;
  }
  uint32_t w[4] = {a.x, a.y, a.z, a.w};
  unsigned long long p1 = 0, p2 = 0;
#pragma unroll 1
  for (int e = 0; e < 8; ++e) {
    const float v = bf16lo(w[0]);
    int c1 = 0, c2 = 0;
    if (alpha > 0.0f) {
      c1 = quant_i8(v, alpha, inv_alpha);
      const float r = __fmaf_rn(-alpha, static_cast<float>(c1), v);
      if (beta > 0.0f) c2 = quant_i8(r, beta, inv_beta);
    }
    p1 |= static_cast<unsigned long long>(c1 & 0xFF) << (8 * e);
    p2 |= static_cast<unsigned long long>(c2 & 0xFF) << (8 * e);
    // the next value moves into the low half of w[0]
    w[0] = __funnelshift_r(w[0], w[1], 16); w[1] = __funnelshift_r(w[1], w[2], 16); w[2] = __funnelshift_r(w[2], w[3], 16); w[3] >>= 16;
  }
  o1 = make_uint2(static_cast<uint32_t>(p1), static_cast<uint32_t>(p1 >> 32));
  o2 = make_uint2(static_cast<uint32_t>(p2), static_cast<uint32_t>(p2 >> 32));
}

}  // namespace msd
