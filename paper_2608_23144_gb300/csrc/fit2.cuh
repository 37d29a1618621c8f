// fit2.cuh — the P_F fit on packed pairs, shared by the searches: reciprocals
// of the LDL^T pivots of several pairs, the quantiser and gain with an
// undoubled Gram, and the quantiser that also returns the codes.
#pragma once

#include "common.cuh"

namespace awsrc {

__device__ __forceinline__ float2 neg2(float2 v) { return make_float2(-v.x, -v.y); }

__device__ __forceinline__ bool pivot_ok(float d) { return d > 0.0f && d <= 3.402823466e38f; }

// Pivots k of NP pairs: the validity of each (pivot_ok) and rcp_rn of each
// component. When every component of the warp's pairs is in [2^-125, 2^125)
// (positive, normal, finite: hence valid), the hardware approximation and
// Markstein's fused correction y + y (1 - x y) as two packed fmas (each
// component rounds as the scalar form does); otherwise, in a branch the lanes
// take together, the exact checks and __frcp_rn for the components outside.
template <int NP>
__device__ __forceinline__ void pivots_rcp(const float2* x, float2* r, bool* okx, bool* oky) {
  bool fx[NP], fy[NP], in = true;
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    float yx, yy;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(yx) : "f"(x[j].x));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(yy) : "f"(x[j].y));
    const float2 y = make_float2(yx, yy);
    const float2 e = __ffma2_rn(make_float2(-x[j].x, -x[j].y), y, make_float2(1.0f, 1.0f));
    r[j] = __ffma2_rn(y, e, y);
    fx[j] = __float_as_uint(x[j].x) - 0x01000000u < 0x7D000000u - 0x01000000u;
    fy[j] = __float_as_uint(x[j].y) - 0x01000000u < 0x7D000000u - 0x01000000u;
    in = in && fx[j] && fy[j];
  }
  if (__any_sync(__activemask(), !in)) {
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      okx[j] = okx[j] && pivot_ok(x[j].x);
      oky[j] = oky[j] && pivot_ok(x[j].y);
      if (!fx[j]) r[j].x = __frcp_rn(x[j].x);
      if (!fy[j]) r[j].y = __frcp_rn(x[j].y);
    }
  }
}

// quant_gain_fast2 with the off-diagonal G as it is rather than doubled: each
// off-diagonal term takes q_p * (2 q_r), the exact double of q_p q_r (codes
// are small integers), so that fma(q_p (2 q_r), G, Qq) rounds the same exact
// value as fma(q_p q_r, 2 G, Qq) (|G| <= 2^38 on the tile domain: 2 G is exact).
template <int P>
__device__ __forceinline__ float2 quant_gain_fast2_g(const Prm& pr, const float2* alpha, const float2* bv,
                                                     float2 gd, const float2* Goff) {
  float m0 = fabsf(alpha[0].x), m1 = fabsf(alpha[0].y);
#pragma unroll
  for (int p = 1; p < P; ++p) {
    m0 = fmaxf(m0, fabsf(alpha[p].x));
    m1 = fmaxf(m1, fabsf(alpha[p].y));
  }
  // an amax out of range gets a gain of -inf below, whatever its bits give
  const uint32_t ab0 = __float_as_uint(m0), ab1 = __float_as_uint(m1);
  const bool in0 = fast_scale_in_range(ab0), in1 = fast_scale_in_range(ab1);
  const uint32_t s0 = fast_scale_bits(pr, ab0), s1 = fast_scale_bits(pr, ab1);
  const float2 sc = make_float2(__uint_as_float(s0), __uint_as_float(s1));
  const float2 nsc = make_float2(__uint_as_float(s0 | 0x80000000u), __uint_as_float(s1 | 0x80000000u));
  const float2 inv = make_float2(__uint_as_float(0x7F000000u - s0), __uint_as_float(0x7F000000u - s1));
  const float2 magic = make_float2(12582912.0f, 12582912.0f);
  const float2 nmagic = make_float2(-12582912.0f, -12582912.0f);
  float2 q[P], q2[P];
#pragma unroll
  for (int p = 0; p < P; ++p) {
    q[p] = __fadd2_rn(__ffma2_rn(alpha[p], inv, magic), nmagic);
    q2[p] = __fadd2_rn(q[p], q[p]);
  }
  float2 Aq = make_float2(0.0f, 0.0f);
#pragma unroll
  for (int p = 0; p < P; ++p) Aq = __ffma2_rn(q[p], bv[p], Aq);
  float2 Qq = make_float2(0.0f, 0.0f);
#pragma unroll
  for (int p = 0; p < P; ++p) {
    Qq = __ffma2_rn(__fmul2_rn(q[p], q[p]), gd, Qq);
#pragma unroll
    for (int r = p + 1; r < P; ++r) Qq = __ffma2_rn(__fmul2_rn(q[p], q2[r]), Goff[tri(r, p)], Qq);
  }
  const float2 tn = __fmul2_rn(nsc, Qq);
  float2 g = __fmul2_rn(sc, __ffma2_rn(make_float2(2.0f, 2.0f), Aq, tn));
  if (!in0) g.x = -__int_as_float(0x7f800000);
  if (!in1) g.y = -__int_as_float(0x7f800000);
  return g;
}

// Codes of a candidate as signed bytes, code p in byte p: t_p = alpha_p 2^-e +
// 1.5 * 2^23 carries the code's two's complement in its low byte.
template <int P>
__device__ __forceinline__ uint32_t pack_low_bytes(const float* t) {
  uint32_t w = __float_as_uint(t[0]) & 0xFFu;
  if constexpr (P == 2) w = __byte_perm(__float_as_uint(t[0]), __float_as_uint(t[1]), 0x0040) & 0xFFFFu;
  if constexpr (P == 4)
    w = __byte_perm(__byte_perm(__float_as_uint(t[0]), __float_as_uint(t[1]), 0x0040),
                    __byte_perm(__float_as_uint(t[2]), __float_as_uint(t[3]), 0x0040), 0x5410);
  return w;
}

// The fast power-of-two quantiser and gain of a pair (quant_gain_fast2, or
// quant_gain_fast2_g when !DOUBLED: Goff holds 2 G_pq or G_pq), which also
// gives each candidate's codes (cw, P <= 4) and exponent (sf).
template <int P, bool DOUBLED>
__device__ __forceinline__ float2 quant_codes_fast2(const Prm& pr, const float2* alpha, const float2* bv, float2 gd,
                                                    const float2* Goff, uint32_t* cw, int* sf) {
  static_assert(P == 2 || P == 4, "codes are packed for two or four atoms");
  float m0 = fabsf(alpha[0].x), m1 = fabsf(alpha[0].y);
#pragma unroll
  for (int p = 1; p < P; ++p) {
    m0 = fmaxf(m0, fabsf(alpha[p].x));
    m1 = fmaxf(m1, fabsf(alpha[p].y));
  }
  const uint32_t ab0 = __float_as_uint(m0), ab1 = __float_as_uint(m1);
  const bool in0 = fast_scale_in_range(ab0), in1 = fast_scale_in_range(ab1);
  const uint32_t s0 = fast_scale_bits(pr, ab0), s1 = fast_scale_bits(pr, ab1);
  const float2 sc = make_float2(__uint_as_float(s0), __uint_as_float(s1));
  const float2 nsc = make_float2(__uint_as_float(s0 | 0x80000000u), __uint_as_float(s1 | 0x80000000u));
  const float2 inv = make_float2(__uint_as_float(0x7F000000u - s0), __uint_as_float(0x7F000000u - s1));
  const float2 magic = make_float2(12582912.0f, 12582912.0f);
  const float2 nmagic = make_float2(-12582912.0f, -12582912.0f);
  float2 q[P], q2[P];
  float tx[P], ty[P];
#pragma unroll
  for (int p = 0; p < P; ++p) {
    const float2 t = __ffma2_rn(alpha[p], inv, magic);
    tx[p] = t.x;
    ty[p] = t.y;
    q[p] = __fadd2_rn(t, nmagic);
    q2[p] = DOUBLED ? q[p] : __fadd2_rn(q[p], q[p]);
  }
  cw[0] = pack_low_bytes<P>(tx);
  cw[1] = pack_low_bytes<P>(ty);
  sf[0] = (int)(s0 >> 23) - 127;
  sf[1] = (int)(s1 >> 23) - 127;
  float2 Aq = make_float2(0.0f, 0.0f);
#pragma unroll
  for (int p = 0; p < P; ++p) Aq = __ffma2_rn(q[p], bv[p], Aq);
  float2 Qq = make_float2(0.0f, 0.0f);
#pragma unroll
  for (int p = 0; p < P; ++p) {
    Qq = __ffma2_rn(__fmul2_rn(q[p], q[p]), gd, Qq);
#pragma unroll
    for (int r = p + 1; r < P; ++r) Qq = __ffma2_rn(__fmul2_rn(q[p], q2[r]), Goff[tri(r, p)], Qq);
  }
  const float2 tn = __fmul2_rn(nsc, Qq);
  float2 g = __fmul2_rn(sc, __ffma2_rn(make_float2(2.0f, 2.0f), Aq, tn));
  if (!in0) g.x = -__int_as_float(0x7f800000);
  if (!in1) g.y = -__int_as_float(0x7f800000);
  return g;
}

}  // namespace awsrc
