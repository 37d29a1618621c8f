// search_mma.cuh — the seed search of Sec. 3.2 for the shapes without a kernel
// of their own: C in {16, 32, 64, 128} and P in {2, 4}, both variants and both
// scale modes (C = 64, P = 4 has the tcgen05 searches). These are the paper's
// operating points, C = 128, P = 2, S = 2 (U) and C = 16, P = 4, S = 16 (P_F):
// few seeds per tile, so a tile's weights are read once for a handful of
// candidates and the kernel sits between the HBM and the issue rate.
//
// The +-1 correlations of a tile with the seeds' atoms (and, P_F, of its D with
// the atom products) are exact integer sums on the tile's fixed-point grid,
// here as mma.sync m16n8k16 on exact FP16 halves X = 2048 hi + lo (|hi|, |lo| <=
// 1024, so every partial sum of C <= 128 terms is an integer below 2^18 and
// binary32 accumulation is exact in any order). The register form fits these
// shapes better than tcgen05: K = C is one to eight k-steps, a warp makes its 16
// tiles' A operand directly from the loaded weights without shared memory, and
// the sums arrive in the registers of the thread that scores them, where TMEM
// would cost a round trip per 16 seeds. The contraction is a few percent of the
// time either way.
//
// A warp takes 16 consecutive tiles. MMA column n is seed n of a group of eight,
// one MMA chain per atom (and product), so thread (g, q) = (lane / 4, lane % 4)
// holds all sums of seeds 2q, 2q + 1 for tiles g and g + 8: two seed pairs, which
// it fits as packed f32x2 streams side by side. The order of the C inputs along
// K is free as long as A and B agree: thread q takes 4 consecutive inputs of
// each k-step (8 of each two), so it loads its inputs as vectors. The B operand
// of a chunk of seeds is built once per block from the masks, in fragment order.
// Blocks are persistent, and each thread copies its next tiles' weights into its
// own shared-memory slots (cp.async) while it scores the present ones.
//
// Measured on the MLP projections of a 3B-shaped layer (67.6 M weights), whole
// encode call, against the scalar search that served these shapes before
// (nibble tables in shared memory, one lane per four seeds): P_F (16, 4, 4, 16)
// 1833 -> 552 us, U (128, 2, 4, 2) 347 -> 98 us. Loading the next tiles without the
// copies: 752 and 181 us (40% of the stalls were global loads); with the element
// types tested at run time: 577 and 121 us. P_F is bound by issue (60% of slots; half
// of the instructions stage and split the inputs, the rest score), U by the latency
// of its loads and the 16 us of table kernels before it.
#pragma once

#include <algorithm>

#include "fit2.cuh"
#include "internal.h"

namespace awsrc {
namespace {

constexpr int kMmaWarps = 8;
constexpr int kMmaTiles = 16 * kMmaWarps;        // tiles per block and pass
constexpr size_t kMmaTableBytes = 40 * 1024;     // B fragments of one seed chunk
constexpr size_t kMmaSmemMax = 226 * 1024;       // dynamic shared memory of one block
constexpr float kMagic = 12582912.0f;            // 1.5 * 2^23

__host__ __device__ constexpr int mma_slots(int P, int VAR) {
  return P + (VAR == AWSRC_VARIANT_PF ? P * (P - 1) / 2 : 0);
}
// groups of eight seeds whose B fragments fit in shared memory
__host__ __device__ constexpr int mma_groups(int P, int VAR, int KS) {
  const int n = (int)(kMmaTableBytes / ((size_t)mma_slots(P, VAR) * KS * 256));
  return n < 1 ? 1 : n;
}

// blocks per SM that the registers allow
__host__ __device__ constexpr int mma_per_sm(int VAR, int KS) { return VAR == AWSRC_VARIANT_PF && KS >= 4 ? 1 : 2; }

__device__ __forceinline__ float ninf() { return -__int_as_float(0x7f800000); }

// D += A B on m16n8k16 (FP16 operands, binary32 accumulation).
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint2 b) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
}

__device__ __forceinline__ uint32_t half2_bits(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

// First input of thread q's run of 4 in k-step ks: runs of 8 over two k-steps
// when there are two (16-byte BF16 loads), else runs of 4.
template <int KS>
__device__ __forceinline__ int mma_input(int ks, int q) {
  return KS == 1 ? 4 * q : 32 * (ks >> 1) + 8 * q + 4 * (ks & 1);
}

// V = 4 or 8 consecutive elements as floats, from their bytes in memory of any
// space (16- or 8-byte aligned).
template <int V>
__device__ __forceinline__ void vec_elems(const void* b, bool bf16, float* out) {
  if (!bf16) {
#pragma unroll
    for (int i = 0; i < V; i += 4) {
      const float4 f = *reinterpret_cast<const float4*>(static_cast<const float*>(b) + i);
      out[i] = f.x; out[i + 1] = f.y; out[i + 2] = f.z; out[i + 3] = f.w;
    }
    return;
  }
  uint32_t w[V / 2];
  if constexpr (V == 8) {
    const uint4 u = *static_cast<const uint4*>(b);
    w[0] = u.x; w[1] = u.y; w[2] = u.z; w[3] = u.w;
  } else {
    const uint2 u = *static_cast<const uint2*>(b);
    w[0] = u.x; w[1] = u.y;
  }
#pragma unroll
  for (int i = 0; i < V / 2; ++i) {
    out[2 * i] = __uint_as_float(w[i] << 16);
    out[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
  }
}

// How a launch's weights reach the registers.
enum : int {
  kLoadScalar = 0,  // some array is not 16-byte aligned: element by element
  kLoadVector = 1,  // vectors from global memory
  kLoadAsync = 2    // vectors through the thread's own shared-memory slots, copied one item ahead
};

// The slots of one thread, in 16-byte columns [slot][thread of the warp]: per
// row half, vector v (of NV) and array (W, W0, then F), 16 or 32 bytes each.
struct MmaSlots {
  int w, w0, f, per_vec;  // 16-byte slots of the arrays' vectors: offsets and total
};

template <int V>
__host__ __device__ inline MmaSlots mma_slots_of(int wbytes, int w0bytes, bool pf) {
  const int a = (V * wbytes + 15) / 16, b = (V * w0bytes + 15) / 16, c = pf ? V * 4 / 16 : 0;
  return {0, a, a + b, a + b + c};
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async8(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}

// n = 8, 16 or 32 bytes into slot `dst` of this thread (slots are 512 bytes apart).
__device__ __forceinline__ void copy_slots(uint32_t dst, const void* src, int n) {
  if (n == 8) {
    cp_async8(dst, src);
  } else {
    cp_async16(dst, src);
    if (n == 32) cp_async16(dst + 512u, static_cast<const char*>(src) + 16);
  }
}

// V elements from slots written by copy_slots.
template <int V>
__device__ __forceinline__ void slot_elems(const unsigned char* slot, bool bf16, float* out) {
  if (V == 8 && !bf16) {
    vec_elems<4>(slot, false, out);
    vec_elems<4>(slot + 512, false, out + 4);
  } else {
    vec_elems<V>(slot, bf16, out);
  }
}

// Exact FP16 halves of four inputs on the grid 2^q (inv = 2^-q, 0 for a zero
// vector): X = rint(x inv), hi = rint(X / 2048), lo = X - 2048 hi, all exact in
// binary32 (|X| <= 2^21). Accumulates the halves' sums into shi, slo.
__device__ __forceinline__ void split4(const float* x, float inv, uint32_t* hi, uint32_t* lo, float2& shi,
                                       float2& slo) {
  const float2 m = make_float2(kMagic, kMagic), nm = make_float2(-kMagic, -kMagic);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const float2 X = __fadd2_rn(__ffma2_rn(make_float2(x[2 * i], x[2 * i + 1]), make_float2(inv, inv), m), nm);
    const float2 h = __fadd2_rn(__ffma2_rn(X, make_float2(0x1p-11f, 0x1p-11f), m), nm);
    const float2 l = __ffma2_rn(h, make_float2(-2048.0f, -2048.0f), X);
    hi[i] = half2_bits(h.x, h.y);
    lo[i] = half2_bits(l.x, l.y);
    shi = __fadd2_rn(shi, h);
    slo = __fadd2_rn(slo, l);
  }
}

// Largest magnitude of three, ignoring NaN, and propagating it.
__device__ __forceinline__ float max3_abs(float a, float b, float c) {
  float r;
  asm("{\n\t.reg .f32 y, z;\n\tabs.f32 y, %2;\n\tabs.f32 z, %3;\n\tmax.f32 %0, %1, y, z;\n\t}"
      : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float max3_abs_nan(float a, float b, float c) {
  float r;
  asm("{\n\t.reg .f32 y, z;\n\tabs.f32 y, %2;\n\tabs.f32 z, %3;\n\tmax.NaN.f32 %0, %1, y, z;\n\t}"
      : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

__device__ __forceinline__ float quad_max(float v) {
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
  return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 2));
}
__device__ __forceinline__ float quad_sum(float v) {
  v = __fadd_rn(v, __shfl_xor_sync(0xffffffffu, v, 1));
  return __fadd_rn(v, __shfl_xor_sync(0xffffffffu, v, 2));
}

// Where a thread's tile lies: its module, tile within the module and column block.
struct MmaPos {
  int mi;
  uint32_t lt, cb;
};

// Tile t (below the launch's last) by 32-bit arithmetic: a call has fewer than
// 2^32 tiles. mi0: a module at or before the tile's.
__device__ __forceinline__ MmaPos mma_pos(const LaunchDesc& ld, int64_t t, int mi0) {
  MmaPos p;
  p.mi = mi0;
  while (p.mi + 1 < ld.n && t >= ld.m[p.mi + 1].tile_off) ++p.mi;
  p.lt = (uint32_t)(t - ld.m[p.mi].tile_off);
  p.cb = p.lt % (uint32_t)ld.m[p.mi].n_cb;
  return p;
}

// The same for tile t, `d` tiles past the one at p0 (one more division only where
// the step leaves the module or passes a row's end twice).
__device__ __forceinline__ MmaPos mma_pos_after(const LaunchDesc& ld, const MmaPos& p0, int64_t t, uint32_t d) {
  const ModDesc& md = ld.m[p0.mi];
  const uint32_t n_cb = (uint32_t)md.n_cb;
  MmaPos p{p0.mi, p0.lt + d, p0.cb + d};
  if (p.cb >= n_cb) p.cb -= n_cb;
  if (p.cb >= n_cb || (p0.mi + 1 < ld.n && t >= ld.m[p0.mi + 1].tile_off)) p = mma_pos(ld, t, p0.mi);
  return p;
}

// What the scoring of one tile needs besides its sums.
struct MmaRow {
  float tqc;                        // 2^qy c
  float tqdc, gd, diag, invd0;      // P_F: 2^qd c2, G_pp, G_pp + eps, 1 / D_0
  uint32_t pair0;                   // U: first entry (float4) of the column block's paired factors
  bool ok;
};

// Starts the copies of one tile's inputs into this thread's slots.
template <int VAR, int KS, bool BF>
__device__ __forceinline__ void mma_copy(const LaunchDesc& ld, const MmaPos& p, int h, int q, const MmaSlots& sl,
                                         uint32_t slots) {
  constexpr int V = KS == 1 ? 4 : 8, NV = 4 * KS / V;
  const ModDesc& md = ld.m[p.mi];
  const int wb = !BF && md.w_dtype == AWSRC_DTYPE_F32 ? 4 : 2, w0b = !BF && md.w0_dtype == AWSRC_DTYPE_F32 ? 4 : 2;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const uint64_t e = (uint64_t)p.lt * (uint32_t)(16 * KS) + (uint32_t)mma_input<KS>(v * (V / 4), q);
    const uint32_t d = slots + (uint32_t)((h * NV + v) * sl.per_vec) * 512u;
    copy_slots(d + (uint32_t)sl.w * 512u, static_cast<const char*>(md.W) + e * wb, V * wb);
    copy_slots(d + (uint32_t)sl.w0 * 512u, static_cast<const char*>(md.W0) + e * w0b, V * w0b);
    if constexpr (VAR == AWSRC_VARIANT_PF) copy_slots(d + (uint32_t)sl.f * 512u, md.fisher + e, V * 4);
  }
}

// Takes one tile's inputs (this thread's 4 KS of C), forms y = d r (and d) on
// the tile's grid and writes the A fragments of row half `h` (rows g or g + 8).
template <int P, int VAR, int KS, bool BF>
__device__ __forceinline__ void mma_stage(const Prm& pr, const LaunchDesc& ld, const MmaPos& p, bool in, int h, int q,
                                          int mode, const MmaSlots& sl, const unsigned char* slots,
                                          uint32_t (*yh)[4], uint32_t (*yl)[4], uint32_t (*dh)[4], uint32_t (*dl)[4],
                                          MmaRow& row) {
  constexpr bool PF = VAR == AWSRC_VARIANT_PF;
  constexpr int V = KS == 1 ? 4 : 8, NV = 4 * KS / V;
  float y[4 * KS], d[PF ? 4 * KS : 1];
  // |r| and |d| over the tile, NaN kept: the tile's domain check is three compares
  float my = 0.0f, mr = 0.0f, dmax = 0.0f, dmin = 0.0f;
  row.pair0 = 0u;
  if (in) {
    const ModDesc& md = ld.m[p.mi];
    const bool bw = BF || md.w_dtype == AWSRC_DTYPE_BF16, bw0 = BF || md.w0_dtype == AWSRC_DTYPE_BF16;
    constexpr uint32_t C = 16 * KS;
    if constexpr (!PF)
      row.pair0 = (uint32_t)(((uint64_t)md.gram_off + (uint64_t)p.cb * (uint32_t)pr.S_pad) >> 1);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const int j = mma_input<KS>(v * (V / 4), q);
      const int64_t e = (int64_t)((uint64_t)p.lt * C + (uint32_t)j);
      float w[V], w0[V], a[V], f[PF ? V : 1];
      if (!BF && mode == kLoadScalar) {
#pragma unroll
        for (int i = 0; i < V; ++i) {
          w[i] = load_elem(md.W, e + i, md.w_dtype);
          w0[i] = load_elem(md.W0, e + i, md.w0_dtype);
          a[i] = md.act[p.cb * C + j + i];
          if constexpr (PF) f[i] = md.fisher[e + i];
        }
      } else {
        if (BF || mode == kLoadAsync) {
          const unsigned char* s = slots + (h * NV + v) * sl.per_vec * 512;
          slot_elems<V>(s + sl.w * 512, bw, w);
          slot_elems<V>(s + sl.w0 * 512, bw0, w0);
          if constexpr (PF) slot_elems<V>(s + sl.f * 512, false, f);
        } else {
          vec_elems<V>(static_cast<const char*>(md.W) + e * (bw ? 2 : 4), bw, w);
          vec_elems<V>(static_cast<const char*>(md.W0) + e * (bw0 ? 2 : 4), bw0, w0);
          if constexpr (PF) vec_elems<V>(md.fisher + e, false, f);
        }
        vec_elems<V>(md.act + p.cb * C + j, false, a);
      }
#pragma unroll
      for (int i = 0; i < V; i += 2) {
        const float2 r = __fadd2_rn(make_float2(w[i], w[i + 1]), make_float2(-w0[i], -w0[i + 1]));
        float2 dv = make_float2(a[i], a[i + 1]);
        if constexpr (PF) {  // three roundings: a packed multiply and add would be contracted to an fma
          dv.x = __fadd_rn(__fmul_rn(md.w_act, a[i]), __fmul_rn(md.w_fisher, f[i]));
          dv.y = __fadd_rn(__fmul_rn(md.w_act, a[i + 1]), __fmul_rn(md.w_fisher, f[PF ? i + 1 : 0]));
        }
        const float2 yv = __fmul2_rn(dv, r);
        y[v * V + i] = yv.x;
        y[v * V + i + 1] = yv.y;
        my = max3_abs(my, yv.x, yv.y);
        mr = max3_abs_nan(mr, r.x, r.y);
        if constexpr (PF) {
          dmax = max3_abs_nan(dmax, dv.x, dv.y);
          dmin = fminf(dmin, fminf(dv.x, dv.y));
          d[v * V + i] = dv.x;
          d[v * V + i + 1] = dv.y;
        }
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < 4 * KS; ++i) {
      y[i] = 0.0f;
      if constexpr (PF) d[i] = 0.0f;
    }
  }
  // in_domain() of every input: |r| <= 2^16 and 0 <= d <= 2^32, no NaN (U: an
  // activation out of range makes its column block's factors invalid)
  bool ok = in && mr <= 65536.0f && dmax <= 4294967296.0f && dmin >= 0.0f;
  // a row's four lanes agree on its grid; a row outside the domain keeps
  // whatever its sums give (rows do not mix) and is dropped at the end
  my = quad_max(my);
  int qy;
  const float iy = fixed_point_inv(my, &qy);
  row.tqc = __fmul_rn(pow2f(qy), pr.c);
  float2 s0 = make_float2(0.0f, 0.0f), s1 = s0;
#pragma unroll
  for (int ks = 0; ks < KS; ++ks) {
    uint32_t hi[2], lo[2];
    split4(y + 4 * ks, iy, hi, lo, s0, s1);
    yh[ks][h] = hi[0]; yh[ks][2 + h] = hi[1];
    yl[ks][h] = lo[0]; yl[ks][2 + h] = lo[1];
  }
  if constexpr (PF) {
    // valid rows: d >= 0, so dmax is the largest |d|
    int qd;
    const float id = fixed_point_inv(quad_max(dmax), &qd);
    float2 sh = make_float2(0.0f, 0.0f), sl2 = sh;
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
      uint32_t hi[2], lo[2];
      split4(d + 4 * ks, id, hi, lo, sh, sl2);
      dh[ks][h] = hi[0]; dh[ks][2 + h] = hi[1];
      dl[ks][h] = lo[0]; dl[ks][2 + h] = lo[1];
    }
    const float two_qd = pow2f(qd);
    // sum of D, rounded once: the halves' sums are exact
    const float sd = __fmaf_rn(2048.0f, quad_sum(__fadd_rn(sh.x, sh.y)), quad_sum(__fadd_rn(sl2.x, sl2.y)));
    row.tqdc = __fmul_rn(two_qd, pr.c2);
    row.gd = __fmul_rn(pr.c2, __fmul_rn(sd, two_qd));
    row.diag = __fadd_rn(row.gd, __fmul_rn(pr.ridge_rel, row.gd));
    row.invd0 = rcp_rn(row.diag);
    ok = ok && pivot_ok(row.diag);
  }
  row.ok = (__ballot_sync(0xffffffffu, ok) >> (threadIdx.x & 28) & 15u) == 15u;
}

// Sums of one atom (or product) of this thread's two tiles and two seeds:
// RN(2048 hi + lo) for (tile g: .x, .y = the seeds) and tile g + 8.
template <int KS>
__device__ __forceinline__ void mma_sums(const uint32_t (*ah)[4], const uint32_t (*al)[4], const uint2* b, float2* u) {
  float hi[4] = {0.0f, 0.0f, 0.0f, 0.0f}, lo[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
  for (int ks = 0; ks < KS; ++ks) {
    const uint2 bf = b[32 * ks];
    mma16816(hi, ah[ks], bf);
    mma16816(lo, al[ks], bf);
  }
  const float2 k = make_float2(2048.0f, 2048.0f);
  u[0] = __ffma2_rn(k, make_float2(hi[0], hi[1]), make_float2(lo[0], lo[1]));
  u[1] = __ffma2_rn(k, make_float2(hi[2], hi[3]), make_float2(lo[2], lo[3]));
}

// Gain, codes and scale field of the two seeds of one tile from the solved fit.
template <int P, bool FAST, bool DOUBLED>
__device__ __forceinline__ float2 mma_gain(const Prm& pr, const float2* alpha, const float2* bv, float2 gd,
                                           const float2* G, uint32_t* cw, int* sf) {
  if constexpr (FAST) {
    return quant_codes_fast2<P, DOUBLED>(pr, alpha, bv, gd, G, cw, sf);
  } else {
    constexpr int NL = P * (P - 1) / 2;
    float g[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      float a[P], b[P], Gs[NL], q[P];
#pragma unroll
      for (int p = 0; p < P; ++p) {
        a[p] = c ? alpha[p].y : alpha[p].x;
        b[p] = c ? bv[p].y : bv[p].x;
      }
#pragma unroll
      for (int i = 0; i < NL; ++i) Gs[i] = c ? G[i].y : G[i].x;
      g[c] = quant_gain<P>(pr, a, b, c ? gd.y : gd.x, Gs, q, &sf[c]);
      cw[c] = 0u;
#pragma unroll
      for (int p = 0; p < P; ++p) cw[c] |= ((uint32_t)(int)q[p] & 0xFFu) << (8 * p);
    }
    return make_float2(g[0], g[1]);
  }
}

// B fragments of the seeds [s0, s0 + 8 ng): entry ((grp * slots + slot) * KS +
// ks) * 32 + lane holds the +-1 of seed 8 grp + lane / 4 at the four inputs
// mma_input(ks, lane % 4) ..; slot p < P: atom p, then (P_F) the products of
// atoms (a, c), c < a, in tri order. Seeds beyond S_pad repeat the last one.
template <int P, int VAR, int KS>
__device__ __forceinline__ void mma_build_table(const Prm& pr, const uint64_t* __restrict__ masks, int s0, int ng,
                                                uint2* tab) {
  constexpr int SL = mma_slots(P, VAR);
  for (int i = threadIdx.x; i < ng * SL * KS * 32; i += 32 * kMmaWarps) {
    const int lane = i & 31, r = i >> 5;
    const int ks = r % KS, slot = (r / KS) % SL, grp = r / (KS * SL);
    const int s = min(s0 + 8 * grp + (lane >> 2), pr.S_pad - 1);
    const int e = mma_input<KS>(ks, lane & 3);
    const uint64_t* mk = masks + (size_t)s * P * pr.W + (e >> 6);
    uint64_t m;
    if (slot < P) {
      m = mk[slot * pr.W];
    } else {
      const int j = slot - P, pa = j < 1 ? 1 : (j < 3 ? 2 : 3), pb = j - (pa * (pa - 1)) / 2;
      m = mk[pa * pr.W] ^ mk[pb * pr.W];
    }
    const uint32_t n = (uint32_t)(m >> (e & 63)) & 15u;
    tab[i] = make_uint2(0x3C003C00u | ((n & 1u) << 15) | ((n & 2u) << 30),
                        0x3C003C00u | ((n & 4u) << 13) | ((n & 8u) << 28));
  }
}

// BF: W and W0 of every module are BF16 and copied ahead (kLoadAsync), known at
// compile time.
template <int P, int VAR, int KS, bool FAST, bool BF>
__global__ void __launch_bounds__(32 * kMmaWarps, mma_per_sm(VAR, KS))
    search_mma_kernel(Prm pr, const __grid_constant__ LaunchDesc ld, const uint64_t* __restrict__ masks,
                      const float4* __restrict__ pairs, awsrc_candidate* __restrict__ cands, int64_t n_items,
                      int mode, MmaSlots sl, int tab_bytes) {
  constexpr bool PF = VAR == AWSRC_VARIANT_PF;
  constexpr int SL = mma_slots(P, VAR), NG = mma_groups(P, VAR, KS), NL = P * (P - 1) / 2;
  constexpr int PS4 = pair_stride(P) / 2;  // float4 per seed pair
  extern __shared__ __align__(16) unsigned char smem[];
  uint2* tab = reinterpret_cast<uint2*>(smem);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, q = lane & 3;
  const int nsplit = ld.m[0].nsplit;
  const int64_t first = ld.m[0].tile_off;
  const int64_t last = ld.m[ld.n - 1].tile_off + ld.m[ld.n - 1].rows * ld.m[ld.n - 1].n_cb;
  const int groups = (pr.S + 7) / 8, per = (groups + nsplit - 1) / nsplit;
  int built = -1;  // first group of the table in shared memory
  // this thread's copy slots (kLoadAsync)
  const unsigned char* slots =
      smem + tab_bytes + (size_t)warp * (2 * (KS == 1 ? 1 : KS / 2) * sl.per_vec) * 512 + 16 * lane;
  const uint32_t slots_u = (uint32_t)__cvta_generic_to_shared(slots);
  MmaPos pos[2];
  // positions of this thread's two tiles of an item and, kLoadAsync, their copies
  auto fetch = [&](int64_t item) {
    const int64_t t0 = first + (item / nsplit) * kMmaTiles + 16 * warp + g;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int64_t t = min(t0 + 8 * r, last - 1);
      pos[r] = r && t == t0 + 8 ? mma_pos_after(ld, pos[0], t, 8u) : mma_pos(ld, t, 0);
      if ((BF || mode == kLoadAsync) && t0 + 8 * r < last) mma_copy<VAR, KS, BF>(ld, pos[r], r, q, sl, slots_u);
    }
    if (BF || mode == kLoadAsync) asm volatile("cp.async.commit_group;" ::: "memory");
  };
  pdl_trigger();
  if (blockIdx.x < n_items) fetch(blockIdx.x);
  pdl_wait();  // the masks and factors; the weights are the caller's, complete since the call's first launch
  for (int64_t item = blockIdx.x; item < n_items; item += gridDim.x) {
    const int z = (int)(item % nsplit);
    const int64_t t0 = first + (item / nsplit) * kMmaTiles + 16 * warp + g;
    uint32_t yh[KS][4], yl[KS][4], dh[PF ? KS : 1][4], dl[PF ? KS : 1][4];
    MmaRow row[2];
    if (BF || mode == kLoadAsync) asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll
    for (int r = 0; r < 2; ++r)
      mma_stage<P, VAR, KS, BF>(pr, ld, pos[r], t0 + 8 * r < last, r, q, mode, sl, slots, yh, yl, dh, dl, row[r]);
    __syncwarp();  // the slots are read: the next item's copies may start
    if (item + gridDim.x < n_items) fetch(item + gridDim.x);
    float bg[2] = {ninf(), ninf()};
    uint32_t bs[2] = {0xffffffffu, 0xffffffffu}, bc[2] = {0u, 0u};
    int bf[2] = {0, 0};
    const int g0 = min(groups, z * per), g1 = min(groups, g0 + per);
    for (int gc = g0; gc < g1; gc += NG) {
      const int ng = min(NG, g1 - gc);
      if (built != gc) {  // one chunk holds every seed unless there are many
        __syncthreads();
        mma_build_table<P, VAR, KS>(pr, masks, 8 * gc, ng, tab);
        __syncthreads();
        built = gc;
      }
      for (int gi = 0; gi < ng; ++gi) {
        const uint2* b = tab + (size_t)gi * SL * KS * 32 + lane;
        const int s = 8 * (gc + gi) + 2 * q;
        float2 bv[2][P], alpha[2][P];
#pragma unroll
        for (int p = 0; p < P; ++p) {
          float2 u[2];
          mma_sums<KS>(yh, yl, b + 32 * KS * p, u);
#pragma unroll
          for (int r = 0; r < 2; ++r) bv[r][p] = __fmul2_rn(u[r], make_float2(row[r].tqc, row[r].tqc));
        }
        float2 gp[2];
        uint32_t cw[2][2];
        int sf[2][2];
        if constexpr (PF) {
          float2 G[2][NL], nL[2][NL], E[2][NL], invD[2][P];
          bool okx[2] = {true, true}, oky[2] = {true, true};
#pragma unroll
          for (int j = 0; j < NL; ++j) {
            float2 u[2];
            mma_sums<KS>(dh, dl, b + 32 * KS * (P + j), u);
#pragma unroll
            for (int r = 0; r < 2; ++r) G[r][j] = __fmul2_rn(u[r], make_float2(row[r].tqdc, row[r].tqdc));
          }
#pragma unroll
          for (int r = 0; r < 2; ++r) invD[r][0] = make_float2(row[r].invd0, row[r].invd0);
          // LDL^T of G + eps I in the recipe's order, both tiles side by side
#pragma unroll
          for (int k = 1; k < P; ++k) {
            float2 dk[2], rk[2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
#pragma unroll
              for (int j = 0; j < k; ++j) {
                float2 v = G[r][tri(k, j)];
#pragma unroll
                for (int i = 0; i < j; ++i) v = __ffma2_rn(nL[r][tri(k, i)], E[r][tri(j, i)], v);
                E[r][tri(k, j)] = v;
                nL[r][tri(k, j)] = __fmul2_rn(v, neg2(invD[r][j]));
              }
              dk[r] = make_float2(row[r].diag, row[r].diag);
#pragma unroll
              for (int i = 0; i < k; ++i) dk[r] = __ffma2_rn(nL[r][tri(k, i)], E[r][tri(k, i)], dk[r]);
            }
            pivots_rcp<2>(dk, rk, okx, oky);
            invD[0][k] = rk[0];
            invD[1][k] = rk[1];
          }
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            ldl_solve2<P>(nL[r], invD[r], bv[r], alpha[r]);
            gp[r] = mma_gain<P, FAST, false>(pr, alpha[r], bv[r], make_float2(row[r].gd, row[r].gd), G[r], cw[r],
                                             sf[r]);
            if (!okx[r]) gp[r].x = ninf();
            if (!oky[r]) gp[r].y = ninf();
          }
        } else {
          // the pair's factors: -L, (invD m), invD, G off-diagonal (doubled when FAST), gd
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            const float4* pe = pairs + (size_t)(row[r].pair0 + (uint32_t)min(s, pr.S_pad - 2) / 2) * PS4;
            float2 f[4 * PS4 / 2];
#pragma unroll
            for (int i = 0; i < PS4; ++i) {
              if (2 * i + 1 >= NL && 2 * i + 1 < NL + P && 2 * i >= NL) continue;  // the bound's entries
              const float4 v = __ldg(pe + i);
              f[2 * i] = make_float2(v.x, v.y);
              f[2 * i + 1] = make_float2(v.z, v.w);
            }
            ldl_solve2<P>(f, f + NL + P, bv[r], alpha[r]);
            gp[r] = mma_gain<P, FAST, FAST>(pr, alpha[r], bv[r], f[2 * NL + 2 * P], f + NL + 2 * P, cw[r], sf[r]);
          }
        }
        // seeds reach a thread in increasing order: a strictly greater gain wins
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          if (s < pr.S && gp[r].x > bg[r]) {
            bg[r] = gp[r].x;
            bs[r] = (uint32_t)s;
            bc[r] = cw[r][0];
            bf[r] = sf[r][0];
          }
          if (s + 1 < pr.S && gp[r].y > bg[r]) {
            bg[r] = gp[r].y;
            bs[r] = (uint32_t)s + 1;
            bc[r] = cw[r][1];
            bf[r] = sf[r][1];
          }
        }
      }
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      // best of the tile's four lanes (larger gain, then smaller seed)
#pragma unroll
      for (int off = 1; off < 4; off <<= 1) {
        const float og = __shfl_xor_sync(0xffffffffu, bg[r], off);
        const uint32_t os = __shfl_xor_sync(0xffffffffu, bs[r], off);
        const uint32_t oc = __shfl_xor_sync(0xffffffffu, bc[r], off);
        const int of = __shfl_xor_sync(0xffffffffu, bf[r], off);
        if (better(og, os, bg[r], bs[r])) { bg[r] = og; bs[r] = os; bc[r] = oc; bf[r] = of; }
      }
      // one word of the candidate per lane: gain, seed and scale, codes, zero codes
      const int64_t t = t0 + 8 * r;
      if (t < last) {
        const bool valid = row[r].ok && bg[r] > ninf();
        const uint32_t word = q == 0   ? __float_as_uint(valid ? bg[r] : ninf())
                              : q == 1 ? (valid ? (bs[r] & 0xFFFFu) | ((uint32_t)bf[r] << 16) : 0u)
                              : q == 2 ? (valid ? bc[r] : 0u)
                                       : 0u;
        reinterpret_cast<uint32_t*>(cands + (size_t)z * ld.T + t)[q] = word;
      }
    }
  }
}

template <int P, int VAR, int KS, bool FAST>
cudaError_t launch_mma_t(const Prm& pr, const LaunchDesc& ld, const uint64_t* masks, const float2* pairs,
                         int64_t n_items, awsrc_candidate* cands, cudaStream_t st) {
  constexpr bool PF = VAR == AWSRC_VARIANT_PF;
  constexpr int V = KS == 1 ? 4 : 8, NV = 4 * KS / V;
  constexpr int most = mma_per_sm(VAR, KS);
  int mode = kLoadAsync, wb = 2, w0b = 2;
  for (int i = 0; i < ld.n; ++i) {
    const ModDesc& m = ld.m[i];
    const uintptr_t a = reinterpret_cast<uintptr_t>(m.W) | reinterpret_cast<uintptr_t>(m.W0) |
                        reinterpret_cast<uintptr_t>(m.act) | (PF ? reinterpret_cast<uintptr_t>(m.fisher) : 0);
    if (a & 15) mode = kLoadScalar;
    if (m.w_dtype == AWSRC_DTYPE_F32) wb = 4;
    if (m.w0_dtype == AWSRC_DTYPE_F32) w0b = 4;
  }
  const MmaSlots sl = mma_slots_of<V>(wb, w0b, PF);
  const int groups = std::min((pr.S + 7) / 8, mma_groups(P, VAR, KS));
  const size_t tab = (size_t)groups * mma_slots(P, VAR) * KS * 256;
  size_t smem = tab + (size_t)kMmaWarps * 2 * NV * sl.per_vec * 512;
  if (mode == kLoadAsync && smem > kMmaSmemMax) mode = kLoadVector;  // wide F32 tiles
  if (mode != kLoadAsync) smem = tab;
  const int per_sm = most == 2 && 2 * (smem + 1024) <= kMmaSmemMax ? 2 : 1;
  // (the binary16-scale and clamped-exponent quantisers keep the one general form)
  auto kern = search_mma_kernel<P, VAR, KS, FAST, false>;
  if constexpr (FAST)
    if (mode == kLoadAsync && wb == 2 && w0b == 2) kern = search_mma_kernel<P, VAR, KS, FAST, true>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMmaSmemMax);
  if (e != cudaSuccess) return e;
  int dev = 0, nsm = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(n_items, (int64_t)nsm * per_sm));
  // early only while every block has an SM of its own: a block that starts beside a
  // table kernel's finds the SM divided for that kernel, and two per SM then came one
  // after the other (205 -> 351 us on 9.4 M weights with C = 32, S = 64)
  e = launch_dep(n_items <= nsm, kern, dim3((unsigned)grid), dim3(32 * kMmaWarps), smem, st, pr, ld, masks,
                 reinterpret_cast<const float4*>(pairs), cands, n_items, mode, sl, (int)tab);
  note_launches(1);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <int P, int VAR>
cudaError_t launch_mma_p(const Prm& pr, const LaunchDesc& ld, const uint64_t* masks, const float2* pairs,
                         int64_t n, awsrc_candidate* cands, cudaStream_t st) {
  const bool f = pr.fast_pow2 != 0;
  switch (pr.C) {
    case 16: return f ? launch_mma_t<P, VAR, 1, true>(pr, ld, masks, pairs, n, cands, st)
                      : launch_mma_t<P, VAR, 1, false>(pr, ld, masks, pairs, n, cands, st);
    case 32: return f ? launch_mma_t<P, VAR, 2, true>(pr, ld, masks, pairs, n, cands, st)
                      : launch_mma_t<P, VAR, 2, false>(pr, ld, masks, pairs, n, cands, st);
    case 64: return f ? launch_mma_t<P, VAR, 4, true>(pr, ld, masks, pairs, n, cands, st)
                      : launch_mma_t<P, VAR, 4, false>(pr, ld, masks, pairs, n, cands, st);
    case 128: return f ? launch_mma_t<P, VAR, 8, true>(pr, ld, masks, pairs, n, cands, st)
                       : launch_mma_t<P, VAR, 8, false>(pr, ld, masks, pairs, n, cands, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace
}  // namespace awsrc
