// gemv_mma.cu — the packed product y[m] = (W0 + r_hat) x[m], m < M <= 8, on the
// tensor cores, for the codes of the code tables (P = 4, b <= 5, C in {16, 32, 64})
// with power-of-two scales, or no sidecar; gemv.cu serves the rest.
//
// One weight matrix against up to eight vectors: every weight is read once (0.68
// bytes with its scale and sidecar), so on the FP32 pipes the unpacking, one FMA
// per weight and vector and the x operands' shared-memory reads decide (24 M warp
// instructions for a 3B layer and one vector; eight vectors took ten times the
// time). With mma.sync m16n8k16 the eight vectors are the N columns of one
// instruction and cost the same as one:
//  * A: 16 rows of 4-bit codes as exact BF16 integers, from the code words by one
//    mask-and-xor into the mantissa of 128 + u and one packed subtraction;
//  * B: x as x = hi + mid + lo, three BF16 numbers whose sum is x exactly (8 + 8 + 8
//    significand bits by truncation), so a product loses nothing that binary32
//    holds. Where it is not (an input below 2^-110 whose last bits BF16 cannot hold,
//    an infinity or NaN), or a group's sum could overflow where gemv.cu's lanes, which
//    sum 32 inputs, do not, the vector's group goes through the FP32 pipes instead. The
//    chain of the hi parts and that of the mid and lo parts have their own binary32
//    accumulators, over one group of 128 inputs each (sums of 32 added with FMAs had a
//    relative error of 1.4e-7 where these have 9.9e-8). A group's sum is multiplied by
//    its scale and added with binary32 FMAs.
//  * The residual: k_j c 2^e is exact in BF16 (|k_j| <= 64), so recorded tiles are a
//    second A operand against the same B (rows without a record: zeros), with its own
//    accumulators; column runs without any record in the 16 rows are skipped.
// The order of the inputs along K is free: in each run of 32 inputs thread (g, q) =
// (lane / 4, lane % 4) takes inputs 8q .. 8q + 7, one code word of rows g and g + 8, one
// nibble-table window, two float4 of vector g.
//
// A warp takes 16 rows and a slice of the columns. A row tile's product is always made
// of the same eight column sums, added two by two through the shared memory of the block
// that has all its slices: how many slices there are (one to eight) depends on what
// else is in the launch, the product's bits do not.
//
// One 3B-shaped layer (77 M weights, 0.162 bits/weight of records, SDQ scales, eight
// vectors, one batched launch): 308 -> 76 us a call. Its relative error against 64 bits
// is 9.3e-8 where the FP32 pipes' sums had 1.4e-7. Bound by latency and issue (43% of
// slots): 695 warp instructions per 16 rows and 128 inputs without records (the split of
// x about half), 910 on average with this layer's; x comes from L1, so the sums' shared
// memory is no larger than needed (32 KB a block for all cases: 3 to 6% slower).
#include <algorithm>

#include "codetab.cuh"
#include "internal.h"

namespace awsrc {

namespace {

constexpr int kWarps = 8;
constexpr int kSums = 8;  // column slices whose sums make up a row tile's

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Upper halves of two binary32 numbers as a BF16 pair (a in the low half).
__device__ __forceinline__ uint32_t upper_pair(float a, float b) {
  return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
}
__device__ __forceinline__ float upper(float a) { return __uint_as_float(__float_as_uint(a) & 0xffff0000u); }

// Largest magnitude, of numbers.
__device__ __forceinline__ float max3_abs(float m, float a, float b) {
  float r;
  asm("{\n\t.reg .f32 y, z;\n\tabs.f32 y, %2;\n\tabs.f32 z, %3;\n\tmax.f32 %0, %1, y, z;\n\t}"
      : "=f"(r) : "f"(m), "f"(a), "f"(b));
  return r;
}

// B operand of a run of 32 inputs (two k-steps): pairs (x_i, x_{i+4}), i < 4, of
// this thread's eight inputs, split into three BF16 parts.
struct BRun {
  uint32_t hi[4], mid[4], lo[4];
};

// What tells whether the MMAs can take a thread's inputs of a group: each is below
// 2^113 (128 of them times codes then sum to less than 2^123) and its three parts are
// the input. They are from 2^-110 on; below, an input may have bits under 2^-133, which
// BF16 has not, and an infinity or NaN leaves a NaN: either way what is left of the
// third part has low bits.
struct XRange {
  float most;
  uint32_t left;
  __device__ bool ok() const { return (left & 0xFFFFu) == 0u && most < 0x1p113f; }
};

__device__ __forceinline__ void split_run(const float4& xa, const float4& xb, BRun& b, XRange& xr) {
  const float a[4] = {xa.x, xa.y, xa.z, xa.w}, c[4] = {xb.x, xb.y, xb.z, xb.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    xr.most = max3_abs(xr.most, a[i], c[i]);
    b.hi[i] = upper_pair(a[i], c[i]);
    const float2 r = __fadd2_rn(make_float2(a[i], c[i]), make_float2(-upper(a[i]), -upper(c[i])));
    b.mid[i] = upper_pair(r.x, r.y);
    const float2 s = __fadd2_rn(r, make_float2(-upper(r.x), -upper(r.y)));
    b.lo[i] = upper_pair(s.x, s.y);
    xr.left |= __float_as_uint(s.x) | __float_as_uint(s.y);
  }
}

// Codes i and i + 4 of a code word as a BF16 pair: 128 + u (u = code + 8) in the
// mantissa, minus 136.
__device__ __forceinline__ uint32_t code_pair(uint32_t w, int i) {
  const uint32_t v = ((w >> (4 * i)) & 0x000F000Fu) ^ 0x43084308u;
  uint32_t r;
  asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(0x43084308u));
  return r;
}

// acc += A B over a run: A as pairs (element i, element i + 4) of rows g and g + 8.
__device__ __forceinline__ void mma_run(float (&h)[4], float (&ml)[4], const uint32_t (&r0)[4],
                                        const uint32_t (&r1)[4], const BRun& b) {
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const uint32_t a[4] = {r0[2 * s], r1[2 * s], r0[2 * s + 1], r1[2 * s + 1]};
    mma_bf16(ml, a, b.lo[2 * s], b.lo[2 * s + 1]);
    mma_bf16(ml, a, b.mid[2 * s], b.mid[2 * s + 1]);
    mma_bf16(h, a, b.hi[2 * s], b.hi[2 * s + 1]);
  }
}

// What a thread needs of a recorded tile of its row: the record's byte tables as
// k_j + 64, and 2^(e - S) in both halves of a BF16 pair (k_j 2^(e - S) is k_j c 2^e
// for C = 64 and 16, k_j 2^e / 8 for C = 32, which is finite where k_j c 2^e is;
// 2^(e - S) may be a subnormal BF16).
struct TileRec {
  KTab kt;
  uint32_t sc;
  uint32_t seed;
};

template <int LC>
__device__ __forceinline__ TileRec tile_rec(const GemvArgs& a, unsigned long long e) {
  TileRec t{{0u, 0u, 0u, 0u}, 0u, 0u};
  if (e == 0ull) return t;
  const uint4 slot = __ldg(a.slots + ((int64_t)(e >> 32) - 1));
  // k_tables() gives k + 128 as bytes of 64 .. 192
  const KTab k = k_tables(slot);
  t.kt = {k.t0 - 0x40404040u, k.t1 - 0x40404040u, k.u0 - 0x40404040u, k.u1 - 0x40404040u};
  constexpr int S = LC == 4 ? 2 : 3;
  const int f = (int)(int16_t)(uint16_t)(e & 0xFFFFull) - S;
  const uint32_t sb = f >= -126 ? (uint32_t)(f + 127) << 7 : 1u << (f + 133);
  t.sc = sb * 0x00010001u;
  t.seed = (uint32_t)(e >> 16) & 0xFFFFu;
  return t;
}

// The residual of this thread's eight inputs (window nb of the seed's nibble
// table) as pairs (i, i + 4): the byte k + 64 completes 128 + (k + 64) in the
// mantissa (128 carries into the next binade, which is right), minus 192, times
// the scale, all exact; zeros where sc is 0 (no record).
__device__ __forceinline__ void residual_pairs(const TileRec& t, const uint4& nb, uint32_t (&r)[4]) {
  const uint32_t s0 = nb.x & 0xFFFFu, s1 = nb.x >> 16;
  const uint32_t a0 = __byte_perm(t.kt.t0, t.kt.t1, s0), b0 = __byte_perm(t.kt.u0, t.kt.u1, s0);
  const uint32_t a1 = __byte_perm(t.kt.t0, t.kt.t1, s1), b1 = __byte_perm(t.kt.u0, t.kt.u1, s1);
  const uint32_t k0 = (a0 & ~nb.y) | (b0 & nb.y), k1 = (a1 & ~nb.z) | (b1 & nb.z);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t v = (__byte_perm(k0, k1, 0x0400u + 0x0101u * i) & 0x00FF00FFu) | 0x43004300u;
    uint32_t d;
    asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(v), "r"(0x43404340u));
    asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(r[i]) : "r"(d), "r"(t.sc));
  }
}

// A run's products with the vectors named by `odd` (any of a quad's four bits: that
// quad's vector), on the FP32 pipes as gemv.cu forms them: x, the thread's inputs of
// vector 0; r0, r1, its A pairs of rows g and g + 8, left out where use0, use1 are
// false. out: the run's sums of rows g, g + 8 and vectors 2q, 2q + 1, like an MMA's.
__device__ __forceinline__ void run_fp32(const float* x, int64_t cols, unsigned odd, int q, const uint32_t (&r0)[4],
                                         const uint32_t (&r1)[4], bool use0, bool use1, float (&out)[4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) out[i] = 0.0f;
#pragma unroll 1
  for (int n = 0; n < 8; ++n) {
    if (((odd >> (4 * n)) & 15u) == 0u) continue;
    const float4 xa = __ldg(reinterpret_cast<const float4*>(x + n * cols));
    const float4 xb = __ldg(reinterpret_cast<const float4*>(x + n * cols + 4));
    const float v[8] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y, xb.z, xb.w};
    float p0 = 0.0f, p1 = 0.0f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      p0 = __fmaf_rn(__uint_as_float(r0[i] << 16), v[i], p0);
      p0 = __fmaf_rn(upper(__uint_as_float(r0[i])), v[i + 4], p0);
      p1 = __fmaf_rn(__uint_as_float(r1[i] << 16), v[i], p1);
      p1 = __fmaf_rn(upper(__uint_as_float(r1[i])), v[i + 4], p1);
    }
    if (!use0) p0 = 0.0f;
    if (!use1) p1 = 0.0f;
#pragma unroll
    for (int off = 1; off < 4; off <<= 1) {
      p0 = __fadd_rn(p0, __shfl_xor_sync(0xffffffffu, p0, off));
      p1 = __fadd_rn(p1, __shfl_xor_sync(0xffffffffu, p1, off));
    }
    if (q == n >> 1) {
      if (n & 1) {
        out[1] = p0;
        out[3] = p1;
      } else {
        out[0] = p0;
        out[2] = p1;
      }
    }
  }
}

template <int LC>
__global__ void __launch_bounds__(32 * kWarps, 2) gemv_mma_kernel(Prm pr, const __grid_constant__ GemvArgs a, int M) {
  extern __shared__ float4 part_mem[];
  float4(*part)[kSums][32] = reinterpret_cast<float4(*)[kSums][32]>(part_mem);  // [row tile of the block][sum][lane]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, q = lane & 3;
  int ti = 0;
  for (int i = 1; i < a.n_task; ++i)
    if ((int)blockIdx.x >= a.t[i].block0) ti = i;
  const GemvTask& tk = a.t[ti];
  const int ks = tk.slices, slice = warp & (ks - 1), per = kWarps / ks;  // slices: a power of two up to kWarps
  const int64_t row0 = ((int64_t)(blockIdx.x - tk.block0) * per + warp / ks) * 16;
  const int gpr = (int)(tk.cols >> 7);
  // the warp's groups: kSums / ks of the row tile's eight sums (some empty when gpr < 8)
  auto bound = [gpr](int i) { return (int)((int64_t)gpr * i / kSums); };
  const int sum0 = kSums / ks * slice, sum1 = row0 < tk.rows ? sum0 + kSums / ks : sum0;
  const int g0 = bound(sum0), g1 = bound(sum1);
  int64_t row[2];
#pragma unroll
  for (int r = 0; r < 2; ++r) row[r] = min(row0 + g + 8 * r, tk.rows - 1);  // rows past the end repeat the last one
  const uint32_t* cp[2];
  const unsigned long long* mp[2];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    cp[r] = reinterpret_cast<const uint32_t*>(tk.codes) + row[r] * (tk.cols >> 3) + q;
    mp[r] = a.map ? a.map + tk.tile_off + row[r] * (tk.cols >> LC) : nullptr;
  }
  const bool live = g < M;  // vector g
  const float* xp = tk.x + (live ? (int64_t)g * tk.cols : 0) + 8 * q;
  auto scale = [&](int r, int gr) {
    const int64_t gid = row[r] * gpr + gr;
    if (tk.sdq) {
      const float2 ms = __ldg(reinterpret_cast<const float2*>(tk.sdq_consts) + (gid >> 8));
      return __fadd_rn(ms.x, __fmul_rn((float)__ldg(tk.sdq_codes + gid), ms.y));
    }
    return __half2float(__ushort_as_half(__ldg(tk.scales + gid)));
  };
  // A group's code words, scales and (a tile per 2^LC inputs) map entries, one group ahead
  constexpr int NT = LC >= 5 ? 128 >> LC : 4;  // entries per group, row and thread
  uint32_t w[2][4];
  unsigned long long e[2][NT];
  float s[2];
  auto load = [&](int gr) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
#pragma unroll
      for (int j = 0; j < 4; ++j) w[r][j] = __ldg(cp[r] + 16 * gr + 4 * j);
      s[r] = scale(r, gr);
#pragma unroll
      for (int t = 0; t < NT; ++t)
        e[r][t] = mp[r] ? __ldg(mp[r] + (LC >= 5 ? NT * gr + t : 8 * gr + 2 * t + (q >> 1))) : 0ull;
    }
  };
  // c = 2^-(LC/2) is folded into the residual for C = 64 and 16; C = 32 had 1/8
  const float cf = LC == 5 ? __fmul_rn(8.0f, pr.c) : 1.0f;
  if (g0 < g1) load(g0);
  int gr = g0;
  for (int sum = sum0; sum < sum1; ++sum) {
    const int first = gr, end = bound(sum + 1);
    if (first == end) continue;
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f}, racc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    for (; gr < end; ++gr) {
      uint32_t wc[2][4];
      unsigned long long ec[2][NT];
      const float sc[2] = {s[0], s[1]};
#pragma unroll
      for (int r = 0; r < 2; ++r) {
#pragma unroll
        for (int j = 0; j < 4; ++j) wc[r][j] = w[r][j];
#pragma unroll
        for (int t = 0; t < NT; ++t) ec[r][t] = e[r][t];
      }
      if (gr + 1 < g1) load(gr + 1);
      float h[4] = {0.0f, 0.0f, 0.0f, 0.0f}, ml[4] = {0.0f, 0.0f, 0.0f, 0.0f};
      float rh[4] = {0.0f, 0.0f, 0.0f, 0.0f}, rml[4] = {0.0f, 0.0f, 0.0f, 0.0f};
      TileRec tr[2];
      XRange xr{0.0f, 0u};
      bool any = false;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float4 xa = make_float4(0.0f, 0.0f, 0.0f, 0.0f), xb = xa;
        if (live) {
          xa = __ldg(reinterpret_cast<const float4*>(xp + 128 * gr + 32 * j));
          xb = __ldg(reinterpret_cast<const float4*>(xp + 128 * gr + 32 * j + 4));
        }
        const int t = LC == 6 ? j >> 1 : j;
        if (LC != 6 || (j & 1) == 0) {  // a new tile
          any = mp[0] && __any_sync(0xffffffffu, (ec[0][t] | ec[1][t]) != 0ull);
          if (any) {
            tr[0] = tile_rec<LC>(a, ec[0][t]);
            tr[1] = tile_rec<LC>(a, ec[1][t]);
          }
        }
        uint4 nb[2];
        if (any) {
          const int win = ((32 * j + 8 * q) & ((1 << LC) - 1)) >> 3;
#pragma unroll
          for (int r = 0; r < 2; ++r) nb[r] = __ldg(a.nib + ((size_t)tr[r].seed << (LC - 3)) + win);
        }
        BRun b;
        split_run(xa, xb, b, xr);
        uint32_t c0[4], c1[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          c0[i] = code_pair(wc[0][j], i);
          c1[i] = code_pair(wc[1][j], i);
        }
        mma_run(h, ml, c0, c1, b);
        if (any) {
          residual_pairs(tr[0], nb[0], c0);
          residual_pairs(tr[1], nb[1], c1);
          mma_run(rh, rml, c0, c1, b);
        }
      }
      // Vectors that the MMAs could not take (inputs too small for the split, too large for
      // the sums, an infinity or NaN) get the group again on the FP32 pipes. Their columns
      // of the accumulators are their own.
      const unsigned odd = __ballot_sync(0xffffffffu, !xr.ok());
      if (odd) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if ((odd >> (8 * q + 4 * (i & 1))) & 15u) h[i] = ml[i] = rh[i] = rml[i] = 0.0f;
#pragma unroll 1
        for (int j = 0; j < 4; ++j) {
          const float* xj = tk.x + 128 * gr + 32 * j + 8 * q;
          uint32_t c0[4], c1[4];
          float o[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            c0[i] = code_pair(__ldg(cp[0] + 16 * gr + 4 * j), i);
            c1[i] = code_pair(__ldg(cp[1] + 16 * gr + 4 * j), i);
          }
          run_fp32(xj, tk.cols, odd, q, c0, c1, true, true, o);
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (sc[i >> 1] != 0.0f) acc[i] = __fmaf_rn(o[i], sc[i >> 1], acc[i]);
          if (!mp[0]) continue;
          unsigned long long en[2];
          const int jt = 32 * j + 8 * q;  // the thread's first input in the group
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            en[r] = __ldg(mp[r] + ((128 * gr + jt) >> LC));
            tr[r] = tile_rec<LC>(a, en[r]);
            const uint4 nb = __ldg(a.nib + ((size_t)tr[r].seed << (LC - 3)) + ((jt & ((1 << LC) - 1)) >> 3));
            residual_pairs(tr[r], nb, r ? c1 : c0);
          }
          run_fp32(xj, tk.cols, odd, q, c0, c1, en[0] != 0ull, en[1] != 0ull, o);
#pragma unroll
          for (int i = 0; i < 4; ++i) racc[i] = __fadd_rn(racc[i], o[i]);
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        racc[i] = __fadd_rn(racc[i], __fadd_rn(rh[i], rml[i]));
        if (LC != 5 && gr == first) {  // a sum starts from its first residual: a rounding less
          acc[i] = __fadd_rn(acc[i], racc[i]);
          racc[i] = 0.0f;
        }
        // an all-zero group (scale 0) adds nothing, whatever x holds
        const float sr = sc[i >> 1];
        if (sr != 0.0f) acc[i] = __fmaf_rn(__fadd_rn(h[i], ml[i]), sr, acc[i]);
      }
    }
    float v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = __fmaf_rn(racc[i], cf, acc[i]);
    part[warp / ks][sum][lane] = make_float4(v[0], v[1], v[2], v[3]);
  }
  __syncthreads();
  // the sums two by two: closer than one after the other
  float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  if (slice == 0 && row0 < tk.rows) {
    float4 p[kSums];
#pragma unroll
    for (int k = 0; k < kSums; ++k)
      p[k] = bound(k) < bound(k + 1) ? part[warp / ks][k][lane] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
    for (int d = 1; d < kSums; d <<= 1)
#pragma unroll
      for (int k = 0; k < kSums; k += 2 * d)
        p[k] = make_float4(__fadd_rn(p[k].x, p[k + d].x), __fadd_rn(p[k].y, p[k + d].y),
                           __fadd_rn(p[k].z, p[k + d].z), __fadd_rn(p[k].w, p[k + d].w));
    v[0] = p[0].x;
    v[1] = p[0].y;
    v[2] = p[0].z;
    v[3] = p[0].w;
  }
  if (slice == 0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int64_t r = row0 + g + 8 * (i >> 1);
      const int m = 2 * q + (i & 1);
      if (r < tk.rows && m < M) tk.y[(int64_t)m * tk.rows + r] = v[i];
    }
  }
}

}  // namespace

// From three vectors on, whatever the shapes: these sums are closer to 64 bits than
// those of the FP32 pipes (6 to 9e-8 against 9 to 14e-8), which would be faster on some
// single modules. In us on the device, FP32 pipes
// against tensor cores (whose time does not depend on M), records at 0.162 bits/weight:
// the layer above (random records), M = 3 and 8: 126 and 268 against 75; one module of
// 4096 x 4096: 19.8 and 92.5 against 20; 11008 x 2048: 24.3 and 47.7 against 27; 2048 x
// 2048: 8.0 and 14.2 against 9.9; 1024 x 1024: 4.1 and 6.6 against 6.4; 512 x 11008: 19.4
// and 38.4 against 36. M = 1 and 2 take 30 and 47 on that layer there.
bool gemv_mma(const Prm& pr, const GemvArgs& a, int M) {
  const bool c = pr.C == 16 || pr.C == 32 || pr.C == 64;
  return M >= 3 && c && (!a.map || (a.nib && pr.scale_mode == AWSRC_SCALE_POW2));
}

cudaError_t launch_gemv_mma(const Prm& pr, const GemvArgs& a, int M, cudaStream_t st) {
  GemvArgs b = a;
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  // Slices of at most eight groups; then the longest are halved, one task after the
  // other, and the division of least estimated time is kept. A block takes, in us, 1.2
  // and per group of its slices 3.3 alone on an SM, 4.4 beside another block, however
  // empty the chip is: up to three blocks per SM go in whole rounds, more keep the SMs
  // busy but for a quarter of a round. A 2048 x 2048 module alone went from 29 us (two
  // slices) to 10 (eight), an 11008 x 2048 one from 35 to 27, q/k/v of a 3B layer from 28
  // to 13; but a 3584-wide attention block takes 34 us in four slices (0.84 of the
  // blocks that are resident at once) and 37 in eight.
  int64_t tiles[kMaxGemvTasks] = {}, gpr[kMaxGemvTasks] = {};
  int ls[kMaxGemvTasks] = {}, best[kMaxGemvTasks] = {};  // log2 of the slices
  auto groups = [&](int i) { return (gpr[i] + (1 << ls[i]) - 1) >> ls[i]; };  // of a slice
  auto estimate = [&]() {
    double n = 0.0, work = 0.0, longest = 0.0;
    for (int i = 0; i < b.n_task; ++i) {
      const double blk = (double)(((tiles[i] << ls[i]) + kWarps - 1) / kWarps), g = (double)groups(i);
      n += blk;
      work += blk * g;
      longest = std::max(longest, g);
    }
    const double pair = 4.4 * work / n + 1.2, one = 3.3 * work / n + 1.2;
    const double t = n > 3.0 * nsm   ? (0.5 * n / nsm + 0.25) * pair
                     : n > 2.0 * nsm ? pair + one
                     : n > nsm       ? pair
                                     : one;
    return std::max(t, 3.3 * longest + 1.2);
  };
  for (int i = 0; i < b.n_task; ++i) {
    tiles[i] = (b.t[i].rows + 15) / 16;
    gpr[i] = b.t[i].cols >> 7;
    ls[i] = 0;
    while ((1 << ls[i]) < kWarps && groups(i) > 8) ++ls[i];
    best[i] = ls[i];
  }
  double least = estimate();
  while (true) {
    int m = -1;  // the task with the longest slices
    for (int i = 0; i < b.n_task; ++i)
      if ((1 << ls[i]) < kWarps && groups(i) > 1 && (m < 0 || groups(i) > groups(m))) m = i;
    if (m < 0) break;
    ++ls[m];
    const double t = estimate();
    if (t < 0.97 * least) {
      least = t;
      std::copy(ls, ls + b.n_task, best);
    }
  }
  for (int i = 0; i < b.n_task; ++i) b.t[i].slices = 1 << best[i];
  // the tasks with the longest slices first, so that their blocks do not end the
  // launch (69 us in the caller's order, the down projection last)
  std::stable_sort(b.t, b.t + b.n_task, [](const GemvTask& x, const GemvTask& y) {
    return (x.cols >> 7) * y.slices > (y.cols >> 7) * x.slices;
  });
  int64_t blocks = 0;
  size_t smem = 0;  // as little as the slices need: the rest of the SM's memory caches x
  for (int i = 0; i < b.n_task; ++i) {
    GemvTask& t = b.t[i];
    const int64_t per = 16 * (kWarps / t.slices);
    t.block0 = (int)blocks;
    smem = std::max(smem, (size_t)(kWarps / t.slices) * kSums * 32 * sizeof(float4));
    blocks += (t.rows + per - 1) / per;
  }
  if (blocks > 0x7fffffffll) return cudaErrorInvalidConfiguration;
  const dim3 grid((unsigned)blocks), block(32 * kWarps);
  switch (pr.C) {
    case 16: gemv_mma_kernel<4><<<grid, block, smem, st>>>(pr, b, M); break;
    case 32: gemv_mma_kernel<5><<<grid, block, smem, st>>>(pr, b, M); break;
    case 64: gemv_mma_kernel<6><<<grid, block, smem, st>>>(pr, b, M); break;
    default: return cudaErrorInvalidValue;
  }
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace awsrc
