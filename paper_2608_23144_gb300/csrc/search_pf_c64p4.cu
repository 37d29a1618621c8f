// search_pf_c64p4.cu — seed search (Sec. 3.2) for AWSRC-P_F with C = 64, P = 4
// on the tcgen05 tensor cores.
//
// P_F weights every element (d_ij = w_act a_j + w_fisher F_ij), so the Gram
// matrix G = B_s^T D B_s / C differs per (tile, seed): its off-diagonal entries
// are the +-1 correlations of the tile's D with the pairwise products
// m_p * m_q of the seed's atoms, and its diagonal is the tile's gd. Both the
// correlations b_p (with y = d r) and the six off-diagonals are exact integer
// sums on the tile's fixed-point grids (|Y|, |D| <= 2^21, FP16 halves
// hi = X >> 11, lo = X & 2047), computed by tcgen05.mma and rounded once in the
// epilogue, which then factors G + eps I (LDL^T), solves, quantises and scores
// every candidate exactly as the binary32 recipe does.
//
// Block: 128 tiles of one column block (row m = TMEM lane m), 14 warps. The
// loader warp streams 12-seed chunks (FP16 atoms 6 KB, a slice of the U search's
// atom table, and FP16 atom products 10 KB) through a 4-stage bulk-copy ring; the
// MMA warp issues per chunk 16 MMAs into one of two TMEM accumulators: Y_hi, Y_lo
// x atoms (N = 48) and D_hi, D_lo x products (N = 80, the last 8 columns zero).
// Epilogue warp w takes TMEM lanes 32(w%4).. and seed pairs 2(w/4), 2(w/4) + 1 of
// each chunk, each as a float2 stream over the pair's two seeds, the two pairs
// factored side by side so that their dependency chains interleave. Every
// mbarrier wait is bounded.
//
// What bounds it, per chunk of 12 seeds on one SM (clock64 in copies of the kernel,
// 1.78 GHz): with one lane issuing the MMAs inside a branch and refilling the ring
// between them, 2140 cycles, 1360 of them the issue, about 500 the refill; a copy
// that scored nothing was hardly faster (1840). The issue by a converged warp (630),
// a loader of its own and the scoring in unit domain (below) each measured nothing
// or a loss alone; together they take an attention block of a 7B-shaped layer
// (29.4 M weights, S = 4096) from 9.16 to 8.61 ms. The epilogue bounds it now: three
// warps per scheduler at 1550 cycles a chunk, their FMA pipe 80% busy meanwhile.
#include "fit2.cuh"
#include "internal.h"
#include "tc05.cuh"

namespace awsrc {

namespace {

using namespace tc05;

constexpr int BM = 128;             // rows (tiles) per block = TMEM lanes
constexpr int CH = 12;              // seeds per chunk
constexpr int NA = 4 * CH;          // atom columns per chunk (MMA N = 48)
constexpr int NQ = 6 * CH;          // product columns per chunk
constexpr int NQP = 80;             // product columns padded to a multiple of 16 (MMA N)
constexpr int EW = 12;              // epilogue warps: 4 lane quarters x 3 groups of 2 seed pairs
constexpr int PPW = CH / 2 / (EW / 4);  // seed pairs per epilogue warp and chunk
constexpr int NT = 32 * (EW + 2);      // + the MMA warp and the loader warp
constexpr int STAGES = 4;
constexpr uint32_t kABytes = NA * 64 * 2;      // 6 KB
constexpr uint32_t kQBytes = NQP * 64 * 2;     // 10 KB (the last 8 columns zero)
constexpr uint32_t kStageBytes = kABytes + kQBytes;
constexpr uint32_t kTmemCols = 512;            // 2 accumulators of 256 columns
constexpr int kYH = 0, kYL = NA, kDH = 2 * NA, kDL = 2 * NA + NQP;  // columns within an accumulator
static_assert(kDL + NQP <= 256, "accumulator of 256 columns");
constexpr uint32_t kIdA = idesc_f16(BM, NA);
constexpr uint32_t kIdQ = idesc_f16(BM, NQP);
static_assert(PPW == 2 && (EW / 4) * PPW * 2 == CH, "two seed pairs per epilogue warp and chunk");
static_assert(kStageBytes % 1024 == 0 && kABytes % 1024 == 0, "stage layout");

struct Smem {
  __half A[4][BM * 64];  // Y_hi, Y_lo, D_hi, D_lo: canonical K-major, no swizzle
  unsigned char stage[STAGES][kStageBytes];
  float Yst[BM][65];
  float Dst[BM][65];
  float tqc[BM];      // 2^qy * c
  float tqdc[BM];     // 2^qd * c2
  float gd[BM];       // G_pp
  float diag[BM];     // fl(gd + eps)
  float invd0[BM];    // 1 / D_0 = 1 / diag
  float gdu[BM];      // unit domain: gd', 2^(7-qd) diag, -1 / that, 2^(qd-2qy), 2^(2qy-qd)
  float diag2[BM], ninvd0[BM], to_unit[BM], from_unit[BM];
  float inv_qy[BM], inv_qd[BM];
  int rowok[BM];
  float red_g[EW / 4][BM];
  uint32_t red_s[EW / 4][BM];
  unsigned long long full[STAGES], afull[2], tempty[2];
  unsigned long long sfree[STAGES];  // a stage's MMAs have completed
  uint32_t tmem_base;
};

__device__ __forceinline__ float neg_inf() { return -__int_as_float(0x7f800000); }

__device__ __forceinline__ int a_offset(int m, int k) {
  return (((m >> 3) * 8 + (k >> 3)) << 7) + ((m & 7) << 4) + ((k & 7) << 1);
}

// Exact sums RN(2048*hi + lo) of two seeds.
__device__ __forceinline__ float2 pair_sum(const float* hi, const float* lo, int i) {
  return __ffma2_rn(make_float2(2048.0f, 2048.0f), make_float2(hi[i], hi[i + 1]), make_float2(lo[i], lo[i + 1]));
}

// Fits of NP seed pairs of this thread's row in the recipe's units, factored
// side by side so that their chains interleave; bv[j]: b of pair j's two seeds,
// G[j]: the off-diagonal G (tri order). Gives alpha and whether each candidate's
// pivots are valid.
template <int NP>
__device__ __forceinline__ void pf_fit(const float2 (*bv)[4], const float2 (*G)[6], float diag, float invd0,
                                       float2 (*alpha)[4], bool* okx, bool* oky) {
  const float2 dg = make_float2(diag, diag);
  float2 nL[NP][6], E[NP][6], invD[NP][4];
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    invD[j][0] = make_float2(invd0, invd0);  // D_0 = diag for every seed
    okx[j] = true;
    oky[j] = true;
  }
  // LDL^T of G + eps I in the recipe's order
#pragma unroll
  for (int k = 1; k < 4; ++k) {
    float2 dk[NP], rk[NP];
#pragma unroll
    for (int jp = 0; jp < NP; ++jp) {
#pragma unroll
      for (int j = 0; j < k; ++j) {
        float2 v = G[jp][tri(k, j)];
#pragma unroll
        for (int i = 0; i < j; ++i) v = __ffma2_rn(nL[jp][tri(k, i)], E[jp][tri(j, i)], v);
        E[jp][tri(k, j)] = v;
        nL[jp][tri(k, j)] = __fmul2_rn(v, neg2(invD[jp][j]));  // -(v * invD_j), exact negation
      }
      dk[jp] = dg;
#pragma unroll
      for (int i = 0; i < k; ++i) dk[jp] = __ffma2_rn(nL[jp][tri(k, i)], E[jp][tri(k, i)], dk[jp]);
    }
    pivots_rcp<NP>(dk, rk, okx, oky);
#pragma unroll
    for (int jp = 0; jp < NP; ++jp) invD[jp][k] = rk[jp];
  }
#pragma unroll
  for (int j = 0; j < NP; ++j) ldl_solve2<4>(nL[j], invD[j], bv[j], alpha[j]);
}

// Gains of NP seed pairs in the recipe's units (operands as for pf_fit).
template <bool FAST, int NP>
__device__ __forceinline__ void pf_gain(const Prm& pr, const float2 (*bv)[4], const float2 (*G)[6], float gd,
                                        float diag, float invd0, float2* g, float2 (*alpha_out)[4] = nullptr) {
  float2 alpha[NP][4];
  bool okx[NP], oky[NP];
  pf_fit<NP>(bv, G, diag, invd0, alpha, okx, oky);
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    if (alpha_out) {
#pragma unroll
      for (int p = 0; p < 4; ++p) alpha_out[j][p] = alpha[j][p];
    }
    if constexpr (FAST) {
      g[j] = quant_gain_fast2_g<4>(pr, alpha[j], bv[j], make_float2(gd, gd), G[j]);
    } else {
      float q4[4];
      int sf;
      float Gx[6], a[4], b[4];
#pragma unroll
      for (int i = 0; i < 6; ++i) Gx[i] = G[j][i].x;
#pragma unroll
      for (int p = 0; p < 4; ++p) { a[p] = alpha[j][p].x; b[p] = bv[j][p].x; }
      g[j].x = quant_gain<4>(pr, a, b, gd, Gx, q4, &sf);
#pragma unroll
      for (int i = 0; i < 6; ++i) Gx[i] = G[j][i].y;
#pragma unroll
      for (int p = 0; p < 4; ++p) { a[p] = alpha[j][p].y; b[p] = bv[j][p].y; }
      g[j].y = quant_gain<4>(pr, a, b, gd, Gx, q4, &sf);
    }
    if (!okx[j]) g[j].x = neg_inf();
    if (!oky[j]) g[j].y = neg_inf();
  }
}

// ------------------------------------------------------------- unit domain --
// For C = 64 every scale of the recipe (c, c2, the grids' 2^qy and 2^qd) is a
// power of two, and the whole fit commutes with powers of two as long as no
// value over- or underflows. So the common case works on the integer sums
// themselves, u (for y) and v2 = 2 v (for the off-diagonals; the D operand of the
// MMAs holds 2 D): with b = 2^(qy-3) u and G = 2^(qd-7) v2,
//   LDL^T of 2^(7-qd) (G + eps I): the same L, D'' = 2^(7-qd) D;
//   alpha'' = 2^(qd-qy-4) alpha, hence the same codes, with sc' = 2^(qd-qy-3) sc;
//   gain = 2^(2qy-qd) sc' (2 sum q u - sc' Qq'), Qq' from gd' = 2^(6-qd) gd and v2
//     (q_p q_r v2 is the recipe's 2 q_p q_r G: no doubling needed).
// A row's gains all carry the same factor, so the argmax needs none of it: 10
// multiplications and 3 additions fewer per seed pair than in the recipe's
// units, of 96 packed FP32 operations on the pipe that bounds this kernel.
//
// The results are those of the recipe bit for bit while nothing leaves the
// normal range in either domain. That is ensured by testing what could: rows need
// 2^-26 <= 2^qd <= 2^20 and 2^qy >= 2^-40 (else the block scores in the recipe's
// units throughout), pivots D'' in [2, 2^40) (so |L| stays moderate and no pivot is a
// rounding residue: gd'' is at least 2^21) and amax'' in [2^-40, 2^12]. With these
// amax lies in the recipe's valid range, and a value could only be subnormal in the
// recipe's units after cancelling more than 80 bits, to where it no longer reaches a
// code. A pair step in which some lane fails a test is scored again in the recipe's
// units. Rows outside the numeric domain and rows whose y is zero on the grid (every
// fit 0, which the recipe calls invalid) have no candidate: their lanes pass.
constexpr int kUnitQdLo = -26, kUnitQdHi = 20, kUnitQyLo = -40;

// min and max of three (the packed kernels' range tests fold several values).
__device__ __forceinline__ float min3(float a, float b, float c) {
  float r;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// Negated gains (in unit domain) of NP seed pairs; false when some candidate of
// this lane leaves the ranges above. Everything after the solve works with
// -alpha'' (the factorisation keeps -1 / D''): rounding is symmetric, so its codes
// are the negated ones, Qq is even in them, and what comes out, sc' (2 sum q u +
// sc' Qq), is exactly the negated gain; the search then takes the smallest.
template <int NP>
__device__ __forceinline__ bool pf_loss_unit(const Prm& pr, const float2 (*u)[4], const float2 (*v2)[6], float gdu,
                                             float diag2, float ninvd0, float2* h) {
  const float2 dg = make_float2(diag2, diag2);
  float2 nL[NP][6], E[NP][6], nD[NP][4];
  float2 piv[NP][4];
#pragma unroll
  for (int j = 0; j < NP; ++j) nD[j][0] = make_float2(ninvd0, ninvd0);
#pragma unroll
  for (int k = 1; k < 4; ++k) {
#pragma unroll
    for (int jp = 0; jp < NP; ++jp) {
#pragma unroll
      for (int j = 0; j < k; ++j) {
        float2 v = v2[jp][tri(k, j)];
#pragma unroll
        for (int i = 0; i < j; ++i) v = __ffma2_rn(nL[jp][tri(k, i)], E[jp][tri(j, i)], v);
        E[jp][tri(k, j)] = v;
        nL[jp][tri(k, j)] = __fmul2_rn(v, nD[jp][j]);
      }
      float2 d = dg;
#pragma unroll
      for (int i = 0; i < k; ++i) d = __ffma2_rn(nL[jp][tri(k, i)], E[jp][tri(k, i)], d);
      piv[jp][k] = d;
      // -1/D'' correctly rounded as in pivots_rcp, y = approx(-D): y + y (1 + D y)
      float yx, yy;
      asm("{\n\t.reg .f32 t;\n\tneg.f32 t, %1;\n\trcp.approx.ftz.f32 %0, t;\n\t}" : "=f"(yx) : "f"(d.x));
      asm("{\n\t.reg .f32 t;\n\tneg.f32 t, %1;\n\trcp.approx.ftz.f32 %0, t;\n\t}" : "=f"(yy) : "f"(d.y));
      const float2 ny = make_float2(yx, yy);
      const float2 e = __ffma2_rn(d, ny, make_float2(1.0f, 1.0f));
      nD[jp][k] = __ffma2_rn(ny, e, ny);
    }
  }
  // A pivot that leaves [2, 2^40) is finite when it does (those before it are
  // fine), so the smallest and the largest tell.
  float dlo = 2.0f, dhi = 0.0f, alo = 1.0f, ahi = 1.0f;
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    dlo = min3(dlo, min3(piv[j][1].x, piv[j][2].x, piv[j][3].x), min3(piv[j][1].y, piv[j][2].y, piv[j][3].y));
    dhi = max3(dhi, max3(piv[j][1].x, piv[j][2].x, piv[j][3].x), max3(piv[j][1].y, piv[j][2].y, piv[j][3].y));
  }
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    float2 al[4];
    ldl_solve2<4>(nL[j], nD[j], u[j], al);
    const float m0 = fmaxf(max3(fabsf(al[0].x), fabsf(al[1].x), fabsf(al[2].x)), fabsf(al[3].x));
    const float m1 = fmaxf(max3(fabsf(al[0].y), fabsf(al[1].y), fabsf(al[2].y)), fabsf(al[3].y));
    alo = min3(alo, m0, m1);
    ahi = max3(ahi, m0, m1);
    // 2^e'' by fast_scale_bits(), sc' = 2^(e'' + 1)
    const uint32_t s0 = fast_scale_bits(pr, __float_as_uint(m0)), s1 = fast_scale_bits(pr, __float_as_uint(m1));
    const float2 inv = make_float2(__uint_as_float(0x7F000000u - s0), __uint_as_float(0x7F000000u - s1));
    const float2 sc = make_float2(__uint_as_float(s0 + 0x00800000u), __uint_as_float(s1 + 0x00800000u));
    const float2 magic = make_float2(12582912.0f, 12582912.0f), nmagic = make_float2(-12582912.0f, -12582912.0f);
    float2 q[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) q[p] = __fadd2_rn(__ffma2_rn(al[p], inv, magic), nmagic);
    float2 Aq = make_float2(0.0f, 0.0f), Qq = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int p = 0; p < 4; ++p) Aq = __ffma2_rn(q[p], u[j][p], Aq);
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      Qq = __ffma2_rn(__fmul2_rn(q[p], q[p]), make_float2(gdu, gdu), Qq);
#pragma unroll
      for (int r = p + 1; r < 4; ++r) Qq = __ffma2_rn(__fmul2_rn(q[p], q[r]), v2[j][tri(r, p)], Qq);
    }
    h[j] = __fmul2_rn(sc, __ffma2_rn(make_float2(2.0f, 2.0f), Aq, __fmul2_rn(sc, Qq)));
  }
  return dlo >= 2.0f && dhi < 0x1p40f && alo >= 0x1p-40f && ahi <= 0x1p12f;
}

// Codes and scale field of the winning seed of row m. The search keeps only
// (gain, seed), so the seed's correlations with Y (atoms) and D (atom
// products) are formed again as the exact integer sums the tensor cores
// accumulate, rounded once, and go through the fit and quantiser in the recipe's
// units. Both halves of the pair get the winner's sums; one is read. Returns the gain
// once more, which must equal the one the search found.
template <bool FAST>
__device__ __forceinline__ float pf_winner(const Prm& pr, const Smem& sm, int m, const uint64_t* mk, bool odd,
                                           uint32_t* cw, int* sf) {
  const float iy = sm.inv_qy[m], idd = sm.inv_qd[m];
  uint64_t w[4];
#pragma unroll
  for (int p = 0; p < 4; ++p) w[p] = mk[p];
  uint64_t wq[6];
#pragma unroll
  for (int a = 1, q = 0; a < 4; ++a)
#pragma unroll
    for (int c = 0; c < a; ++c, ++q) wq[q] = w[a] ^ w[c];  // products in tri order
  int ty = 0, td = 0, ny[4] = {0, 0, 0, 0}, nd[6] = {0, 0, 0, 0, 0, 0};
  for (int j = 0; j < 64; ++j) {
    const int y = iy == 0.0f ? 0 : fixed_point_int(sm.Yst[m][j], iy);
    const int d = idd == 0.0f ? 0 : fixed_point_int(sm.Dst[m][j], idd);
    ty += y;
    td += d;
#pragma unroll
    for (int p = 0; p < 4; ++p) ny[p] += ((w[p] >> j) & 1ull) ? y : 0;
#pragma unroll
    for (int q = 0; q < 6; ++q) nd[q] += ((wq[q] >> j) & 1ull) ? d : 0;
  }
  float2 bv[1][4], G[1][6];
#pragma unroll
  for (int p = 0; p < 4; ++p) {  // |sum| <= 64 * 2^21, rounded once
    const float u = __fmul_rn(__int2float_rn(ty - 2 * ny[p]), sm.tqc[m]);
    bv[0][p] = make_float2(u, u);
  }
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    const float u = __fmul_rn(__int2float_rn(td - 2 * nd[q]), sm.tqdc[m]);
    G[0][q] = make_float2(u, u);
  }
  float2 alpha[1][4], g;
  pf_gain<FAST, 1>(pr, bv, G, sm.gd[m], sm.diag[m], sm.invd0[m], &g, alpha);
  float a[4], q4[4], zero[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
  for (int p = 0; p < 4; ++p) a[p] = odd ? alpha[0][p].y : alpha[0][p].x;
  if constexpr (FAST) (void)quant_gain_fast<4>(pr, a, zero, 0.0f, zero, q4, sf);
  else (void)quant_gain<4>(pr, a, zero, 0.0f, zero, q4, sf);
  uint32_t c = 0u;
#pragma unroll
  for (int p = 0; p < 4; ++p) c |= ((uint32_t)(int)q4[p] & 0xFFu) << (8 * p);
  *cw = c;
  return odd ? g.y : g.x;
}

// STALL: the loader issues no copies from chunk pr.stall_chunk on (a test of the waits).
// An instance of its own: with the comparison in the loader of every call, however it
// is written, the search lost 3% (8.61 -> 8.85 ms on an attention block of a 7B layer).
template <bool FAST, bool STALL>
__global__ void __launch_bounds__(NT, 1)
    search_pf_kernel(Prm pr, LaunchDesc ld, const unsigned char* __restrict__ atoms,
                     const unsigned char* __restrict__ prods, const uint64_t* __restrict__ masks,
                     awsrc_candidate* __restrict__ cands, uint32_t* __restrict__ status) {
  extern __shared__ unsigned char smem_raw[];
  // 1 KB aligned through an integer cast, which leaves the accesses generic:
  // measured faster here than the shared-space form the U search uses
  Smem& sm = *reinterpret_cast<Smem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int mi = find_mod(ld, blockIdx.x);
  const ModDesc& md = ld.m[mi];
  const int64_t b = blockIdx.x - md.block_off;
  const int z = (int)(b % md.nsplit);
  const int64_t rest = b / md.nsplit;
  const int64_t rb = rest % md.n_rb;
  const int64_t cb = rest / md.n_rb;

  const int nchunks = pr.S_pad / CH;
  const int per = (nchunks + md.nsplit - 1) / md.nsplit;
  const int c0 = min(nchunks, z * per);
  const int c1 = min(nchunks, c0 + per);
  const int nck = c1 - c0;
  const unsigned char* a_src = atoms + (size_t)c0 * kABytes;
  const unsigned char* q_src = prods + (size_t)c0 * kQBytes;

  if (warp == EW) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_addr(&sm.tmem_base)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    if (lane == 0) {
      for (int i = 0; i < STAGES; ++i) {
        mbar_init(&sm.full[i], 1);
        mbar_init(&sm.sfree[i], 1);
      }
      for (int i = 0; i < 2; ++i) {
        mbar_init(&sm.afull[i], 1);
        mbar_init(&sm.tempty[i], EW);
      }
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
  }
  if (tid < BM) sm.rowok[tid] = 1;
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm.tmem_base;

  int issued = 0;  // chunks whose copies the loader issued
  auto load_chunk = [&]() {
    const int st = issued % STAGES;
    mbar_expect_tx(&sm.full[st], kStageBytes);
    bulk_g2s(&sm.stage[st][0], a_src + (size_t)issued * kABytes, kABytes, &sm.full[st]);
    bulk_g2s(&sm.stage[st][kABytes], q_src + (size_t)issued * kQBytes, kQBytes, &sm.full[st]);
    ++issued;
  };
  if (warp == EW + 1 && lane == 0)
    while (issued < STAGES && issued < nck && !(STALL && issued == pr.stall_chunk)) load_chunk();
  // stage y = d * r and d, d = w_act * a + w_fisher * F (per element)
  for (int e = tid; e < BM * 64; e += NT) {
    const int r = e >> 6, j = e & 63;
    const int64_t row = rb * BM + r;
    float y = 0.0f, d = 0.0f;
    if (row < md.rows) {
      const int64_t idx = row * md.cols + cb * 64 + j;
      const float rr = __fsub_rn(load_elem(md.W, idx, md.w_dtype), load_elem(md.W0, idx, md.w0_dtype));
      d = __fadd_rn(__fmul_rn(md.w_act, md.act[cb * 64 + j]), __fmul_rn(md.w_fisher, md.fisher[idx]));
      if (!in_domain(rr, d)) sm.rowok[r] = 0;
      y = __fmul_rn(d, rr);
    }
    sm.Yst[r][j] = y;
    sm.Dst[r][j] = d;
  }
  __syncthreads();
  bool safe = true;
  if (tid < BM) {  // per row: fixed-point exponents, gd, eps and the first pivot
    float my = 0.0f, mdd = 0.0f;
    for (int j = 0; j < 64; ++j) {
      my = fmaxf(my, fabsf(sm.Yst[tid][j]));
      mdd = fmaxf(mdd, fabsf(sm.Dst[tid][j]));
    }
    int qy, qd;
    const float iy = fixed_point_inv(my, &qy);
    const float idd = fixed_point_inv(mdd, &qd);
    const float two_qd = pow2f(qd);
    int sd = 0;
    for (int j = 0; j < 64; ++j) sd += idd == 0.0f ? 0 : fixed_point_int(sm.Dst[tid][j], idd);
    const float gd = __fmul_rn(pr.c2, __fmul_rn(__int2float_rn(sd), two_qd));
    const float eps = __fmul_rn(pr.ridge_rel, gd);
    const float diag = __fadd_rn(gd, eps);
    // a y of zeros on its grid: every fit is 0, no candidate is valid
    const bool ok = sm.rowok[tid] && pivot_ok(diag) && iy != 0.0f;
    sm.rowok[tid] = ok ? 1 : 0;
    sm.inv_qy[tid] = ok ? iy : 0.0f;
    sm.inv_qd[tid] = ok ? idd : 0.0f;
    sm.tqc[tid] = __fmul_rn(pow2f(qy), pr.c);
    sm.tqdc[tid] = __fmul_rn(two_qd, pr.c2);
    sm.gd[tid] = gd;
    sm.diag[tid] = diag;
    sm.invd0[tid] = __frcp_rn(diag);
    // unit domain (a row that is no candidate gets harmless constants)
    safe = !ok || (qd >= kUnitQdLo && qd <= kUnitQdHi && qy >= kUnitQyLo);
    const bool un = ok && safe;
    sm.gdu[tid] = un ? __fmul_rn(gd, pow2f(6 - qd)) : 1.0f;
    sm.diag2[tid] = un ? __fmul_rn(diag, pow2f(7 - qd)) : 0x1p21f;
    sm.ninvd0[tid] = -__frcp_rn(sm.diag2[tid]);
    sm.to_unit[tid] = un ? pow2f(qd - 2 * qy) : 1.0f;
    sm.from_unit[tid] = un ? pow2f(2 * qy - qd) : 1.0f;
  }
  const bool unit = __syncthreads_and(safe) && FAST;
  // A operands: one thread writes one 16-byte core-matrix row of both halves
  for (int e = tid; e < 2 * BM * 8; e += NT) {
    const int which = e >= BM * 8;  // 0: Y, 1: D
    const int ee = e - which * BM * 8;
    const int m = ee >> 3, k0 = (ee & 7) * 8;
    const float inv = which ? sm.inv_qd[m] : sm.inv_qy[m];
    const float* src = which ? &sm.Dst[m][k0] : &sm.Yst[m][k0];
    uint32_t wh[4], wl[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int x0 = inv == 0.0f ? 0 : fixed_point_int(src[2 * i], inv);
      const int x1 = inv == 0.0f ? 0 : fixed_point_int(src[2 * i + 1], inv);
      // D doubled: 2 hi <= 2048 and the even 2 lo <= 4094 are exact in FP16
      wh[i] = (uint32_t)__half_as_ushort(__int2half_rn((x0 >> 11) << which)) |
              ((uint32_t)__half_as_ushort(__int2half_rn((x1 >> 11) << which)) << 16);
      wl[i] = (uint32_t)__half_as_ushort(__int2half_rn((x0 & 2047) << which)) |
              ((uint32_t)__half_as_ushort(__int2half_rn((x1 & 2047) << which)) << 16);
    }
    const int off = a_offset(m, k0);
    *reinterpret_cast<uint4*>(reinterpret_cast<unsigned char*>(sm.A[2 * which]) + off) =
        make_uint4(wh[0], wh[1], wh[2], wh[3]);
    *reinterpret_cast<uint4*>(reinterpret_cast<unsigned char*>(sm.A[2 * which + 1]) + off) =
        make_uint4(wl[0], wl[1], wl[2], wl[3]);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();

  bool timed_out = false;
  if (warp == EW) {
    // ----------------------------------------------------------------- MMAs --
    uint32_t ab[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) ab[i] = smem_addr(sm.A[i]);
    const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
    int k = 0;
    for (; k < nck; ++k) {
      const int st = k % STAGES, tb = k & 1;
      if (!mbar_wait_warp(&sm.full[st], (uint32_t)((k / STAGES) & 1), pr.wait_ns)) { timed_out = true; break; }
      if (k >= 2 && !mbar_wait_warp(&sm.tempty[tb], (uint32_t)(((k - 2) >> 1) & 1), pr.wait_ns)) {
        timed_out = true;
        break;
      }
      tc_fence_after();
      const uint32_t sa = smem_addr(&sm.stage[st][0]), sq = sa + kABytes;
      const uint32_t acc = tm + (uint32_t)(tb * 256);
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) {
        const uint32_t kb = (uint32_t)ks * 256u, en = ks > 0 ? 1u : 0u;
        umma_f16_warp(acc + kYH, smem_desc(ab[0] + kb), smem_desc(sa + kb), kIdA, en);
        umma_f16_warp(acc + kYL, smem_desc(ab[1] + kb), smem_desc(sa + kb), kIdA, en);
        umma_f16_warp(acc + kDH, smem_desc(ab[2] + kb), smem_desc(sq + kb), kIdQ, en);
        umma_f16_warp(acc + kDL, smem_desc(ab[3] + kb), smem_desc(sq + kb), kIdQ, en);
      }
      umma_commit_warp(&sm.afull[tb]);
    }
    // on a timeout wait (bounded) for the MMAs still in flight
    if (timed_out && k > 0) (void)mbar_wait_warp(&sm.afull[(k - 1) & 1], (uint32_t)(((k - 1) >> 1) & 1), pr.wait_ns);
  } else if (warp == EW + 1) {
    // --------------------------------------------------------------- loader --
    if (lane == 0) {
      // each time the stage of chunk issued - STAGES, once its MMAs are complete
      while (issued < nck && !(STALL && issued == pr.stall_chunk)) {
        if (!mbar_wait(&sm.sfree[issued % STAGES], (uint32_t)((issued / STAGES - 1) & 1), pr.wait_ns)) {
          timed_out = true;
          break;
        }
        load_chunk();
      }
      // the copies in flight land before the block ends, whoever timed out
      for (int j = max(0, issued - STAGES); j < issued; ++j)
        if (!mbar_wait(&sm.full[j % STAGES], (uint32_t)((j / STAGES) & 1), pr.wait_ns)) timed_out = true;
    }
  } else {
    // ------------------------------------------------------------ epilogue --
    const int m = 32 * (warp & 3) + lane;
    const int grp = warp >> 2;  // seed pairs 2 grp and 2 grp + 1 of each chunk
    const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
    const float gdu = sm.gdu[m], diag2 = sm.diag2[m], ninvd0 = sm.ninvd0[m];
    // the recipe's units, for the pair steps that need them
    auto recipe = [&](const float2 (*u)[4], const float2 (*v2)[6], float2* g) {
      const float tqc = sm.tqc[m], tqdc = __fmul_rn(0.5f, sm.tqdc[m]);  // v2 = 2 v
      float2 bv[2][4], G[2][6];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
#pragma unroll
        for (int p = 0; p < 4; ++p) bv[j][p] = __fmul2_rn(u[j][p], make_float2(tqc, tqc));
#pragma unroll
        for (int q = 0; q < 6; ++q) G[j][q] = __fmul2_rn(v2[j][q], make_float2(tqdc, tqdc));
      }
      pf_gain<FAST, 2>(pr, bv, G, sm.gd[m], sm.diag[m], sm.invd0[m], g);
    };
    const bool dead = sm.rowok[m] == 0;
    float bg = -neg_inf();  // smallest negated gain
    uint32_t bsd = 0xffffffffu;
    for (int k = 0; k < nck; ++k) {
      const int tb = k & 1;
      if (!mbar_wait(&sm.afull[tb], (uint32_t)((k >> 1) & 1), pr.wait_ns)) { timed_out = true; break; }
      if (tid == 0) mbar_arrive(&sm.sfree[k % STAGES]);
      tc_fence_after();
      const uint32_t base = tmem + lane_base + (uint32_t)(tb * 256);
      // both pairs' columns are loaded before the accumulator is released, so
      // the next MMAs into it wait for no scoring; a pair's 12 product columns
      // start at 12 pi, 8-aligned for the even pair, 4 past for the odd one
      float ah[2][8], al[2][8], qh[2][12], ql[2][12];
      const int p0 = 2 * grp, p1 = p0 + 1;
      tmem_ld8(base + kYH + 8 * p0, ah[0]);
      tmem_ld8(base + kYL + 8 * p0, al[0]);
      tmem_ld8(base + kDH + 12 * p0, qh[0]);
      tmem_ld4(base + kDH + 12 * p0 + 8, qh[0] + 8);
      tmem_ld8(base + kDL + 12 * p0, ql[0]);
      tmem_ld4(base + kDL + 12 * p0 + 8, ql[0] + 8);
      tmem_ld8(base + kYH + 8 * p1, ah[1]);
      tmem_ld8(base + kYL + 8 * p1, al[1]);
      tmem_ld4(base + kDH + 12 * p1, qh[1]);
      tmem_ld8(base + kDH + 12 * p1 + 4, qh[1] + 4);
      tmem_ld4(base + kDL + 12 * p1, ql[1]);
      tmem_ld8(base + kDL + 12 * p1 + 4, ql[1] + 4);
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        tmem_tie8(ah[j]);
        tmem_tie8(al[j]);
#pragma unroll
        for (int i = 0; i < 3; ++i) { tmem_tie4(qh[j] + 4 * i); tmem_tie4(ql[j] + 4 * i); }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.tempty[tb]);
      float2 u[2][4], v2[2][6], g2[2];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
#pragma unroll
        for (int p = 0; p < 4; ++p) u[j][p] = pair_sum(ah[j], al[j], 2 * p);
#pragma unroll
        for (int q = 0; q < 6; ++q) v2[j][q] = pair_sum(qh[j], ql[j], 2 * q);
      }
      if (!unit) {
        recipe(u, v2, g2);
#pragma unroll
        for (int j = 0; j < 2; ++j) g2[j] = neg2(g2[j]);
      } else {
        const bool in = pf_loss_unit<2>(pr, u, v2, gdu, diag2, ninvd0, g2) || dead;
        if (__any_sync(0xffffffffu, !in)) {
          recipe(u, v2, g2);
          const float f = -sm.to_unit[m];
#pragma unroll
          for (int j = 0; j < 2; ++j) g2[j] = __fmul2_rn(g2[j], make_float2(f, f));
        }
      }
      // the smallest negated gain; seeds reach a thread in increasing order, so a
      // strictly smaller one wins. Padding selectors (all-zero masks, in the last
      // chunk only) are not candidates.
      const int sx = (c0 + k) * CH + 2 * p0;
      if (sx + 3 >= pr.S) {
        if (sx >= pr.S) g2[0].x = -neg_inf();
        if (sx + 1 >= pr.S) g2[0].y = -neg_inf();
        if (sx + 2 >= pr.S) g2[1].x = -neg_inf();
        if (sx + 3 >= pr.S) g2[1].y = -neg_inf();
      }
      const float cm = fminf(min3(g2[0].x, g2[0].y, g2[1].x), g2[1].y);
      if (cm < bg) {
        bg = cm;
        bsd = (uint32_t)(sx + (g2[0].x == cm ? 0 : g2[0].y == cm ? 1 : g2[1].x == cm ? 2 : 3));
      }
    }
    // (a loss of +0 is a gain of +0, not -0)
    sm.red_g[grp][m] = unit ? __fadd_rn(0.0f, __fmul_rn(-bg, sm.from_unit[m])) : -bg;
    sm.red_s[grp][m] = bsd;
  }
  tc_fence_before();
  if (__syncthreads_or(timed_out)) {
    if (tid == 0) atomicOr(status, kFaultTimeout);
  } else if (tid < BM) {
    float g = sm.red_g[0][tid];
    uint32_t s = sm.red_s[0][tid];
#pragma unroll
    for (int i = 1; i < EW / 4; ++i) {
      if (better(sm.red_g[i][tid], sm.red_s[i][tid], g, s)) { g = sm.red_g[i][tid]; s = sm.red_s[i][tid]; }
    }
    const int64_t row = rb * BM + tid;
    if (row < md.rows) {
      const int64_t tt = md.tile_off + row * md.n_cb + cb;
      const bool valid = sm.rowok[tid] && g > neg_inf();
      uint32_t cw = 0u;
      int sf = 0;
      if (valid) {
        const float gw = pf_winner<FAST>(pr, sm, tid, masks + (size_t)s * 4, (s & 1u) != 0u, &cw, &sf);
        if (__float_as_uint(gw) != __float_as_uint(g)) atomicOr(status, kFaultSelfCheck);
      }
      awsrc_candidate cd;
      cd.gain = valid ? g : neg_inf();
      cd.seed = valid ? (uint16_t)s : (uint16_t)0;
      cd.scale = (int16_t)sf;
#pragma unroll
      for (int p = 0; p < 4; ++p) cd.code[p] = (int8_t)(cw >> (8 * p));
#pragma unroll
      for (int p = 4; p < 8; ++p) cd.code[p] = 0;
      cands[(size_t)z * ld.T + tt] = cd;
    }
  }
  if (warp == EW) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols)
                 : "memory");
  }
}

// FP16 products of atom pairs in the order the MMAs read them: chunk c
// (12 seeds) is an 80 x 64 K-major operand in 10 KB; item i (16 bytes, one
// core-matrix row) is chunk i / 640, column group n8 = (i >> 6) % 10, k group
// (i >> 3) & 7, row i & 7; column n = 8*n8 + r < 72 carries product q =
// (n % 12) / 2 (pairs (1,0), (2,0), (2,1), (3,0), (3,1), (3,2)) of seed
// 12c + 2*(n / 12) + n % 2, and columns 72 .. 79 are zero.
constexpr int kQItems = NQP * 8;  // 16-byte items per chunk

__global__ void products_kernel(const uint64_t* __restrict__ masks, uint4* __restrict__ out, int S_pad) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t n_items = (int64_t)(S_pad / CH) * kQItems;
  if (i >= n_items) return;
  const int64_t chunk = i / kQItems;
  const int w = (int)(i % kQItems);
  const int r = w & 7, kg = (w >> 3) & 7, n8 = w >> 6;
  const int n = 8 * n8 + r;
  if (n >= NQ) {
    out[i] = make_uint4(0u, 0u, 0u, 0u);
    return;
  }
  const int q = (n % 12) >> 1;
  const int64_t seed = chunk * CH + 2 * (n / 12) + (n & 1);
  const int pa = q < 1 ? 1 : (q < 3 ? 2 : 3);
  const int pb = q - (pa * (pa - 1)) / 2;
  const uint64_t m = masks[(size_t)seed * 4 + pa] ^ masks[(size_t)seed * 4 + pb];
  uint32_t wv[4];
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    const int k = 8 * kg + 2 * h;
    const uint32_t lo = ((m >> k) & 1ull) ? 0xBC00u : 0x3C00u;  // -1 : +1 in FP16
    const uint32_t hi = ((m >> (k + 1)) & 1ull) ? 0xBC00u : 0x3C00u;
    wv[h] = lo | (hi << 16);
  }
  out[i] = make_uint4(wv[0], wv[1], wv[2], wv[3]);
}

}  // namespace

int search_pf_c64p4_chunk() { return CH; }
size_t search_pf_c64p4_table_bytes(int S_pad) { return (size_t)(S_pad / CH) * kQBytes; }

cudaError_t launch_products_pf_c64p4(const Prm& pr, const uint64_t* masks, void* out, cudaStream_t st) {
  const int64_t n = (int64_t)(pr.S_pad / CH) * kQItems;
  products_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(masks, static_cast<uint4*>(out), pr.S_pad);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_search_pf_c64p4(const Prm& pr, const LaunchDesc& ld, const void* atoms, const void* prods,
                                   const uint64_t* masks, int64_t n_blocks, awsrc_candidate* cands,
                                   uint32_t* status, cudaStream_t st) {
  const size_t smem = sizeof(Smem) + 1024;
  auto kern = pr.stall_chunk >= 0 ? search_pf_kernel<false, true>
              : pr.fast_pow2      ? search_pf_kernel<true, false>
                                  : search_pf_kernel<false, false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<(unsigned)n_blocks, NT, smem, st>>>(pr, ld, static_cast<const unsigned char*>(atoms),
                                             static_cast<const unsigned char*>(prods), masks, cands, status);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace awsrc
