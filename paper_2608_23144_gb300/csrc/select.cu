// select.cu — byte-aware allocation (Sec. 3.3) and serialisation (Sec. 3.4, Eq. 5).
//
// rho_t = gain_t / L with one L for all records, so the stream order is gain
// descending, ties by tile ascending, within each module (U) or over the whole
// call (PF, whose prefixes are the rate cuts). Every candidate gets a 31-bit
// field that ascends in that order; non-positive or non-finite gains get the
// largest one and are never kept. U's modules, or PF's one range of all tiles,
// are the segments below.
//
// Only the records that fit the budget are sorted (16% of the tiles at 0.162
// bits/weight and C = 64). One cooperative kernel does it all, its steps
// separated by grid barriers:
//  1. fields of all tiles, and per segment a histogram of their upper 11 bits;
//  2. per segment, from the histogram: the eligible count, hence the records
//     kept, and the bin in which the last of them lies;
//  3. the tiles up to that bin, compacted in tile order (count, then write);
//  4. a stable LSD radix sort of those within their segments, three or four
//     passes over as many bits as the kept fields of the widest segment span (per
//     pass: digit histograms of runs of keys, prefix sums over runs, ranked
//     scatter). Equal fields keep the tile order of step 3, so tiles are no part
//     of the key.
//  5. the records are packed, and the header and counts written.
// The whole step is asynchronous on the caller's stream.
//
// What bounds it: a small call the barriers and the latency of a phase between two of
// them (one 3B-shaped layer, 1.2 M tiles: 84 us), a large one the scattered candidate
// reads of the pack and the passes over the kept keys (four 7B-shaped layers, 14.6 M
// tiles, 25% kept: 340 us, of which 35 read the gains, 37 compact, 138 are the three
// passes and 98 pack). Sorting every key in 16 to 20 launches per call took 160 and 901 us.
#include <algorithm>
#include <cfloat>
#include <cuda.h>

#include "internal.h"
#include "tc05.cuh"

namespace awsrc {

namespace {

constexpr int kMaxSelMods = 1024;
constexpr int kMaxRates = 64;
constexpr int kBins = 2048;             // bins of the fields' upper bits
constexpr int kBinShift = 20;
constexpr int kMaxDigits = 512;         // 27 bits in three passes, 31 in four
constexpr int ST = 512;                 // threads of the sort kernel
constexpr int SW = ST / 32;
constexpr int kRankIpt = 8;              // keys a thread ranks at once, at most
constexpr int kRound = kRankIpt * ST;
constexpr int kPackIpt = 4;              // records a thread packs at once
constexpr int kRunMin = 512;            // keys per run at least
constexpr int64_t kMaxBlocks = 1024;    // blocks of the kernel at most
constexpr uint32_t kIneligible = 0x7FFFFFFFu;

struct SelArgs {
  int n_mod, n_rates, variant;
  int64_t T, L, h;
  int64_t tile_off[kMaxSelMods + 1];
  int64_t kcap[kMaxSelMods];     // U: per module; PF: per rate
};

struct SegInfo {                 // a segment after step 2
  uint32_t lo, end;              // kept fields lie in [lo, end): whole bins
  uint32_t kept, K;              // keys kept for the sort, records of the stream
};

// Device arrays of the sort kernel.
struct SortWs {
  // zeroed before the launch
  unsigned* bar;                 // [0]: barrier arrivals, [1]: a wait gave up
  uint32_t* per_mod;             // PF: records of each module in the stream
  uint32_t* bins;                // [segment][kBins]
  SegInfo* seg;                  // [segment]
  uint32_t* cnt;                 // [block] keys kept by a block's tiles
  uint32_t *k0, *v0, *k1, *v1;   // field and tile, ping-pong; k1 first holds the fields of all tiles
  uint32_t* hist;                // [run][digit]; in step 1 [block + segment][kBins]
  uint32_t* total;               // [segment][digit]
};

__device__ __forceinline__ uint32_t gain_field(float g) {
  const bool ok = (g > 0.0f) && (g <= FLT_MAX);
  return ok ? (0x7F7FFFFFu - __float_as_uint(g)) : kIneligible;
}

// Grid barrier of a cooperative launch, bounded in time: false when some
// block's wait gave up (then every block leaves the kernel).
enum : int {
  kGrid = 0,      // the default limit, known at compile time
  kOneBlock = 1,  // a single block: nothing to wait for
  kTestGrid = 2   // a limit of its own, set by a test of the waits
};  // (one instance for all three took 0.3 to 0.7% longer: 83.9 against 83.3 us a 3B layer)

template <int MODE>
struct GridBarrier {
  unsigned* bar;
  unsigned phase;
  uint64_t limit_ns;
  __device__ bool sync() {
    __syncthreads();
    if (MODE == kOneBlock) return true;
    bool ok = true;
    if (threadIdx.x == 0) {
      __threadfence();
      ++phase;
      const unsigned target = phase * gridDim.x;
      atomicAdd(bar, 1u);
      const volatile unsigned* vb = bar;
      if (vb[0] < target) {
        const uint64_t t0 = tc05::globaltimer();
        while (vb[0] < target) {
          if (vb[1] != 0u || tc05::globaltimer() - t0 > (MODE == kTestGrid ? limit_ns : kWaitLimitNs)) {
            atomicExch(bar + 1, 1u);
            ok = false;
            break;
          }
        }
      }
      __threadfence();
    }
    return !__syncthreads_or(!ok);
  }
};

// Block-wide exclusive scan of one value per thread (ST threads).
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* total, uint32_t* warp_sums) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_sums[w] = x;
  __syncthreads();
  if (w == 0) {
    uint32_t s = lane < SW ? warp_sums[lane] : 0u;
#pragma unroll
    for (int o = 1; o < SW; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    if (lane < SW) warp_sums[lane] = s;
  }
  __syncthreads();
  const uint32_t before = (w > 0 ? warp_sums[w - 1] : 0u) + x - v;
  if (total) *total = warp_sums[SW - 1];
  __syncthreads();
  return before;
}

__device__ __forceinline__ uint32_t warp_inclusive(uint32_t x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

struct SortSmem {
  union {
    uint32_t bins[kBins];                // step 1
    struct {
      uint32_t base[kMaxDigits];         // next position of each digit
      uint32_t first[kMaxDigits];        // first place of each digit in a round's sorted keys
    } d;
    uint32_t rec_off[kMaxSelMods + 1];   // step 5: first record of each segment
  };
  union {
    struct {
      uint32_t mask[SW][kMaxDigits];     // per warp: lanes holding each digit (zero between uses)
      uint16_t wcnt[SW][kMaxDigits];     // per warp: keys of each digit, then those of earlier warps
    } r;
    uint2 sorted[kRound];                // a round's keys, sorted by digit
    uint8_t buf[kPackIpt * ST * 16 + 16];  // step 5: packed records
  };
  uint32_t key_off[kMaxSelMods + 1];     // first kept key of each segment
  uint32_t run_off[kMaxSelMods + 1];     // first run of each segment; step 5: PF's records per module
  uint32_t tile_off[kMaxSelMods];        // step 5
  uint32_t part[SW][32];
  uint32_t ws[32];
  uint32_t maxbits, maxruns, carry;
};

// First segment index whose range [off[i], off[i + 1]) holds x.
template <typename T>
__device__ __forceinline__ int find_seg(const T* off, int n, T x) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) / 2;
    if (x >= off[mid]) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Exclusive offsets of n <= kMaxSelMods per-segment values into off[0 .. n].
template <typename F>
__device__ __forceinline__ void seg_scan(SortSmem& sm, int n, uint32_t* off, F value) {
  if (threadIdx.x == 0) sm.carry = 0u;
  __syncthreads();
  for (int m0 = 0; m0 < n; m0 += ST) {
    const int m = m0 + threadIdx.x;
    const uint32_t v = m < n ? value(m) : 0u;
    uint32_t tot;
    const uint32_t e = block_exclusive_scan(v, &tot, sm.ws) + sm.carry;
    if (m < n) off[m] = e;
    __syncthreads();
    if (threadIdx.x == 0) sm.carry += tot;
    __syncthreads();
  }
  if (threadIdx.x == 0) off[n] = sm.carry;
  __syncthreads();
}

__device__ __forceinline__ int ceil_log2_dev(uint64_t x) {
  return x <= 1 ? 0 : 64 - __clzll((long long)(x - 1));
}

// Append the low nbits (<= 64) of v at bit *pos of the 128-bit record (w1:w0).
__device__ __forceinline__ void put_bits(uint64_t* w0, uint64_t* w1, int* pos, uint64_t v, int nbits) {
  if (nbits == 0) return;
  v &= nbits >= 64 ? ~0ull : ((1ull << nbits) - 1ull);
  const int p = *pos;
  if (p >= 64) {
    *w1 |= v << (p - 64);
  } else {
    *w0 |= v << p;
    if (p + nbits > 64) *w1 |= v >> (64 - p);
  }
  *pos += nbits;
}

// Packs n <= kPackIpt * ST consecutive records, the stream's i0 .. i0 + n - 1,
// from their tiles in rank order. What a record costs is one DRAM access to its
// candidate, scattered over the tiles, and L bytes written: a thread has several
// candidates in flight, the records are assembled in shared memory at the
// stream's own 16-byte phase and leave as whole 16-byte words (bytes at the two
// ends), and PF's records per module are counted in shared memory (with one
// global atomic per record, 3.64 M records of 28 modules took 1420 us). Making
// the records in tile order before the sort and gathering them here was no
// faster: it reads the candidates from DRAM a second time.
__device__ __forceinline__ void pack_block(const SelArgs& a, const Prm& pr, const uint32_t* tiles,
                                           const awsrc_candidate* __restrict__ cands, uint8_t* __restrict__ stream,
                                           const uint32_t* key_off, const uint32_t* rec_off,
                                           const uint32_t* tile_off, uint32_t* per_mod, uint8_t* buf, int64_t i0,
                                           int n) {
  const bool pf = a.variant != AWSRC_VARIANT_U;
  const int L = (int)a.L;
  uint8_t* const dst = stream + a.h + i0 * L;
  const int phase = (int)(reinterpret_cast<uintptr_t>(dst) & 15);
  const int tile_bits = ceil_log2_dev((uint64_t)a.T), seed_bits = ceil_log2_dev((uint64_t)pr.S);
  uint32_t tile[kPackIpt], ss[kPackIpt], c03[kPackIpt], c47[kPackIpt];
#pragma unroll
  for (int u = 0; u < kPackIpt; ++u) {
    const int li = u * ST + (int)threadIdx.x;
    if (li < n) {
      const uint32_t i = (uint32_t)i0 + (uint32_t)li;
      const int m = pf ? 0 : find_seg(rec_off, a.n_mod, i);
      tile[u] = __ldcg(tiles + key_off[m] + (i - rec_off[m]));
    }
  }
#pragma unroll
  for (int u = 0; u < kPackIpt; ++u) {
    if (u * ST + (int)threadIdx.x < n) {
      const uint32_t* c = reinterpret_cast<const uint32_t*>(cands + tile[u]);
      ss[u] = __ldg(c + 1);
      c03[u] = __ldg(c + 2);
      c47[u] = pr.P > 4 ? __ldg(c + 3) : 0u;
    }
  }
#pragma unroll
  for (int u = 0; u < kPackIpt; ++u) {
    const int li = u * ST + (int)threadIdx.x;
    if (li >= n) continue;
    if (pf) atomicAdd(&per_mod[find_seg(tile_off, a.n_mod, tile[u])], 1u);
    uint64_t w0 = 0, w1 = 0;
    int pos = 0;
    put_bits(&w0, &w1, &pos, (uint64_t)tile[u], tile_bits);
    put_bits(&w0, &w1, &pos, ss[u] & 0xFFFFu, seed_bits);
    const int16_t scale = (int16_t)(ss[u] >> 16);
    const uint64_t sf = pr.scale_mode == AWSRC_SCALE_POW2 ? (uint64_t)(int64_t)(scale - pr.e_bias)
                                                          : (uint64_t)(uint16_t)scale;
    put_bits(&w0, &w1, &pos, sf, pr.b_e);
    for (int p = 0; p < pr.P; ++p)
      put_bits(&w0, &w1, &pos, (uint64_t)(int64_t)(int8_t)((p < 4 ? c03[u] : c47[u]) >> (8 * (p & 3))), pr.b);
    uint8_t* o = buf + phase + li * L;
    if (L == 8 && (phase & 7) == 0) {
      *reinterpret_cast<uint64_t*>(o) = w0;
    } else {
      for (int k = 0; k < L; ++k) o[k] = (uint8_t)(k < 8 ? (w0 >> (8 * k)) : (w1 >> (8 * (k - 8))));
    }
  }
  __syncthreads();
  // bytes [phase, end) of buf are the block's part of the stream
  const int end = phase + n * L;
  for (int w = threadIdx.x; 16 * w < end; w += ST) {
    const int b0 = 16 * w, b1 = b0 + 16;
    if (b0 >= phase && b1 <= end) {
      *reinterpret_cast<uint4*>(dst - phase + b0) = *reinterpret_cast<const uint4*>(buf + b0);
    } else {
      for (int b = max(b0, phase); b < min(b1, end); ++b) dst[b - phase] = buf[b];
    }
  }
  __syncthreads();
}

__device__ __forceinline__ void put_le(uint8_t* p, uint64_t v, int n) {
  for (int i = 0; i < n; ++i) p[i] = (uint8_t)(v >> (8 * i));
}

// The header's fixed 40 bytes; K records.
__device__ __forceinline__ void put_header(const SelArgs& a, const Prm& pr, uint64_t K, uint8_t* stream) {
  for (int k = 0; k < 40; ++k) stream[k] = 0;
  put_le(stream + 0, 0x52535741u, 4);
  put_le(stream + 4, 1, 2);
  stream[6] = (uint8_t)pr.variant;
  stream[7] = (uint8_t)pr.scale_mode;
  put_le(stream + 8, (uint64_t)pr.C, 2);
  stream[10] = (uint8_t)pr.P;
  stream[11] = (uint8_t)pr.b;
  stream[12] = (uint8_t)pr.b_e;
  stream[13] = (uint8_t)(int8_t)pr.e_bias;
  stream[14] = (uint8_t)pr.permute;
  put_le(stream + 16, (uint64_t)pr.S, 4);
  put_le(stream + 20, (uint64_t)a.n_mod, 4);
  put_le(stream + 24, pr.gen_seed, 8);
  put_le(stream + 32, K, 8);
}

template <int MODE>
__global__ void __launch_bounds__(ST, 2) select_kernel(const awsrc_candidate* __restrict__ cands,
                                                     const __grid_constant__ SelArgs a,
                                                     const __grid_constant__ SortWs w, Prm pr,
                                                     uint8_t* __restrict__ stream, int64_t* __restrict__ d_counts,
                                                     int64_t* __restrict__ d_bytes, uint32_t* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SortSmem& sm = *reinterpret_cast<SortSmem*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool pf = a.variant != AWSRC_VARIANT_U;
  const int nseg = pf ? 1 : a.n_mod;
  GridBarrier<MODE> bar{w.bar, 0u, pr.wait_ns};
  // tiles of this block, and of segment m
  const int64_t per = (a.T + gridDim.x - 1) / gridDim.x;
  const int64_t t0 = min(a.T, (int64_t)blockIdx.x * per), t1 = min(a.T, t0 + per);
  auto seg_begin = [&](int m) { return pf ? (int64_t)0 : a.tile_off[m]; };
  auto seg_end = [&](int m) { return pf ? a.T : a.tile_off[m + 1]; };
  const int m0 = t0 >= t1 ? nseg : (pf ? 0 : find_seg(a.tile_off, a.n_mod, t0));

  // 1. fields and histograms
  for (int m = m0; m < nseg && seg_begin(m) < t1; ++m) {
    const int64_t b = max(t0, seg_begin(m)), e = min(t1, seg_end(m));
    for (int i = tid; i < kBins; i += ST) sm.bins[i] = 0u;
    __syncthreads();
    for (int64_t t = b + tid; t < e; t += 4 * ST) {
      float g[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (t + u * ST < e) g[u] = __ldcs(&cands[t + u * ST].gain);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (t + u * ST < e) {
          const uint32_t f = gain_field(g[u]);
          w.k1[t + u * ST] = f;
          atomicAdd(&sm.bins[f >> kBinShift], 1u);
        }
      }
    }
    __syncthreads();
    // the block's own counts stay in row blockIdx + m of the run histograms (free
    // until step 4), which no other (block, segment) has
    uint32_t* own = w.hist + ((size_t)blockIdx.x + m) * kBins;
    for (int i = tid; i < kBins; i += ST) {
      const uint32_t c = sm.bins[i];
      own[i] = c;
      if (c) atomicAdd(&w.bins[(size_t)m * kBins + i], c);
    }
    __syncthreads();
  }
  if (!bar.sync()) { if (tid == 0) atomicOr(status, kFaultTimeout); return; }

  // 2. one warp per segment: lane l sums bins 64 l .. 64 l + 63, then the warp
  // looks into the one range that decides
  for (int m = blockIdx.x * SW + warp; m < nseg; m += gridDim.x * SW) {
    const uint32_t* h = w.bins + (size_t)m * kBins;
    uint32_t s = 0u, lastv = 0u;
#pragma unroll 4
    for (int i = 0; i < 16; ++i) {
      const uint4 v = __ldcg(reinterpret_cast<const uint4*>(h + 64 * lane) + i);
      s += v.x + v.y + v.z + v.w;
      lastv = v.w;
    }
    if (lane == 31) s -= lastv;  // the last bin holds the ineligible tiles
    const uint32_t inc = warp_inclusive(s);
    const uint32_t npos = __shfl_sync(0xffffffffu, inc, 31);
    int64_t cap = 0;
    if (pf) {
      for (int r = 0; r < a.n_rates; ++r) cap = max(cap, a.kcap[r]);
    } else {
      cap = a.kcap[m];
    }
    const uint32_t K = (uint32_t)min((int64_t)npos, cap);
    SegInfo si{0u, 0u, 0u, K};
    if (K > 0u) {
      const int first = __ffs(__ballot_sync(0xffffffffu, s != 0u)) - 1;   // range of the first non-empty bin
      const int lastl = __ffs(__ballot_sync(0xffffffffu, inc >= K)) - 1;  // range in which K is reached
      const uint2 vf = __ldcg(reinterpret_cast<const uint2*>(h + 64 * first) + lane);
      const unsigned nz = __ballot_sync(0xffffffffu, (vf.x | vf.y) != 0u);
      const int fl = __ffs(nz) - 1;
      const uint32_t fx = __shfl_sync(0xffffffffu, vf.x, fl);
      si.lo = (uint32_t)(64 * first + 2 * fl + (fx ? 0 : 1)) << kBinShift;
      const uint2 vl = __ldcg(reinterpret_cast<const uint2*>(h + 64 * lastl) + lane);
      const uint32_t before = __shfl_sync(0xffffffffu, inc - s, lastl);
      const uint32_t iy = before + warp_inclusive(vl.x + vl.y), ix = iy - vl.y;
      const int ll = __ffs(__ballot_sync(0xffffffffu, iy >= K)) - 1;
      const uint32_t cx = __shfl_sync(0xffffffffu, ix, ll), cy = __shfl_sync(0xffffffffu, iy, ll);
      si.end = (uint32_t)(64 * lastl + 2 * ll + (cx >= K ? 1 : 2)) << kBinShift;
      si.kept = cx >= K ? cx : cy;
    }
    if (lane == 0) w.seg[m] = si;
    if (!pf && lane == 0) d_counts[m] = K;
    if (pf && lane == 0) {
      for (int r = 0; r < a.n_rates; ++r) {
        const int64_t Kr = min((int64_t)npos, a.kcap[r]);
        d_counts[r] = Kr;
        d_bytes[r] = a.h + Kr * a.L;
      }
    }
  }
  if (!bar.sync()) { if (tid == 0) atomicOr(status, kFaultTimeout); return; }

  // segment offsets, the radix width and the runs (every block for itself)
  auto seg = [&](int m) {
    const uint4 v = __ldcg(reinterpret_cast<const uint4*>(w.seg + m));
    return SegInfo{v.x, v.y, v.z, v.w};
  };
  if (tid == 0) { sm.maxbits = 0u; sm.maxruns = 0u; }
  seg_scan(sm, nseg, sm.key_off, [&](int m) {
    const SegInfo s = seg(m);
    if (s.kept) atomicMax(&sm.maxbits, (uint32_t)(32 - __clz((int)(s.end - s.lo - 1u))));
    return s.kept;
  });
  const uint32_t nkeys = sm.key_off[nseg];
  // one run of keys per block, as far as the segments' ends allow
  const uint32_t nblk = gridDim.x > 2u * nseg ? gridDim.x - nseg : gridDim.x;
  const uint32_t run = max((uint32_t)kRunMin, (nkeys / nblk + 32u) & ~31u);
  seg_scan(sm, nseg, sm.run_off, [&](int m) {
    const uint32_t n = (sm.key_off[m + 1] - sm.key_off[m] + run - 1) / run;
    atomicMax(&sm.maxruns, n);
    return n;
  });
  const int nruns = (int)sm.run_off[nseg];
  const int passes = sm.maxbits > 27u ? 4 : 3;
  const int wbits = max(5, ((int)sm.maxbits + passes - 1) / passes), nd = 1 << wbits;
  const bool wide = sm.maxruns > 32u;  // a block per 32 digits of a segment's runs, else a warp

  // 3. compaction in tile order: the block's kept tiles from its own histograms,
  // then, from the sums of the blocks before it, their places
  uint32_t mine = 0u;
  for (int m = m0; m < nseg && seg_begin(m) < t1; ++m) {
    const int end = (int)(seg(m).end >> kBinShift);
    const uint32_t* own = w.hist + ((size_t)blockIdx.x + m) * kBins;
    for (int i = tid; i < end; i += ST) mine += own[i];
  }
  {
    uint32_t tot;
    (void)block_exclusive_scan(mine, &tot, sm.ws);
    if (tid == 0) w.cnt[blockIdx.x] = tot;
  }
  if (!bar.sync()) { if (tid == 0) atomicOr(status, kFaultTimeout); return; }
  {
    uint32_t before = 0u, pos;
    for (int i = tid; i < (int)blockIdx.x; i += ST) before += __ldcg(w.cnt + i);
    (void)block_exclusive_scan(before, &pos, sm.ws);
    constexpr int CT = 12;  // consecutive tiles per thread and turn
    for (int m = m0; m < nseg && seg_begin(m) < t1; ++m) {
      const int64_t b = max(t0, seg_begin(m)), e = min(t1, seg_end(m));
      const SegInfo si = seg(m);
      uint4 v[CT / 4];
      auto load = [&](int64_t tt) {
#pragma unroll
        for (int u = 0; u < CT / 4; ++u)  // the last words may lie past T
          v[u] = tt + 4 * u < e ? *reinterpret_cast<const uint4*>(w.k1 + tt + 4 * u) : make_uint4(0u, 0u, 0u, 0u);
      };
      load((b & ~3ll) + CT * tid);
      for (int64_t tb = b & ~3ll; tb < e; tb += CT * ST) {
        const int64_t tt = tb + CT * tid;
        uint32_t f[CT], n = 0u;
#pragma unroll
        for (int u = 0; u < CT; u += 4) {
          f[u] = v[u / 4].x; f[u + 1] = v[u / 4].y; f[u + 2] = v[u / 4].z; f[u + 3] = v[u / 4].w;
        }
        load(tt + CT * ST);
#pragma unroll
        for (int u = 0; u < CT; ++u) {
          if (tt + u < b || tt + u >= e) f[u] = kIneligible;
          n += f[u] < si.end ? 1u : 0u;
        }
        uint32_t tot;
        uint32_t at = pos + block_exclusive_scan(n, &tot, sm.ws);
#pragma unroll
        for (int u = 0; u < CT; ++u) {
          if (f[u] < si.end) {
            w.k0[at] = f[u] - si.lo;
            w.v0[at] = (uint32_t)(tt + u);
            ++at;
          }
        }
        pos += tot;
      }
    }
  }
  if (!bar.sync()) { if (tid == 0) atomicOr(status, kFaultTimeout); return; }

  // 4. stable passes over wbits each
  uint32_t *kin = w.k0, *vin = w.v0, *kout = w.k1, *vout = w.v1;
  for (int ps = 0; ps < passes; ++ps) {
    const int shift = ps * wbits;
    for (int r = blockIdx.x; r < nruns; r += gridDim.x) {  // digits of each run
      const int m = find_seg(sm.run_off, nseg, (uint32_t)r);
      const uint32_t b = sm.key_off[m] + ((uint32_t)r - sm.run_off[m]) * run, n = min(run, sm.key_off[m + 1] - b);
      const uint32_t* kr = kin + b;
      for (int i = tid; i < nd; i += ST) sm.d.base[i] = 0u;
      __syncthreads();
      for (uint32_t k = tid; k < n; k += 4 * ST) {
        uint32_t f[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (k + u * ST < n) f[u] = __ldcg(kr + k + u * ST);
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (k + u * ST < n) atomicAdd(&sm.d.base[(f[u] >> shift) & (uint32_t)(nd - 1)], 1u);
      }
      __syncthreads();
      for (int i = tid; i < nd; i += ST) w.hist[(size_t)r * nd + i] = sm.d.base[i];
      __syncthreads();
    }
    if (!bar.sync()) { if (tid == 0) atomicOr(status, kFaultTimeout); return; }
    // exclusive prefixes over a segment's runs, 32 digits at a time
    const int groups = nd >> 5;
    if (wide) {
      for (int64_t t = blockIdx.x; t < (int64_t)nseg * groups; t += gridDim.x) {
        const int m = (int)(t / groups), d = (int)(t % groups) * 32 + lane;
        const uint32_t r0 = sm.run_off[m], n = sm.run_off[m + 1] - r0, sub = (n + SW - 1) / SW;
        const uint32_t rb = min(n, warp * sub), re = min(n, rb + sub);
        uint32_t* col = w.hist + (size_t)r0 * nd + d;
        uint32_t s = 0u;
#pragma unroll 8
        for (uint32_t r = rb; r < re; ++r) s += __ldcg(col + (size_t)r * nd);
        sm.part[warp][lane] = s;
        __syncthreads();
        uint32_t at = 0u;
        for (int i = 0; i < warp; ++i) at += sm.part[i][lane];
        if (warp == SW - 1) w.total[(size_t)m * nd + d] = at + s;
#pragma unroll 8
        for (uint32_t r = rb; r < re; ++r) {
          const uint32_t v = __ldcg(col + (size_t)r * nd);
          col[(size_t)r * nd] = at;
          at += v;
        }
        __syncthreads();
      }
    } else {
      for (int64_t t = (int64_t)blockIdx.x * SW + warp; t < (int64_t)nseg * groups; t += (int64_t)gridDim.x * SW) {
        const int m = (int)(t / groups), d = (int)(t % groups) * 32 + lane;
        const uint32_t r0 = sm.run_off[m], n = sm.run_off[m + 1] - r0;
        uint32_t* col = w.hist + (size_t)r0 * nd + d;
        uint32_t at = 0u;
#pragma unroll 8
        for (uint32_t r = 0; r < n; ++r) {
          const uint32_t v = __ldcg(col + (size_t)r * nd);
          col[(size_t)r * nd] = at;
          at += v;
        }
        w.total[(size_t)m * nd + d] = at;
      }
    }
    if (!bar.sync()) { if (tid == 0) atomicOr(status, kFaultTimeout); return; }
    // ranked scatter
    for (int r = blockIdx.x; r < nruns; r += gridDim.x) {
      const int m = find_seg(sm.run_off, nseg, (uint32_t)r);
      const uint32_t b = sm.key_off[m] + ((uint32_t)r - sm.run_off[m]) * run, n = min(run, sm.key_off[m + 1] - b);
      const uint32_t *kr = kin + b, *vr = vin + b;
      uint32_t f[kRankIpt], v[kRankIpt], rank[kRankIpt];
      // keys rb .. of the run: a warp takes 32 ipt consecutive ones
      auto per_warp = [&](uint32_t rb) { return (min((uint32_t)kRound, n - rb) + ST - 1) / ST; };
      auto load = [&](uint32_t rb) {
        const uint32_t ipt = per_warp(rb), kw = rb + 32u * ipt * warp + lane;
#pragma unroll
        for (int u = 0; u < kRankIpt; ++u) {
          const uint32_t k = kw + 32u * u;
          const bool in = (uint32_t)u < ipt && k < n;
          f[u] = in ? __ldcg(kr + k) : 0u;
          v[u] = in ? __ldcg(vr + k) : 0u;
        }
      };
      load(0u);
      for (int i = tid; i < SW * nd; i += ST) sm.r.mask[i >> wbits][i & (nd - 1)] = 0u;
      {  // first position of each digit of this run; a thread per digit
        const uint32_t tot = tid < nd ? __ldcg(w.total + (size_t)m * nd + tid) : 0u;
        const uint32_t own = tid < nd ? __ldcg(w.hist + (size_t)r * nd + tid) : 0u;
        const uint32_t at = sm.key_off[m] + block_exclusive_scan(tot, nullptr, sm.ws);
        if (tid < nd) sm.d.base[tid] = at + own;
      }
      for (uint32_t rb = 0; rb < n; rb += kRound) {
        const uint32_t left = min((uint32_t)kRound, n - rb), ipt = per_warp(rb);
        const uint32_t kw = rb + 32u * ipt * warp + lane;
        if (rb > 0u)  // the sorted keys of the last round lay here
          for (int i = tid; i < SW * nd; i += ST) sm.r.mask[i >> wbits][i & (nd - 1)] = 0u;
        for (int i = tid; i < SW * (nd >> 1); i += ST)
          reinterpret_cast<uint32_t*>(sm.r.wcnt[i >> (wbits - 1)])[i & ((nd >> 1) - 1)] = 0u;
        __syncthreads();
#pragma unroll
        for (int u = 0; u < kRankIpt; ++u) {
          if ((uint32_t)u >= ipt) break;
          // Lanes with the same digit, through a word of lane bits per digit in
          // shared memory (on 4096 keys: 7 us with one ballot per digit bit, more
          // than 20 with a match instruction, which takes the digits in turn).
          const bool in = kw + 32u * u < n;
          const uint32_t dg = (f[u] >> shift) & (uint32_t)(nd - 1);
          if (in) atomicOr(&sm.r.mask[warp][dg], 1u << lane);
          __syncwarp();
          uint32_t peers = 0u, c = 0u;
          if (in) {
            peers = sm.r.mask[warp][dg];
            c = sm.r.wcnt[warp][dg];
          }
          const uint32_t below = __popc(peers & ((1u << lane) - 1u));
          rank[u] = c + below;
          __syncwarp();
          if (in && below == 0u) {
            sm.r.mask[warp][dg] = 0u;
            sm.r.wcnt[warp][dg] = (uint16_t)(c + __popc(peers));
          }
          __syncwarp();
        }
        __syncthreads();
        // keys of earlier warps and of smaller digits of this round: where the
        // round's keys go in shared memory, sorted by digit
        uint32_t cnt = 0u;
        if (tid < nd) {
          uint16_t c[SW];
#pragma unroll
          for (int ww = 0; ww < SW; ++ww) c[ww] = sm.r.wcnt[ww][tid];
#pragma unroll
          for (int ww = 0; ww < SW; ++ww) {
            sm.r.wcnt[ww][tid] = (uint16_t)cnt;
            cnt += c[ww];
          }
        }
        const uint32_t at0 = block_exclusive_scan(cnt, nullptr, sm.ws);
        if (tid < nd) sm.d.first[tid] = at0;
        __syncthreads();
#pragma unroll
        for (int u = 0; u < kRankIpt; ++u) {
          if ((uint32_t)u < ipt && kw + 32u * u < n) {
            const uint32_t dg = (f[u] >> shift) & (uint32_t)(nd - 1);
            rank[u] += sm.d.first[dg] + sm.r.wcnt[warp][dg];
          }
        }
        __syncthreads();  // the counts are read: their memory takes the keys
#pragma unroll
        for (int u = 0; u < kRankIpt; ++u)
          if ((uint32_t)u < ipt && kw + 32u * u < n) sm.sorted[rank[u]] = make_uint2(f[u], v[u]);
        if (rb + kRound < n) load(rb + kRound);
        __syncthreads();
        // neighbouring threads now write neighbouring keys of a digit
        for (uint32_t i = tid; i < left; i += ST) {
          const uint2 kv = sm.sorted[i];
          const uint32_t dg = (kv.x >> shift) & (uint32_t)(nd - 1);
          const uint32_t at = sm.d.base[dg] + (i - sm.d.first[dg]);
          if (ps + 1 < passes) kout[at] = kv.x;
          vout[at] = kv.y;
        }
        __syncthreads();
        if (tid < nd) sm.d.base[tid] += cnt;
      }
      __syncthreads();
    }
    if (!bar.sync()) { if (tid == 0) atomicOr(status, kFaultTimeout); return; }
    uint32_t* t = kin; kin = kout; kout = t;
    t = vin; vin = vout; vout = t;
  }

  // 5. records and header
  uint32_t* rec_off = sm.rec_off;  // first record of each segment
  seg_scan(sm, nseg, rec_off, [&](int m) { return seg(m).K; });
  const uint32_t total = rec_off[nseg];
  uint32_t* per_mod = sm.run_off;
  // a copy of the modules' first tiles: lanes look up different ones, which
  // constant memory serves one at a time
  uint32_t* tile_off = sm.tile_off;
  if (pf) {
    for (int m = tid; m < a.n_mod; m += ST) {
      per_mod[m] = 0u;
      tile_off[m] = (uint32_t)a.tile_off[m];
    }
  }
  __syncthreads();
  // a run of records per block, as even as whole warps allow
  const int64_t share = ((int64_t)total / gridDim.x + 32) & ~31ll;
  const int64_t i1 = min((int64_t)total, (blockIdx.x + 1) * share);
  for (int64_t i0 = blockIdx.x * share; i0 < i1; i0 += kPackIpt * ST)
    pack_block(a, pr, vin, cands, stream, sm.key_off, rec_off, tile_off, per_mod, sm.buf, i0,
               (int)min((int64_t)kPackIpt * ST, i1 - i0));
  if (pf) {
    __syncthreads();
    for (int m = tid; m < a.n_mod; m += ST)
      if (per_mod[m]) atomicAdd(w.per_mod + m, per_mod[m]);
    if (!bar.sync()) { if (tid == 0) atomicOr(status, kFaultTimeout); return; }
  }
  if (blockIdx.x == 0) {
    for (int m = tid; m < a.n_mod; m += ST) {
      const uint32_t K = pf ? __ldcg(w.per_mod + m) : rec_off[m + 1] - rec_off[m];
      put_le(stream + 40 + 8 * m, (uint64_t)(a.tile_off[m + 1] - a.tile_off[m]), 4);
      put_le(stream + 44 + 8 * m, K, 4);
    }
    if (tid == 0) {
      put_header(a, pr, total, stream);
      if (!pf) d_bytes[0] = a.h + (int64_t)total * a.L;
    }
  }
}

// Offsets of the kernel's arrays in the workspace; [0, zero) is cleared by every
// call: the status word, the barrier, the module counts and the bins.
struct SelLayout {
  size_t bar, per_mod, bins, zero, seg, cnt, k0, v0, k1, v1, hist, total, bytes;
};

// Blocks worth launching: two rounds of tiles each (a barrier costs more, the more
// blocks meet at it), but one per segment at least, since a segment's bins, offsets and
// runs cost a block some microseconds however few tiles it has (700 modules of 7 tiles in
// three blocks took 4270 us).
int64_t want_blocks(const SelectPlan& sp, bool pf) {
  const int64_t by_tiles = (sp.T + 4 * ST - 1) / (4 * ST), by_segments = pf ? 1 : std::min<int64_t>(sp.n_mod, sp.T);
  return std::min(kMaxBlocks, std::max(by_tiles, by_segments));
}

SelLayout select_layout(const SelectPlan& sp, bool pf) {
  const size_t nseg = pf ? 1 : (size_t)sp.n_mod, T = (size_t)sp.T;
  // sort runs: one per block, and a shorter one per segment; rows of kBins counters for
  // step 1: row (block + segment) for each pair that meets, at most blocks + nseg - 1
  const size_t runs = (size_t)want_blocks(sp, pf) + 1 + nseg;
  SelLayout l;
  size_t off = kStatusBytes;
  auto take = [&off](size_t n) {
    const size_t at = off;
    off += align_up(n, 256);
    return at;
  };
  l.bar = take(2 * sizeof(unsigned));
  l.per_mod = take((size_t)sp.n_mod * 4);
  l.bins = take(nseg * kBins * 4);
  l.zero = off;
  l.seg = take(nseg * sizeof(SegInfo));
  l.cnt = take((size_t)kMaxBlocks * 4);
  l.k0 = take(T * 4);
  l.v0 = take(T * 4);
  l.k1 = take(T * 4);
  l.v1 = take(T * 4);
  l.hist = take(runs * std::max(kMaxDigits, kBins) * 4);
  l.total = take(nseg * kMaxDigits * 4);
  l.bytes = off;
  return l;
}

// SMs that kernels of stream `st` may use, of the device's nsm: fewer in a green
// context. A cooperative launch is checked against the device's count only, and
// blocks beyond what the stream's SMs hold would never meet the others at a barrier.
int stream_sms(cudaStream_t st, int nsm) {
  using GetCtx = CUresult (*)(CUstream, CUcontext*, CUgreenCtx*);
  using GetRes = CUresult (*)(CUgreenCtx, CUdevResource*, CUdevResourceType);
  auto entry = [](const char* name, unsigned version) {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult found = cudaDriverEntryPointSymbolNotFound;
    const cudaError_t e = cudaGetDriverEntryPointByVersion(name, &f, version, cudaEnableDefault, &found);
    return e == cudaSuccess && found == cudaDriverEntryPointSuccess ? f : nullptr;
  };
  static const GetCtx get_ctx = reinterpret_cast<GetCtx>(entry("cuStreamGetCtx", 12050));
  static const GetRes get_res = reinterpret_cast<GetRes>(entry("cuGreenCtxGetDevResource", 12040));
  CUcontext ctx = nullptr;
  CUgreenCtx green = nullptr;
  CUdevResource r;
  if (!get_ctx || !get_res || get_ctx(st, &ctx, &green) != CUDA_SUCCESS || !green ||
      get_res(green, &r, CU_DEV_RESOURCE_TYPE_SM) != CUDA_SUCCESS)
    return nsm;
  return std::max(1, std::min(nsm, (int)r.sm.smCount));
}

}  // namespace

size_t select_ws_bytes(const Prm& pr, const SelectPlan& sp) {
  return select_layout(sp, pr.variant != AWSRC_VARIANT_U).bytes;
}

awsrc_status select_run(const Prm& pr, const SelectPlan& sp, const int64_t* tile_off, const int64_t* kcap,
                        const awsrc_candidate* cands, uint8_t* stream_out, int64_t* d_counts, int64_t* d_bytes,
                        void* ws, size_t ws_bytes, cudaStream_t st) {
  if (sp.n_mod > kMaxSelMods || sp.n_rates > kMaxRates) return AWSRC_ERR_UNSUPPORTED;
  const bool pf = pr.variant != AWSRC_VARIANT_U;
  const SelLayout l = select_layout(sp, pf);
  if (ws_bytes < l.bytes) return AWSRC_ERR_WORKSPACE;
  SelArgs a;
  a.n_mod = sp.n_mod;
  a.n_rates = sp.n_rates;
  a.variant = pr.variant;
  a.T = sp.T;
  a.L = sp.L;
  a.h = sp.h;
  for (int m = 0; m <= sp.n_mod; ++m) a.tile_off[m] = tile_off[m];
  const int nk = pf ? sp.n_rates : sp.n_mod;
  for (int i = 0; i < nk; ++i) a.kcap[i] = kcap[i];
  uint8_t* p = static_cast<uint8_t*>(ws);
  SortWs w;
  w.bar = reinterpret_cast<unsigned*>(p + l.bar);
  w.per_mod = reinterpret_cast<uint32_t*>(p + l.per_mod);
  w.bins = reinterpret_cast<uint32_t*>(p + l.bins);
  w.seg = reinterpret_cast<SegInfo*>(p + l.seg);
  w.cnt = reinterpret_cast<uint32_t*>(p + l.cnt);
  w.k0 = reinterpret_cast<uint32_t*>(p + l.k0);
  w.v0 = reinterpret_cast<uint32_t*>(p + l.v0);
  w.k1 = reinterpret_cast<uint32_t*>(p + l.k1);
  w.v1 = reinterpret_cast<uint32_t*>(p + l.v1);
  w.hist = reinterpret_cast<uint32_t*>(p + l.hist);
  w.total = reinterpret_cast<uint32_t*>(p + l.total);
  uint32_t* status = static_cast<uint32_t*>(ws);

  cudaError_t e = cudaMemsetAsync(ws, 0, l.zero, st);
  if (e != cudaSuccess) return cuda_fail(e, "select: clear");
  int dev = 0, nsm = 0, per_sm = 0;
  const size_t smem = sizeof(SortSmem);
  const int64_t want = want_blocks(sp, pf);
  auto kern = want == 1                    ? select_kernel<kOneBlock>
              : pr.wait_ns == kWaitLimitNs ? select_kernel<kGrid>
                                           : select_kernel<kTestGrid>;
  if ((e = cudaGetDevice(&dev)) == cudaSuccess &&
      (e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) == cudaSuccess &&
      (e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, ST, smem);
  if (e != cudaSuccess) return cuda_fail(e, "select");
  // at most as many blocks as are resident at once
  const int64_t grid = std::max<int64_t>(1, std::min(want, (int64_t)stream_sms(st, nsm) * per_sm));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(ST);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;  // the grid barriers need every block resident
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, kern, cands, a, w, pr, stream_out, d_counts, d_bytes, status);
  note_launches(1);
  if (e != cudaSuccess) return cuda_fail(e, "select");
  return AWSRC_OK;
}

}  // namespace awsrc
