// The gaps of Eqs. 5-17 from the SET of 16-bit patterns a matrix (or a tile of one) holds.
//
// Neighbours in the sorted order that are equal contribute a gap of zero, so for 16-bit weights everything
// the proxy needs is which of the 65 536 patterns occur and how many weights there are: a bitmap of 8 KB
// instead of a sorted array or a table of 65 536 counters.  Marking is one shared-memory read per weight (and an
// atomic only the first time a pattern is met), so a streaming pass is bound by HBM, and the walk below touches
// 2 048 words.
#pragma once
#include <cuda_fp16.h>
#include <math.h>
#include <stdint.h>

namespace rwkvq {

constexpr int kPatternWords = 2048;        // bit p of the bitmap = bit (p & 31) of word p >> 5; p = raw bit pattern
constexpr int kGapList = 2048;             // gaps evaluated per round of the walk

__device__ __forceinline__ void mark_pattern(uint32_t* bm, uint32_t p) {
  uint32_t* w = bm + (p >> 5);
  if (!((*reinterpret_cast<volatile uint32_t*>(w) >> (p & 31u)) & 1u)) atomicOr(w, 1u << (p & 31u));
}
__device__ __forceinline__ void mark_pair(uint32_t* bm, uint32_t two) {
  mark_pattern(bm, two & 0xFFFFu);
  mark_pattern(bm, two >> 16);
}

// Value of a magnitude (the low 15 bits of a pattern).
__device__ __forceinline__ double magnitude_value(uint32_t mag, bool bf16) {
  return bf16 ? (double)__uint_as_float(mag << 16) : (double)__half2float(__ushort_as_half((unsigned short)mag));
}

// Natural logarithm of a positive normal number by table, after P. T. P. Tang, "Table-driven implementation of the logarithm function in
// IEEE floating-point arithmetic" (1990): with v = 2^e m and 1/c the table's reciprocal of the middle of m's interval (one of 128),
//   ln v = e ln 2 - ln(1/c) + ln(1 + r),   r = m (1/c) - 1 (one rounding), |r| <= 2^-8,
// and the series of ln(1 + r) up to r^7 leaves 2^-67.  Off by at most 2^-52 of the result or of ln 2, whichever is larger.  A gap's
// logarithm was most of its fp64 work: 25 operations a gap instead of about 90.
constexpr int kLogEntries = 128;
struct LogTable {
  double inv[kLogEntries], neg_log[kLogEntries];
};
__device__ __forceinline__ void fill_log_table(LogTable& t) {
  for (int i = threadIdx.x; i < kLogEntries; i += blockDim.x) {
    const double inv = 1.0 / (1.0 + ((double)i + 0.5) / kLogEntries);
    t.inv[i] = inv;
    t.neg_log[i] = -log(inv);
  }
}
__device__ __forceinline__ double log_by(const LogTable& t, double v) {
  const int hi = __double2hiint(v), i = (hi >> 13) & (kLogEntries - 1);
  const double m = __hiloint2double((hi & 0x000FFFFF) | 0x3FF00000, __double2loint(v));
  const double e = __hiloint2double(0x43300000, (int)((uint32_t)((hi >> 20) - 1023) ^ 0x80000000u)) - 4503601774854144.0;      // 2^52 + 2^31
  const double r = fma(m, t.inv[i], -1.0);
  double q = fma(r, 1.0 / 7.0, -1.0 / 6.0);
  q = fma(r, q, 0.2);
  q = fma(r, q, -0.25);
  q = fma(r, q, 1.0 / 3.0);
  q = fma(r, q, -0.5);
  return fma(e, 0.6931471805599453094, t.neg_log[i] + fma(r * r, q, r));
}

struct SetStats {
  double sum_glng;            // sum g' ln g' over the positive gaps
  double pw[7];               // sum t^k for k = 2..8 over the positive gaps, t = n g' - 1
  double abs_t, gmax, gmin;   // sum |t|, largest and smallest positive g'
  int distinct;
  bool nonfinite, degenerate; // degenerate: fewer than two distinct values or weights
};

template <int T>
struct SetShared {
  LogTable logs;
  int first[T / 32], last[T / 32], count[T / 32], bad[T / 32];
  uint32_t gaps[kGapList];    // magnitude << 16 | predecessor's magnitude
  uint32_t run_info[1024];    // of the runs that hold patterns: place of their first gap in the list << 16 | magnitude in front (0xFFFF: none)
  uint16_t run_id[1024];
  double red[T / 32][11];
};

// All T threads call it with the same bitmap and a filled table of logarithms, a barrier behind both; thread 0 receives the sums (the flags and
// `distinct` are valid in every thread).  `n` = weights - 1.  Thread t owns 1024 / T runs of 64 consecutive patterns.  Positive and negative patterns
// are two chains in order of magnitude, joined at zero if it occurs and by one gap across it if not.  Gaps
// between neighbouring patterns of a run (most of them, in a dense matrix) are all one ulp of the run's binade: they
// are counted and evaluated once; the others are put in a list and evaluated by all threads in turn.  The runs that hold patterns are dealt out
// over the threads for that: they lie close together, and listed by the threads that own them they kept a few warps busy (kernels for the tiles of 4096^2
// weights, with the table filled and the next vectors under way while a tile is marked: 256 x 256 of bf16 27.9 -> 23.2 us, of fp16 38.6 -> 31.3, 128 x
// 128 of fp16 83 -> 50, 1 x 4096 239 -> 121; a run by a warp, a pattern a lane: 222 for the last).  All sums have a
// fixed order, so results are reproducible.  kFamily: also sum |t| and the extreme gaps.
template <int T, bool kFamily = true>
__device__ void set_gaps(const uint32_t* bm, bool bf16, double n, int K, SetShared<T>& sh, SetStats& out) {
  static_assert(T % 64 == 0 && T <= 1024 && 1024 % T == 0, "block size");
  constexpr int P = 1024 / T, W = T / 32;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const bool zero = ((bm[0] | bm[kPatternWords / 2]) & 1u) != 0u;       // +0 and -0 are the same value
  const int inf_run = bf16 ? 0x7F80 / 64 : 0x7C00 / 64;
  int first = 0x10000, last = -1, count = 0, bad = 0;
  uint64_t bits[P];
#pragma unroll
  for (int i = 0; i < P; ++i) {
    const int run = t * P + i, mrun = run & 511;
    uint64_t b = *reinterpret_cast<const uint64_t*>(bm + 2 * run);
    if (mrun == 0) b = (b & ~1ull) | (zero ? 1ull : 0ull);
    if (mrun >= inf_run) { bad |= b != 0ull; b = 0ull; }
    bits[i] = b;
    if (b) {
      first = min(first, mrun * 64 + __ffsll((long long)b) - 1);
      last = mrun * 64 + 63 - __clzll((long long)b);
      count += __popcll(b);
    }
  }
  // predecessor of this thread's first pattern within its side (warps 0 .. W/2 - 1 hold the positive side)
  int prev = last, mn = first, cnt = count;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int v = __shfl_up_sync(0xFFFFFFFFu, prev, d);
    if (lane >= d) prev = max(prev, v);
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    mn = min(mn, __shfl_xor_sync(0xFFFFFFFFu, mn, d));
    cnt += __shfl_xor_sync(0xFFFFFFFFu, cnt, d);
  }
  const int any_bad = __any_sync(0xFFFFFFFFu, bad);
  if (lane == 31) { sh.last[warp] = prev; sh.first[warp] = mn; sh.count[warp] = cnt; sh.bad[warp] = any_bad; }
  prev = __shfl_up_sync(0xFFFFFFFFu, prev, 1);
  if (lane == 0) prev = -1;
  __syncthreads();
  int lo[2] = {0x10000, 0x10000}, hi[2] = {-1, -1}, distinct = zero ? -1 : 0, nf = 0;
  for (int w = 0; w < W; ++w) {
    const int side = w >= W / 2;
    if (w < warp && side == (warp >= W / 2)) prev = max(prev, sh.last[w]);
    lo[side] = min(lo[side], sh.first[w]);
    hi[side] = max(hi[side], sh.last[w]);
    distinct += sh.count[w];
    nf |= sh.bad[w];
  }
  out.distinct = distinct; out.nonfinite = nf != 0;
  out.degenerate = distinct < 2 || n < 1.0;
  if (out.degenerate) return;
  const double vmax = hi[0] >= 0 ? magnitude_value((uint32_t)hi[0], bf16) : -magnitude_value((uint32_t)lo[1], bf16);
  const double vmin = hi[1] >= 0 ? -magnitude_value((uint32_t)hi[1], bf16) : magnitude_value((uint32_t)lo[0], bf16);
  const double inv_R = 1.0 / (vmax - vmin);
  double acc[11];
#pragma unroll
  for (int i = 0; i < 11; ++i) acc[i] = 0.0;
  acc[10] = INFINITY;
  auto add = [&](double gap, double times) {
    const double gp = gap * inv_R, tt = n * gp - 1.0;
    acc[0] += times * (gp * log_by(sh.logs, gp));
    double pw = tt;
#pragma unroll
    for (int k = 2; k <= 8; ++k)
      if (k <= K) { pw *= tt; acc[k - 1] += times * pw; }
    if (kFamily) {
      acc[8] += times * fabs(tt);
      acc[9] = fmax(acc[9], gp);
      acc[10] = fmin(acc[10], gp);
    }
  };
  if (t == 0 && !zero && hi[0] >= 0 && hi[1] >= 0) add(magnitude_value((uint32_t)lo[0], bf16) + magnitude_value((uint32_t)lo[1], bf16), 1.0);
  // the list: this thread's runs that hold patterns, and how many gaps longer than one pattern they have
  auto lone_of = [](uint64_t b, bool first_of_side) -> uint64_t {      // patterns whose neighbour below is not in the run
    const uint64_t lone = b & ~(b << 1);
    return first_of_side ? lone & (lone - 1ull) : lone;                // a side's smallest magnitude has no gap in front
  };
  int mine = 0, before = prev;                     // gaps, and runs << 17
#pragma unroll
  for (int i = 0; i < P; ++i) {
    if (!bits[i]) continue;
    mine += __popcll(lone_of(bits[i], before < 0)) + (1 << 17);
    before = ((t * P + i) & 511) * 64 + 63 - __clzll(bits[i]);
  }
  int incl = mine;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int v = __shfl_up_sync(0xFFFFFFFFu, incl, d);
    if (lane >= d) incl += v;
  }
  __syncthreads();                                 // sh.count is reused
  if (lane == 31) sh.count[warp] = incl;
  __syncthreads();
  int pos = incl - mine, total = 0;
  for (int w = 0; w < W; ++w) {
    if (w < warp) pos += sh.count[w];
    total += sh.count[w];
  }
  const int runs = total >> 17;
  total &= (1 << 17) - 1;
  before = prev;
#pragma unroll
  for (int i = 0; i < P; ++i) {
    if (!bits[i]) continue;
    sh.run_info[pos >> 17] = (uint32_t)pos << 16 | ((uint32_t)before & 0xFFFFu);       // at most 32 gaps a run: 32 768
    sh.run_id[pos >> 17] = (uint16_t)(t * P + i);
    pos += __popcll(lone_of(bits[i], before < 0)) + (1 << 17);
    before = ((t * P + i) & 511) * 64 + 63 - __clzll(bits[i]);
  }
  __syncthreads();
  auto run_bits = [&](int run) -> uint64_t {
    const uint64_t b = *reinterpret_cast<const uint64_t*>(bm + 2 * run);
    return (run & 511) == 0 ? (b & ~1ull) | (zero ? 1ull : 0ull) : b;
  };
  for (int k = t; k < runs; k += T) {
    const int run = sh.run_id[k];
    const uint64_t b = run_bits(run), adj = b & (b << 1);
    const uint32_t base = (uint32_t)(run & 511) * 64u;
    if (adj) add(magnitude_value(base + 1u, bf16) - magnitude_value(base, bf16), (double)__popcll(adj));
  }
  for (int c0 = 0; c0 < total; c0 += kGapList) {
    const int c1 = min(c0 + kGapList, total);
    for (int k = t; k < runs; k += T) {
      const uint32_t info = sh.run_info[k];
      int j = (int)(info >> 16);
      const int stop = k + 1 < runs ? (int)(sh.run_info[k + 1] >> 16) : total;
      if (j >= c1 || stop <= max(j, c0)) continue;
      const int run = sh.run_id[k];
      const uint64_t b = run_bits(run), lone = lone_of(b, (info & 0xFFFFu) == 0xFFFFu);
      uint32_t base = (uint32_t)(run & 511) * 64u, front = info & 0xFFFFu;
#pragma unroll
      for (int h = 0; h < 2; ++h, base += 32u) {
        const uint32_t word = (uint32_t)(b >> (32 * h));
        for (uint32_t alone = (uint32_t)(lone >> (32 * h)); alone; alone &= alone - 1u, ++j) {
          const uint32_t below = word & ((alone & (0u - alone)) - 1u);
          const uint32_t p = below ? base + 31u - __clz((int)below) : front;
          if (j >= c0 && j < c1) sh.gaps[j - c0] = (base + (uint32_t)__ffs((int)alone) - 1u) << 16 | p;
        }
        if (word) front = base + 31u - __clz((int)word);
      }
    }
    __syncthreads();
    for (int j = t; j < c1 - c0; j += T)
      add(magnitude_value(sh.gaps[j] >> 16, bf16) - magnitude_value(sh.gaps[j] & 0xFFFFu, bf16), 1.0);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 11; ++i) {
    if (i >= (kFamily ? 11 : 8)) break;
    if (i >= K && i < 8) continue;                 // sums of powers that are not asked for
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      const double o = __shfl_xor_sync(0xFFFFFFFFu, acc[i], d);
      acc[i] = i == 9 ? fmax(acc[i], o) : i == 10 ? fmin(acc[i], o) : acc[i] + o;
    }
    if (lane == 0) sh.red[warp][i] = acc[i];
  }
  __syncthreads();
  if (t == 0) {
#pragma unroll
    for (int i = 0; i < (kFamily ? 11 : 8); ++i) acc[i] = i >= K && i < 8 ? 0.0 : sh.red[0][i];
    for (int w = 1; w < W; ++w) {
#pragma unroll
      for (int i = 0; i < (kFamily ? 11 : 8); ++i) {
        if (i >= K && i < 8) continue;
        const double o = sh.red[w][i];
        acc[i] = i == 9 ? fmax(acc[i], o) : i == 10 ? fmin(acc[i], o) : acc[i] + o;
      }
    }
    out.sum_glng = acc[0];
#pragma unroll
    for (int i = 0; i < 7; ++i) out.pw[i] = acc[i + 1];
    out.abs_t = acc[8]; out.gmax = acc[9]; out.gmin = acc[10];
  }
}

// P_c of Eq. 9 and P_f of Eq. 17 from the sums; `n` = weights - 1, the n - (distinct - 1) ties have t = -1.  Two weights have one gap, R itself, and
// proxies of zero: by its reciprocal the gap over R is 1 - 2^-53 for one in nine, and a threshold of zero would choose SQ.
__device__ __forceinline__ void proxy_from_set(const SetStats& s, double n, int K, double* pc, double* pf) {
  const double ties = n - (double)(s.distinct - 1);
  double f = 0.0;
  for (int k = 2; k <= K; ++k) f += fabs((s.pw[k - 2] + ((k & 1) ? -ties : ties)) / n) / (double)(k * (k - 1));
  *pc = n == 1.0 ? 0.0 : log(n) + s.sum_glng;
  *pf = n == 1.0 ? 0.0 : f;
}

}  // namespace rwkvq
