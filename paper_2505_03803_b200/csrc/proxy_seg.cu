// Coarse-to-fine proxy (Section 4.1) at finer granularity and for other input types.
//
// The paper evaluates the proxy per weight matrix and names finer granularity as future work; its
// inputs are the model's weights, whatever their type.  Two routes besides the fp16 histogram of
// proxy.cu:
//   * segments -- every seg_rows x seg_cols tile of a matrix (one output channel = a 1 x ic tile,
//     one block = e.g. 256 x 256) is reduced by ONE thread block in shared memory: 16-bit types through the
//     set of patterns that occur (proxy_core.cuh), fp32 by sorting order-preserving
//     integer keys (the sort of Eq. 5 literally), gaps reduced in fp64 in a fixed order (Eqs. 6-17);
//   * a whole fp32 matrix too large for shared memory is sorted by the radix sort of the CUDA
//     toolkit's CUB (a library primitive for the sort of Eq. 5), then the same gap reduction runs over
//     the sorted array in two fixed-order passes.
// Formulas as in proxy.cu: n gaps (n = count - 1), R = sum of gaps, g' = gap / R,
//   P_c = ln n + sum g' ln g'  (0 ln 0 := 0),   t = n g' - 1,
//   P_f = sum_{k=2..K} | sum t^k / n | / (k (k-1)).
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <cub/device/device_radix_sort.cuh>
#include <vector>

#include "../../include/rwkvq.h"
#include "host_util.h"
#include "proxy_core.cuh"
#include "unpack.cuh"

namespace rwkvq {
namespace pseg {

constexpr uint32_t kSmemKeysBytes = 131072;        // a tile holds at most 65 536 16-bit or 32 768 32-bit weights
constexpr int kMaxK = 8;

struct SegResult {
  double pc, pf;
  unsigned count;
  int nonfinite;
};

// Order-preserving keys: flip all bits of negatives, the sign bit of the others.
__device__ __forceinline__ uint32_t key32(uint32_t bits) { return (bits & 0x80000000u) ? ~bits : (bits | 0x80000000u); }
__device__ __forceinline__ uint32_t bits_of_key32(uint32_t key) { return (key & 0x80000000u) ? (key & 0x7FFFFFFFu) : ~key; }
__device__ __forceinline__ double value_of_key32(uint32_t key) { return (double)__uint_as_float(bits_of_key32(key)); }

// Terms of one gap (the difference of two neighbouring sorted values, already divided by R).
__device__ __forceinline__ void gap_terms(const LogTable& logs, double gp, double n, int K, double (&acc)[kMaxK]) {
  if (gp > 0.0) acc[0] += gp * log_by(logs, gp);
  const double t = n * gp - 1.0;
  double pw = t * t;
  acc[1] += pw;
  if (K > 2) { pw *= t; acc[2] += pw; }
  if (K > 3) { pw *= t; acc[3] += pw; }
  if (K > 4) {
#pragma unroll
    for (int k = 5; k <= kMaxK; ++k)
      if (k <= K) { pw *= t; acc[k - 1] += pw; }
  }
}
__device__ __forceinline__ void finish(const double (&tot)[kMaxK], double n, int K, SegResult* res) {
  double pf = 0.0;
  for (int k = 2; k <= K; ++k) pf += fabs(tot[k - 1] / n) / (double)(k * (k - 1));
  res->pc = log(n) + tot[0];
  res->pf = pf;
}

// 16-bit types: one block of T threads per tile marks the tile's patterns (8 KB) and walks them.  `wide`: rows start on
// 16-byte boundaries and hold whole vectors of eight.  A 256 x 256 tile by the bitonic network in 128 KB of
// shared memory took two waves of 0.4 ms; this form holds two or more tiles per SM.
template <int T, int CTAS>
__global__ void __launch_bounds__(T, CTAS) proxy_segment_set_kernel(const uint16_t* w, int oc, int ic, int seg_rows, int seg_cols, int wide,
                                                                   int bf16, int K, SegResult* out) {
  __shared__ __align__(16) uint32_t bm[kPatternWords];
  __shared__ SetShared<T> sh;
  const int r0 = blockIdx.y * seg_rows, c0 = blockIdx.x * seg_cols;
  const int nr = min(seg_rows, oc - r0), nc = min(seg_cols, ic - c0);
  for (int j = threadIdx.x; j < kPatternWords / 4; j += T) reinterpret_cast<uint4*>(bm)[j] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  const uint16_t* src = w + (size_t)r0 * ic + c0;
  if (wide) {
    // the next vectors, or the table of logarithms, are on their way while these are marked
    const int per_row = nc >> 3, total = nr * per_row, step_r = T / per_row, step_c = T % per_row;
    int r = threadIdx.x / per_row, c = threadIdx.x % per_row;
    uint4 v[4], next[4];
    auto fetch = [&](uint4 (&to)[4], int i0) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (i0 + u * T < total) to[u] = ldg_stream(src + (size_t)r * ic + 8 * c);
        r += step_r; c += step_c;
        if (c >= per_row) { c -= per_row; ++r; }
      }
    };
    fetch(v, threadIdx.x);
    fill_log_table(sh.logs);
    for (int i0 = threadIdx.x; i0 < total; i0 += 4 * T) {
      fetch(next, i0 + 4 * T);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (i0 + u * T < total) { mark_pair(bm, v[u].x); mark_pair(bm, v[u].y); mark_pair(bm, v[u].z); mark_pair(bm, v[u].w); }
        v[u] = next[u];
      }
    }
  } else {
    fill_log_table(sh.logs);
    const int total = nr * nc;
    for (int i = threadIdx.x; i < total; i += T) mark_pattern(bm, src[(size_t)(i / nc) * ic + i % nc]);
  }
  __syncthreads();
  const double n = (double)(nr * nc - 1);
  SetStats s;
  set_gaps<T, false>(bm, bf16 != 0, n, K, sh, s);
  if (threadIdx.x == 0) {
    SegResult r;
    r.pc = r.pf = INFINITY; r.count = (unsigned)(nr * nc); r.nonfinite = s.nonfinite ? 1 : 0;
    if (!s.nonfinite && !s.degenerate) proxy_from_set(s, n, K, &r.pc, &r.pf);
    out[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = r;
  }
}

// fp32: one block of T threads, KPT keys each, per segment: tile (blockIdx.y, blockIdx.x) of seg_rows x seg_cols elements, ragged at the
// right and bottom edges.  The keys are sorted in shared memory in one pass: counted in buckets by sign, exponent and the leading 23 - SHIFT
// mantissa bits (sixteen octaves below the tile's largest magnitude, the rest in one bucket a sign), put into their buckets, and then every key
// counts the smaller ones of its own bucket: in the densest octave of a Gaussian tile four.  A tile with more than 255 keys in one bucket, or
// more comparisons a key than kMostCompared (many equal weights, or all of them close together around a number other than zero), is sorted by a
// bitonic network instead, as every tile was before, unless it has one value only.  Bound by instructions (about 300 a key and warp, 66 % of the issue
// slots).  Calls of 4096^2 weights, us, tiles of 128 x 256, 128 x 128 and 1 x 4096, by the network -> by this:
// Gaussian 1054 -> 290, 907 -> 254, 1039 -> 260; of bf16 numbers 1073 -> 389, 931 -> 318, 1066 -> 263; half of them zero 1026 -> 947, 881 -> 809, 1028 -> 605;
// around one 1071 -> 971, 918 -> 826, 1038 -> 624; one value 865 -> 156, 731 -> 155, 752 -> 155; 256 values alike often 1034 -> 805, 902 -> 491, 1058 -> 333.
template <int T, int KPT, int SHIFT, int CTAS>
struct TileSort {
  static constexpr int kSide = 16 << (23 - SHIFT);       // buckets of a sign
  static constexpr int kKeys = T * KPT;
  // From there the network is faster: by ranks, 64 / 128 comparisons a key, tiles of 128 x 256 525 / 805 us and by the network 920; of 128 x 128 491 / 739
  // and 790; of 1 x 4096, 32 / 43 / 64 comparisons, 393 / 463 / 546 and 593.
  static constexpr uint32_t kMostCompared = T == 1024 ? 140 : 72;
  static constexpr size_t kSmem = (size_t)(kKeys + 4) * 4 + (size_t)kSide * 8;     // four keys of padding
};
template <int T, int KPT, int SHIFT, int CTAS>
__global__ void __launch_bounds__(T, CTAS) proxy_segment_f32_kernel(const uint32_t* src, int oc, int ic, int seg_rows, int seg_cols,
                                                                  int K, SegResult* out) {
  using S = TileSort<T, KPT, SHIFT, CTAS>;
  constexpr int kWarps = T / 32, kPer = 2 * S::kSide / T;          // counters a thread
  static_assert(kPer % 4 == 0 && KPT % 4 == 0, "vectors");
  extern __shared__ __align__(16) uint8_t smem_raw[];
  uint32_t* keys = reinterpret_cast<uint32_t*>(smem_raw);
  uint32_t* starts = keys + S::kKeys + 4;        // of the buckets; counts at first
  __shared__ LogTable logs;
  __shared__ double red[kWarps][kMaxK], total[kMaxK];
  __shared__ uint32_t warp_sum[kWarps], s_max, s_compared;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r0 = blockIdx.y * seg_rows, c0 = blockIdx.x * seg_cols;
  const int nr = min(seg_rows, oc - r0), nc = min(seg_cols, ic - c0);
  const int count = nr * nc;
  SegResult* res = out + (size_t)blockIdx.y * gridDim.x + blockIdx.x;
  fill_log_table(logs);
  for (int i = tid; i < S::kSide / 2; i += T) reinterpret_cast<uint4*>(starts)[i] = make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) s_max = s_compared = 0u;
  __syncthreads();
  uint32_t b[KPT];
  uint32_t top = 0u;
  {
    const int step_r = T / nc, step_c = T % nc;
    int r = tid / nc, c = tid % nc;
    const uint32_t* base = src + (size_t)r0 * ic + c0;
#pragma unroll
    for (int j = 0; j < KPT; ++j) {
      b[j] = 0u;
      if (tid + j * T < count) b[j] = __ldg(base + (size_t)r * ic + c);
      r += step_r; c += step_c;
      if (c >= nc) { c -= nc; ++r; }
    }
#pragma unroll
    for (int j = 0; j < KPT; ++j) top = max(top, b[j] & 0x7FFFFFFFu);
  }
  top = __reduce_max_sync(0xFFFFFFFFu, top);
  if (lane == 0) atomicMax(&s_max, top);
  __syncthreads();
  top = s_max;
  const bool bad = top >= 0x7F800000u;
  if (bad || count < 2) {
    if (tid == 0) { res->pc = INFINITY; res->pf = INFINITY; res->count = (unsigned)count; res->nonfinite = bad ? 1 : 0; }
    return;
  }
  // bucket of a key, in the order of the keys
  const int top_at = (int)(top >> SHIFT);
  auto bucket = [&](uint32_t key) -> int {
    const uint32_t positive = (uint32_t)((int)key >> 31);            // all ones or zero
    const int below = min(top_at - (int)(((key ^ ~positive) & 0x7FFFFFFFu) >> SHIFT), S::kSide - 1);
    return below ^ (int)(positive & (2 * S::kSide - 1));
  };
  uint32_t came[KPT / 4];                        // keys of the same bucket that came before, four to a word; only used where they are at most 255
#pragma unroll
  for (int j = 0; j < KPT; ++j) {
    if (j % 4 == 0) came[j / 4] = 0u;
    b[j] = key32(b[j]);
    if (tid + j * T < count) came[j / 4] |= (atomicAdd(starts + bucket(b[j]), 1u) & 0xFFu) << (8 * (j % 4));
  }
  __syncthreads();
  bool many = false;
  {
    uint32_t sum = 0u, compared = 0u;
    uint4* const mine = reinterpret_cast<uint4*>(starts + tid * kPer);
#pragma unroll
    for (int i = 0; i < kPer / 4; ++i) {
      const uint4 v = mine[i];
      sum += v.x + v.y + v.z + v.w;
      many |= max(max(v.x, v.y), max(v.z, v.w)) > 255u;
      compared += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;      // 2^30 at most
    }
    uint32_t incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, d);
      if (lane >= d) incl += v;
    }
    if (lane == 31) warp_sum[warp] = incl;
    compared = __reduce_add_sync(0xFFFFFFFFu, compared);
    if (lane == 0) atomicAdd(&s_compared, compared);
    __syncthreads();
    many |= s_compared > S::kMostCompared * (uint32_t)count;
    uint32_t at = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? warp_sum[lane] : 0u) + incl - sum;
#pragma unroll
    for (int i = 0; i < kPer / 4; ++i) {
      const uint4 v = mine[i];
      mine[i] = make_uint4(at, at + v.x, at + v.x + v.y, at + v.x + v.y + v.z);
      at += v.x + v.y + v.z + v.w;
    }
  }
  many = __syncthreads_or(many);
  if (!many) {
    if (tid < 4) keys[count + tid] = 0xFFFFFFFFu;
#pragma unroll
    for (int j = 0; j < KPT; ++j)
      if (tid + j * T < count) keys[starts[bucket(b[j])] + ((came[j / 4] >> (8 * (j % 4))) & 0xFFu)] = b[j];
    __syncthreads();
#pragma unroll
    for (int j = 0; j < KPT; ++j) {
      if (j % 4 == 0) came[j / 4] = 0u;
      const int p = tid + j * T;
      if (p >= count) continue;
      const uint32_t k = keys[p];
      const int bk = bucket(k), first = (int)starts[bk], stop = bk + 1 < 2 * S::kSide ? (int)starts[bk + 1] : count;
      // the buckets behind hold larger keys, so steps of four may overshoot; equal ones keep the order of their places
      uint32_t smaller = 0u;
      for (int q = first; q < stop; q += 4) {
#pragma unroll
        for (int i = 0; i < 4; ++i) smaller += keys[q + i] < k + (q + i < p ? 1u : 0u) ? 1u : 0u;
      }
      b[j] = k;
      came[j / 4] |= smaller << (8 * (j % 4));
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < KPT; ++j)
      if (tid + j * T < count) keys[starts[bucket(b[j])] + ((came[j / 4] >> (8 * (j % 4))) & 0xFFu)] = b[j];
    __syncthreads();
  } else {
    // all equal (every bit of a key the same, or zeros of either sign): nothing to sort
    const float one = __uint_as_float(__ldg(src + (size_t)r0 * ic + c0));
    bool same = true;
#pragma unroll
    for (int j = 0; j < KPT; ++j) same &= tid + j * T >= count || __uint_as_float(bits_of_key32(b[j])) == one;
    if (__syncthreads_and(same)) {
      if (tid == 0) { res->pc = INFINITY; res->pf = INFINITY; res->count = (unsigned)count; res->nonfinite = 0; }
      return;
    }
    // bitonic sorting network, ascending; the padding keys are the largest and end up behind the data
#pragma unroll
    for (int j = 0; j < KPT; ++j)
      if (tid + j * T < count) keys[tid + j * T] = b[j];
    int np2 = 2;
    while (np2 < count) np2 <<= 1;
    for (int i = count + tid; i < np2; i += T) keys[i] = 0xFFFFFFFFu;
    __syncthreads();
    for (int size = 2; size <= np2; size <<= 1)
      for (int stride = size >> 1; stride > 0; stride >>= 1) {
        for (int p = tid; p < np2 / 2; p += T) {
          const int lo = 2 * p - (p & (stride - 1));          // index with the `stride` bit clear
          const int hi = lo + stride;
          const bool up = (lo & size) == 0;
          const uint32_t a = keys[lo], c = keys[hi];
          if ((a > c) == up) { keys[lo] = c; keys[hi] = a; }
        }
        __syncthreads();
      }
  }
  const double R = value_of_key32(keys[count - 1]) - value_of_key32(keys[0]), n = (double)(count - 1);
  if (!(R > 0.0)) {     // constant segment: G' is undefined
    if (tid == 0) { res->pc = INFINITY; res->pf = INFINITY; res->count = (unsigned)count; res->nonfinite = 0; }
    return;
  }
  const double inv_R = 1.0 / R;
  double acc[kMaxK];
#pragma unroll
  for (int i = 0; i < kMaxK; ++i) acc[i] = 0.0;
  for (int i = tid; i + 1 < count; i += T) {
    // gap / R by its reciprocal with one correction: a tile of two weights has a gap of one, exactly, and proxies of zero
    const double gap = value_of_key32(keys[i + 1]) - value_of_key32(keys[i]), q = gap * inv_R;
    gap_terms(logs, fma(fma(-q, R, gap), inv_R, q), n, K, acc);
  }
#pragma unroll
  for (int i = 0; i < kMaxK; ++i) {
    if (i >= K) break;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) acc[i] += __shfl_xor_sync(0xFFFFFFFFu, acc[i], d);
    if (lane == 0) red[warp][i] = acc[i];
  }
  __syncthreads();
  if (tid < kMaxK) {
    double sum = 0.0;
    if (tid < K)
      for (int w = 0; w < kWarps; ++w) sum += red[w][tid];
    total[tid] = sum;
  }
  __syncthreads();
  if (tid == 0) { finish(total, n, K, res); res->count = (unsigned)count; res->nonfinite = 0; }
}

// ---- whole fp32 matrix: keys sorted by the library's radix sort, then two fixed-order passes ----
__global__ void __launch_bounds__(256) f32_keys_kernel(const uint32_t* w, unsigned long long count, uint32_t* keys, int* nonfinite) {
  int bad = 0;
  for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < count;
       i += (unsigned long long)gridDim.x * blockDim.x) {
    const uint32_t b = w[i];
    if ((b & 0x7F800000u) == 0x7F800000u) bad = 1;
    keys[i] = key32(b);
  }
  if (bad) *nonfinite = 1;
}
constexpr int kGapBlocks = 1024;      // partial sums: [kGapBlocks][kMaxK] doubles, summed in block order
__global__ void __launch_bounds__(256) f32_gap_partials_kernel(const uint32_t* sorted, unsigned long long count, int K, double* partials) {
  __shared__ double red[256];
  __shared__ LogTable logs;
  fill_log_table(logs);
  __syncthreads();
  const double vmin = (double)__uint_as_float(bits_of_key32(sorted[0]));
  const double vmax = (double)__uint_as_float(bits_of_key32(sorted[count - 1]));
  const double R = vmax - vmin, n = (double)(count - 1);
  double acc[kMaxK];
#pragma unroll
  for (int i = 0; i < kMaxK; ++i) acc[i] = 0.0;
  if (R > 0.0) {
    const unsigned long long per = (count - 1 + kGapBlocks - 1) / kGapBlocks;
    const unsigned long long lo = (unsigned long long)blockIdx.x * per;
    const unsigned long long hi = lo + per < count - 1 ? lo + per : count - 1;
    for (unsigned long long i = lo + threadIdx.x; i < hi; i += blockDim.x) {
      const double a = (double)__uint_as_float(bits_of_key32(sorted[i])), b = (double)__uint_as_float(bits_of_key32(sorted[i + 1]));
      gap_terms(logs, (b - a) / R, n, K, acc);
    }
  }
  for (int q = 0; q < kMaxK; ++q) {
    __syncthreads();
    red[threadIdx.x] = acc[q];
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
      if ((int)threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
      __syncthreads();
    }
    if (threadIdx.x == 0) partials[(size_t)blockIdx.x * kMaxK + q] = red[0];
  }
}
__global__ void f32_gap_final_kernel(const uint32_t* sorted, unsigned long long count, int K, const double* partials,
                                     const int* nonfinite, SegResult* res) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  res->count = (unsigned)count; res->nonfinite = *nonfinite;
  const double vmin = (double)__uint_as_float(bits_of_key32(sorted[0]));
  const double vmax = (double)__uint_as_float(bits_of_key32(sorted[count - 1]));
  if (*nonfinite || count < 2 || !(vmax - vmin > 0.0)) { res->pc = INFINITY; res->pf = INFINITY; return; }
  double tot[kMaxK];
  for (int q = 0; q < kMaxK; ++q) {
    double s = 0.0;
    for (int b = 0; b < kGapBlocks; ++b) s += partials[(size_t)b * kMaxK + q];
    tot[q] = s;
  }
  finish(tot, (double)(count - 1), K, res);
}

template <int T, int KPT, int SHIFT, int CTAS>
static cudaError_t launch_f32(const uint32_t* w, int oc, int ic, int seg_rows, int seg_cols, int K, SegResult* res, dim3 grid, cudaStream_t s) {
  constexpr size_t smem = TileSort<T, KPT, SHIFT, CTAS>::kSmem;
  static SmemOptIn opt_in;
  const cudaError_t e = opt_in((const void*)proxy_segment_f32_kernel<T, KPT, SHIFT, CTAS>, (int)smem);
  if (e == cudaSuccess) proxy_segment_f32_kernel<T, KPT, SHIFT, CTAS><<<grid, T, smem, s>>>(w, oc, ic, seg_rows, seg_cols, K, res);
  return e;
}
static size_t elem_bytes(int dtype) { return dtype == RWKVQ_F32 ? 4 : 2; }

}  // namespace pseg
}  // namespace rwkvq

using namespace rwkvq;

extern "C" {

size_t rwkvq_proxy_segments_workspace_bytes(int oc, int ic, int seg_rows, int seg_cols) {
  if (oc <= 0 || ic <= 0 || seg_rows <= 0 || seg_cols <= 0) return 0;
  const size_t nseg = (size_t)((oc + seg_rows - 1) / seg_rows) * (size_t)((ic + seg_cols - 1) / seg_cols);
  return round_up_sz(nseg * sizeof(pseg::SegResult), 256);
}

rwkvq_status rwkvq_proxy_segments(const void* w, int dtype, int oc, int ic, int seg_rows, int seg_cols, int K, double tau_c,
                                  double tau_f, double* Pc, double* Pf, int* phi, void* ws, size_t ws_bytes, void* stream) {
  if (!w || !Pc || !Pf || !phi || oc <= 0 || ic <= 0 || seg_rows <= 0 || seg_cols <= 0) return RWKVQ_EINVAL;
  if (dtype != RWKVQ_F16 && dtype != RWKVQ_BF16 && dtype != RWKVQ_F32) return RWKVQ_EINVAL;
  if (K < 2 || K > pseg::kMaxK) return RWKVQ_EINVAL;
  if (seg_rows > oc) seg_rows = oc;
  if (seg_cols > ic) seg_cols = ic;
  const long long seg_elems = (long long)seg_rows * seg_cols;
  if (seg_elems > (long long)(pseg::kSmemKeysBytes / pseg::elem_bytes(dtype))) return RWKVQ_EUNSUPPORTED;
  if (!aligned16(w)) return RWKVQ_EALIGN;
  const size_t need = rwkvq_proxy_segments_workspace_bytes(oc, ic, seg_rows, seg_cols);
  if (!ws || ws_bytes < need) return RWKVQ_ENOMEM;
  if (!aligned16(ws)) return RWKVQ_EALIGN;
  const int gx = (ic + seg_cols - 1) / seg_cols, gy = (oc + seg_rows - 1) / seg_rows;
  if (gy > 65535) return RWKVQ_EUNSUPPORTED;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const size_t nseg = (size_t)gx * gy;
  pseg::SegResult* const pinned = static_cast<pseg::SegResult*>(pinned_results(nseg * sizeof(pseg::SegResult)));
  pseg::SegResult* const res = pinned ? pinned : static_cast<pseg::SegResult*>(ws);
  const dim3 grid((unsigned)gx, (unsigned)gy, 1);
  cudaError_t e = cudaSuccess;
  if (dtype == RWKVQ_F32) {
    const uint32_t* w32 = static_cast<const uint32_t*>(w);
    // blocks as large as the tile needs; the number of buckets grows with the keys
    if (seg_elems <= 4096) e = pseg::launch_f32<256, 16, 16, 4>(w32, oc, ic, seg_rows, seg_cols, K, res, grid, s);
    else if (seg_elems <= 16384) e = pseg::launch_f32<1024, 16, 14, 1>(w32, oc, ic, seg_rows, seg_cols, K, res, grid, s);
    else e = pseg::launch_f32<1024, 32, 14, 1>(w32, oc, ic, seg_rows, seg_cols, K, res, grid, s);
    if (e != cudaSuccess) return cuda_status(e);
  } else {
    const uint16_t* w16 = static_cast<const uint16_t*>(w);
    const int wide = ic % 8 == 0 && seg_cols % 8 == 0, bf16 = dtype == RWKVQ_BF16;
    // small tiles (a channel of a few thousand weights): the walk over the patterns is most of the work, and more blocks of
    // fewer threads hide its latencies; large ones: the marking is, and wants threads
    if (seg_elems <= 16384) pseg::proxy_segment_set_kernel<256, 4><<<grid, 256, 0, s>>>(w16, oc, ic, seg_rows, seg_cols, wide, bf16, K, res);
    else pseg::proxy_segment_set_kernel<512, 2><<<grid, 512, 0, s>>>(w16, oc, ic, seg_rows, seg_cols, wide, bf16, K, res);
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_status_behind(e, s);
  std::vector<pseg::SegResult> copy;
  const pseg::SegResult* host = pinned;
  if (!pinned) {
    copy.resize(nseg);
    e = cudaMemcpyAsync(copy.data(), res, nseg * sizeof(pseg::SegResult), cudaMemcpyDeviceToHost, s);
    host = copy.data();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_status_behind(e, s);
  rwkvq_status st = RWKVQ_OK;
  for (size_t i = 0; i < nseg; ++i) {
    Pc[i] = host[i].pc; Pf[i] = host[i].pf;
    phi[i] = (host[i].pc < tau_c && host[i].pf < tau_f) ? RWKVQ_SQ : RWKVQ_VQ;   // Eq. 18, strict <
    if (host[i].nonfinite) st = RWKVQ_ENONFINITE;
  }
  return st;
}

size_t rwkvq_proxy_f32_workspace_bytes(int oc, int ic) {
  if (oc <= 0 || ic <= 0) return 0;
  const size_t n = (size_t)oc * (size_t)ic;
  size_t temp = 0;
  if (cub::DeviceRadixSort::SortKeys(nullptr, temp, (const uint32_t*)nullptr, (uint32_t*)nullptr, (long long)n) != cudaSuccess) return 0;
  return round_up_sz(n * 4, 256) * 2 + round_up_sz(temp, 256) + round_up_sz((size_t)pseg::kGapBlocks * pseg::kMaxK * 8, 256) + 512;
}

rwkvq_status rwkvq_proxy_select_f32(const void* w, int oc, int ic, int K, double tau_c, double tau_f, double* Pc, double* Pf,
                                    int* phi, void* ws, size_t ws_bytes, void* stream) {
  if (!w || !Pc || !Pf || !phi || oc <= 0 || ic <= 0) return RWKVQ_EINVAL;
  if (K < 2 || K > pseg::kMaxK) return RWKVQ_EINVAL;
  if (!aligned16(w)) return RWKVQ_EALIGN;
  const size_t need = rwkvq_proxy_f32_workspace_bytes(oc, ic);
  if (need == 0) return RWKVQ_ECUDA;
  if (!ws || ws_bytes < need) return RWKVQ_ENOMEM;
  if ((reinterpret_cast<uintptr_t>(ws) & 255u) != 0) return RWKVQ_EALIGN;
  const size_t n = (size_t)oc * (size_t)ic;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  uint8_t* p = static_cast<uint8_t*>(ws);
  uint32_t* keys = reinterpret_cast<uint32_t*>(p); p += round_up_sz(n * 4, 256);
  uint32_t* sorted = reinterpret_cast<uint32_t*>(p); p += round_up_sz(n * 4, 256);
  size_t temp = 0;
  cub::DeviceRadixSort::SortKeys(nullptr, temp, (const uint32_t*)nullptr, (uint32_t*)nullptr, (long long)n);
  void* temp_ptr = p; p += round_up_sz(temp, 256);
  double* partials = reinterpret_cast<double*>(p); p += round_up_sz((size_t)pseg::kGapBlocks * pseg::kMaxK * 8, 256);
  int* nonfinite = reinterpret_cast<int*>(p);
  pseg::SegResult* res = reinterpret_cast<pseg::SegResult*>(p + 256);
  cudaError_t e = cudaMemsetAsync(nonfinite, 0, 512, s);
  if (e != cudaSuccess) return cuda_status(e);
  pseg::f32_keys_kernel<<<1184, 256, 0, s>>>(static_cast<const uint32_t*>(w), n, keys, nonfinite);
  e = cub::DeviceRadixSort::SortKeys(temp_ptr, temp, keys, sorted, (long long)n, 0, 32, s);
  if (e != cudaSuccess) return cuda_status(e);
  pseg::f32_gap_partials_kernel<<<pseg::kGapBlocks, 256, 0, s>>>(sorted, n, K, partials);
  pseg::f32_gap_final_kernel<<<1, 32, 0, s>>>(sorted, n, K, partials, nonfinite, res);
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_status(e);
  pseg::SegResult host;
  e = cudaMemcpyAsync(&host, res, sizeof(host), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_status(e);
  *Pc = host.pc; *Pf = host.pf;
  *phi = (host.pc < tau_c && host.pf < tau_f) ? RWKVQ_SQ : RWKVQ_VQ;
  return host.nonfinite ? RWKVQ_ENONFINITE : RWKVQ_OK;
}

}  // extern "C"
