// Coarse-to-fine proxy (Section 4.1).  The paper sorts the flattened weights (Eq. 5) and works on
// the gaps between neighbours.  For 16-bit weights the sort reduces to the set of bit patterns that occur
// (proxy_core.cuh): one streaming pass marks them and a second, tiny kernel walks the set in value order:
//   D distinct values v_1 < ... < v_D give D-1 positive gaps; the other n-(D-1) gaps are ties (0).
//   R = v_D - v_1 = sum of gaps;  g'_j = (v_{j+1} - v_j) / R                          (Eq. 6)
//   P_c = ln n + sum_j g'_j ln g'_j            (Eqs. 7-9, 0 ln 0 := 0, n = oc*ic - 1)
//   t_j = n g'_j - 1 (= n delta_j, Eq. 10);  ties have t = -1
//   P_f = sum_{k=2..K} | ( sum_j t_j^k + ties * (-1)^k ) / n | / (k (k-1))            (Eq. 17 with
//         v_k = n^k / (k(k-1)) folded into the moment so nothing overflows)
// The selection rule (Eq. 18) is applied on the host from the two numbers.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "../../include/rwkvq.h"
#include "host_util.h"
#include "proxy_core.cuh"
#include "unpack.cuh"

namespace rwkvq {

constexpr size_t kMatrixBytes = 65536 * 4;   // workspace share of one matrix; its bitmap takes the first 8 KB

struct ProxyResult {
  double pc, pf;
  double variance, cv, range, mad, ie;   // the ablation's statistics of G' (Section 5.3)
  unsigned long long count;
  int distinct, nonfinite;
};

struct MarkArgs {
  static constexpr int kMost = 96;             // matrices per launch
  const uint4* w[kMost];
  unsigned long long n[kMost];                 // weights
  unsigned long long start[kMost + 1];         // first 16-byte vector of each matrix in the launch's common numbering
  int count;
};

// Marks the patterns of all matrices of a call.  A block takes an equal run of the matrices' vectors laid end to end, two
// blocks of 1024 threads per SM, two vectors in flight per thread (64 KB per SM); a run that crosses into the
// next matrix writes its bitmap out and starts a new one.  One launch instead of one per matrix, and 8 KB to clear and merge
// per block instead of 192 KB of counters.
__global__ void __launch_bounds__(1024, 2) proxy_mark_kernel(const __grid_constant__ MarkArgs a, uint8_t* ws) {
  __shared__ __align__(16) uint32_t bm[kPatternWords];
  const unsigned long long total = a.start[a.count];
  unsigned long long at = total * blockIdx.x / gridDim.x;
  const unsigned long long end = total * (blockIdx.x + 1) / gridDim.x;
  int m = 0;
  while (at < end) {
    while (at >= a.start[m + 1]) ++m;
    const unsigned long long stop = min(end, a.start[m + 1]);
    for (int j = threadIdx.x; j < kPatternWords; j += 1024) bm[j] = 0u;
    __syncthreads();
    const uint4* w = a.w[m];
    const unsigned long long full = a.n[m] / 8, hi = min(stop - a.start[m], full);
    unsigned long long i = at - a.start[m] + threadIdx.x;
    for (; i + 1024 < hi; i += 2048) {
      const uint4 v = ldg_stream(w + i), u = ldg_stream(w + i + 1024);
      mark_pair(bm, v.x); mark_pair(bm, v.y); mark_pair(bm, v.z); mark_pair(bm, v.w);
      mark_pair(bm, u.x); mark_pair(bm, u.y); mark_pair(bm, u.z); mark_pair(bm, u.w);
    }
    if (i < hi) {
      const uint4 v = ldg_stream(w + i);
      mark_pair(bm, v.x); mark_pair(bm, v.y); mark_pair(bm, v.z); mark_pair(bm, v.w);
    }
    if (stop == a.start[m + 1] && threadIdx.x < a.n[m] % 8)      // the weights behind the last whole vector
      mark_pattern(bm, reinterpret_cast<const unsigned short*>(w + full)[threadIdx.x]);
    __syncthreads();
    uint32_t* all = reinterpret_cast<uint32_t*>(ws + (size_t)m * kMatrixBytes);
    for (int j = threadIdx.x; j < kPatternWords; j += 1024) {
      const uint32_t v = bm[j];
      if (v && (v & ~__ldcg(all + j))) atomicOr(all + j, v);
    }
    __syncthreads();
    at = stop;
  }
}

// One block per matrix.
__global__ void __launch_bounds__(1024, 1) proxy_reduce_kernel(const uint8_t* ws, const __grid_constant__ MarkArgs a, ProxyResult* res_all, int K, int bf16) {
  __shared__ __align__(16) uint32_t bm[kPatternWords];
  __shared__ SetShared<1024> sh;
  const uint2* all = reinterpret_cast<const uint2*>(ws + (size_t)blockIdx.x * kMatrixBytes);
  fill_log_table(sh.logs);
  reinterpret_cast<uint2*>(bm)[threadIdx.x] = __ldcg(all + threadIdx.x);
  __syncthreads();
  const double n = (double)(a.n[blockIdx.x] - 1ull);
  SetStats s;
  set_gaps<1024>(bm, bf16 != 0, n, K, sh, s);
  if (threadIdx.x != 0) return;
  ProxyResult r;
  r.count = a.n[blockIdx.x]; r.distinct = s.distinct; r.nonfinite = s.nonfinite ? 1 : 0;
  r.pc = r.pf = r.variance = r.cv = r.range = r.mad = r.ie = INFINITY;
  if (!s.nonfinite && !s.degenerate) {
    const double ties = n - (double)(s.distinct - 1);
    // with t = n G' - 1 (ties: t = -1):  variance = sum t^2 / n^3,  mad = sum |t| / n^2
    r.variance = (s.pw[0] + ties) / (n * n * n);
    r.cv = sqrt(r.variance) * n;
    r.range = s.gmax - (ties > 0.0 ? 0.0 : s.gmin);
    r.mad = (s.abs_t + ties) / (n * n);
    r.ie = -s.sum_glng;
    proxy_from_set(s, n, K, &r.pc, &r.pf);
  }
  res_all[blockIdx.x] = r;
}

}  // namespace rwkvq

using namespace rwkvq;

extern "C" {

size_t rwkvq_proxy_workspace_bytes(int n_mats) {
  if (n_mats <= 0) return 0;
  return (size_t)n_mats * kMatrixBytes + round_up_sz((size_t)n_mats * sizeof(ProxyResult), 256);
}

static rwkvq_status run_proxy(const void* const* w, const int* oc, const int* ic, int n_mats, int K, void* ws,
                              size_t ws_bytes, void* stream, std::vector<ProxyResult>* out, int bf16 = 0) {
  if (!w || !oc || !ic || n_mats <= 0) return RWKVQ_EINVAL;
  if (K < 2 || K > 8) return RWKVQ_EINVAL;
  if (!ws || ws_bytes < rwkvq_proxy_workspace_bytes(n_mats)) return RWKVQ_ENOMEM;
  if (!aligned16(ws)) return RWKVQ_EALIGN;
  for (int m = 0; m < n_mats; ++m) {
    if (!w[m] || oc[m] <= 0 || ic[m] <= 0) return RWKVQ_EINVAL;
    if (!aligned16(w[m])) return RWKVQ_EALIGN;
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  uint8_t* base = static_cast<uint8_t*>(ws);
  ProxyResult* const pinned = static_cast<ProxyResult*>(pinned_results((size_t)n_mats * sizeof(ProxyResult)));
  ProxyResult* const res = pinned ? pinned : reinterpret_cast<ProxyResult*>(base + (size_t)n_mats * kMatrixBytes);
  cudaError_t e = cudaMemset2DAsync(base, kMatrixBytes, 0, kPatternWords * 4, n_mats, s);
  if (e != cudaSuccess) return cuda_status(e);
  const int sms = sm_count();
  for (int m0 = 0; m0 < n_mats; m0 += MarkArgs::kMost) {
    MarkArgs a;
    a.count = std::min(n_mats - m0, MarkArgs::kMost);
    a.start[0] = 0;
    for (int i = 0; i < a.count; ++i) {
      a.w[i] = static_cast<const uint4*>(w[m0 + i]);
      a.n[i] = (unsigned long long)oc[m0 + i] * (unsigned long long)ic[m0 + i];
      a.start[i + 1] = a.start[i] + (a.n[i] + 7) / 8;
    }
    // two blocks per SM, and no more than one per 1024 vectors: a block's clearing and merging should not outweigh its share
    const unsigned long long blocks = std::min<unsigned long long>(2ull * (unsigned)sms, (a.start[a.count] + 1023) / 1024);
    uint8_t* part = base + (size_t)m0 * kMatrixBytes;
    proxy_mark_kernel<<<(unsigned)blocks, 1024, 0, s>>>(a, part);
    proxy_reduce_kernel<<<a.count, 1024, 0, s>>>(part, a, res + m0, K, bf16);
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_status_behind(e, s);
  out->resize(n_mats);
  if (!pinned) e = cudaMemcpyAsync(out->data(), res, (size_t)n_mats * sizeof(ProxyResult), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_status_behind(e, s);
  if (pinned) std::copy(pinned, pinned + n_mats, out->begin());
  for (int m = 0; m < n_mats; ++m)
    if ((*out)[m].nonfinite) return RWKVQ_ENONFINITE;
  return RWKVQ_OK;
}

rwkvq_status rwkvq_proxy_select(const void* const* w, const int* oc, const int* ic, int n_mats, int K,
                                double tau_c, double tau_f, double* Pc, double* Pf, int* phi, void* ws,
                                size_t ws_bytes, void* stream) {
  if (!Pc || !Pf || !phi) return RWKVQ_EINVAL;
  std::vector<ProxyResult> host;
  const rwkvq_status st = run_proxy(w, oc, ic, n_mats, K, ws, ws_bytes, stream, &host);
  if (st != RWKVQ_OK && st != RWKVQ_ENONFINITE) return st;
  for (int m = 0; m < n_mats; ++m) {
    Pc[m] = host[m].pc; Pf[m] = host[m].pf;
    phi[m] = (host[m].pc < tau_c && host[m].pf < tau_f) ? RWKVQ_SQ : RWKVQ_VQ;   // Eq. 18, strict <
  }
  return st;
}

rwkvq_status rwkvq_proxy_select_bf16(const void* const* w, const int* oc, const int* ic, int n_mats, int K,
                                     double tau_c, double tau_f, double* Pc, double* Pf, int* phi, void* ws,
                                     size_t ws_bytes, void* stream) {
  if (!Pc || !Pf || !phi) return RWKVQ_EINVAL;
  std::vector<ProxyResult> host;
  const rwkvq_status st = run_proxy(w, oc, ic, n_mats, K, ws, ws_bytes, stream, &host, 1);
  if (st != RWKVQ_OK && st != RWKVQ_ENONFINITE) return st;
  for (int m = 0; m < n_mats; ++m) {
    Pc[m] = host[m].pc; Pf[m] = host[m].pf;
    phi[m] = (host[m].pc < tau_c && host[m].pf < tau_f) ? RWKVQ_SQ : RWKVQ_VQ;   // Eq. 18, strict <
  }
  return st;
}

rwkvq_status rwkvq_proxy_family(const void* const* w, const int* oc, const int* ic, int n_mats, double* stats,
                                void* ws, size_t ws_bytes, void* stream) {
  if (!stats) return RWKVQ_EINVAL;
  std::vector<ProxyResult> host;
  const rwkvq_status st = run_proxy(w, oc, ic, n_mats, 2, ws, ws_bytes, stream, &host);
  if (st != RWKVQ_OK && st != RWKVQ_ENONFINITE) return st;
  for (int m = 0; m < n_mats; ++m) {
    double* o = stats + (size_t)m * 5;
    o[0] = host[m].variance; o[1] = host[m].cv; o[2] = host[m].range; o[3] = host[m].mad; o[4] = host[m].ie;
  }
  return st;
}

rwkvq_status rwkvq_tau_for_fraction(const double* values, int n, double sq_fraction, double* tau_out) {
  if (!values || !tau_out || n <= 0 || !(sq_fraction >= 0.0) || !(sq_fraction <= 1.0)) return RWKVQ_EINVAL;
  std::vector<double> v(values, values + n);
  for (double x : v) if (x != x) return RWKVQ_EINVAL;
  std::sort(v.begin(), v.end());
  const long k = lrint(sq_fraction * (double)n);
  if (k <= 0) *tau_out = -INFINITY;
  else if (k >= n) *tau_out = INFINITY;
  else *tau_out = 0.5 * (v[k - 1] + v[k]);
  return RWKVQ_OK;
}

rwkvq_status rwkvq_tau_largest_gap(const double* values, int n, double* tau_out) {
  if (!values || !tau_out || n <= 0) return RWKVQ_EINVAL;
  std::vector<double> v;
  v.reserve((size_t)n);
  for (int i = 0; i < n; ++i) {
    if (values[i] != values[i]) return RWKVQ_EINVAL;
    if (std::isfinite(values[i])) v.push_back(values[i]);
  }
  std::sort(v.begin(), v.end());
  *tau_out = INFINITY;
  if (v.size() < 2 || v.back() == v.front()) return RWKVQ_OK;
  size_t best = 0;
  double widest = -1.0;
  for (size_t i = 0; i + 1 < v.size(); ++i) {
    const double gap = v[i + 1] - v[i];
    if (gap > widest) { widest = gap; best = i; }     // the first of equally wide gaps
  }
  *tau_out = 0.5 * (v[best] + v[best + 1]);
  return RWKVQ_OK;
}

}  // extern "C"
