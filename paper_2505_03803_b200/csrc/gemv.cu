// Decode products (Appendix A.1: the W.(...) products of time- and channel-mixing) over the two
// packed formats, with the token-shift mix fused into the input stage, and the dequantisation
// probe.  One launch per product; the whole-step persistent launch lives in step.cu and reuses
// the per-record routines below.
#include <cuda_runtime.h>

#include <algorithm>

#include "../../include/rwkvq.h"
#include "gemv_core.cuh"
#include "host_util.h"

namespace rwkvq {

// ---------------------------------------------------------------------------------------------
// Single-product kernel.  CTA = 8 warps; block (rb, ks) covers RPC rows (128 for SQ, 256 for
// VQ) and the column tiles [ks*nkt, min(KT, (ks+1)*nkt)).  Warp w owns record w of each chunk.
//
// A product of a few MB is a chain of latencies: launch, inputs and weights (one trip to memory: the first records are requested before
// the inputs are mixed), the tensor-core steps, and the sum over the K splits.  Up to eight splits form a cluster and add
// up in distributed shared memory; more go through global memory and a last-arriver reduction.  The launch is
// a programmatic dependent one: its start overlaps the end of the kernel in front, which it waits for before it touches memory.
// 512 x 512, one token, calls back to back: 10.5 -> 4.6 us a call (now the host enqueueing them).
// ---------------------------------------------------------------------------------------------
template <int FMT, int NB>
__global__ void __launch_bounds__(256, 2) gemv_kernel(const __grid_constant__ GemvArgs a) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int rb = blockIdx.x, ks = blockIdx.y;
  const int kt0 = ks * a.nkt, kt1 = min(a.KT, kt0 + a.nkt);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int REC = (FMT == FMT_SQ3) ? 1 : 2;
  constexpr int RPC = 128 * REC;
  constexpr int BITS = (FMT == FMT_VQ8) ? 8 : 6;
  constexpr int RBYTES = FMT == FMT_SQ3 ? RWKVQ_SQ_RECORD_BYTES : 64 * 32 * BITS / 8;

  const SmemLayout L = smem_layout<FMT>(a.nkt, a.B, a.mu ? a.mu_entries : 0, a.entries);
  const uint8_t* rec = a.payload + ((size_t)(REC * rb) * a.KT * 8 + warp) * RBYTES;      // record of tile 0; tiles 8 * RBYTES apart
  asm volatile("griddepcontrol.launch_dependents;");
  asm volatile("griddepcontrol.wait;" ::: "memory");

  float acc[REC][NB][4];
#pragma unroll
  for (int r = 0; r < REC; ++r)
#pragma unroll
    for (int n = 0; n < NB; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[r][n][i] = 0.f;

  if constexpr (FMT == FMT_SQ3) {
    SqRecord cur, nxt;
    cur.load(rec + (size_t)kt0 * 8 * RBYTES, lane);
    if (kt0 + 1 < kt1) nxt.load(rec + (size_t)(kt0 + 1) * 8 * RBYTES, lane);
    stage_input<FMT>(smem, L, a, kt0, kt1);
    for (int kt = kt0; kt < kt1; ++kt) {
      uint32_t w[12];
      cur.words(w);
      const uint4 sz = cur.sz;
      cur = nxt;
      if (kt + 2 < kt1) nxt.load(rec + (size_t)(kt + 2) * 8 * RBYTES, lane);
      const XLane xl = make_xlane(smem + (size_t)(kt - kt0) * 512, L.xstride,
                                  reinterpret_cast<const float*>(smem + L.gs_off) + (size_t)(kt - kt0) * 2 * 3 * 16, 16, a.B, lane);
      sq_record_mma<NB>(w, sz, xl, acc[0]);
    }
  } else {
    const int E = a.entries;
    const uint32_t* cbg = reinterpret_cast<const uint32_t*>(a.aux) + (size_t)(rb * a.KT) * E;
    // registers suffice to request the first tile's records ahead of the inputs, and those of the others a tile ahead
    constexpr bool kEarly = !(BITS == 8 && NB == 2), kAhead = NB == 1;
    VqRecord<BITS> v[REC];
#pragma unroll
    for (int r = 0; r < REC; ++r)
      if (kEarly) v[r].load(rec + ((size_t)r * a.KT + kt0) * 8 * RBYTES, lane);
    stage_codebook(smem + L.cb_off, cbg + (size_t)kt0 * E, E);
    stage_input<FMT>(smem, L, a, kt0, kt1);      // ends with a barrier
    // A tile's sum starts at zero and is added with a rounding of its own: the tensor core's accumulation cuts off, and its error grows with
    // the chain (4096 x 4096, two tiles a block: 6.9e-7 of the result in one chain, 3.5e-7 like this).
    float before[REC][NB][4] = {};
    auto bank = [&]() {
#pragma unroll
      for (int r = 0; r < REC; ++r)
#pragma unroll
        for (int n = 0; n < NB; ++n)
#pragma unroll
          for (int i = 0; i < 4; ++i) { before[r][n][i] += acc[r][n][i]; acc[r][n][i] = 0.f; }
    };
    for (int kt = kt0; kt < kt1; ++kt) {
      if (kt > kt0) { bank(); __syncthreads(); }
      if (kt + 1 < kt1)
        stage_codebook(smem + L.cb_off + (size_t)((kt + 1 - kt0) & 1) * E * 128, cbg + (size_t)(kt + 1) * E, E);
      const uint32_t* cb_lane = reinterpret_cast<const uint32_t*>(smem + L.cb_off + (size_t)((kt - kt0) & 1) * E * 128) + lane;
      const XLane xl = make_xlane(smem + (size_t)(kt - kt0) * 512, L.xstride, nullptr, 16, a.B, lane);
#pragma unroll
      for (int r = 0; r < REC; ++r) {
        if (!kAhead && !(kEarly && kt == kt0)) v[r].load(rec + ((size_t)r * a.KT + kt) * 8 * RBYTES, lane);
        vq_record_mma<BITS, NB>(v[r].w, cb_lane, xl, acc[r]);
        if (kAhead && kt + 1 < kt1) v[r].load(rec + ((size_t)r * a.KT + kt + 1) * 8 * RBYTES, lane);
      }
    }
    if (kt1 - kt0 > 1) {
#pragma unroll
      for (int r = 0; r < REC; ++r)
#pragma unroll
        for (int n = 0; n < NB; ++n)
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[r][n][i] += before[r][n][i];
    }
  }

  // ---- epilogue: direct store, or partial sums + a reduction over the K splits
  const int g = lane >> 2, t = lane & 3;
  if (a.S == 1) {
#pragma unroll
    for (int r = 0; r < REC; ++r)
#pragma unroll
      for (int n = 0; n < NB; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          int row = rb * RPC + r * 128 + warp * 16 + g + 8 * (i >> 1);
          int b = n * 8 + 2 * t + (i & 1);
          if (b < a.B && row < a.oc) store_y(a.y, a.y_dtype, (size_t)b * a.oc + row, acc[r][n][i]);
        }
    return;
  }
  float* part = a.cluster ? reinterpret_cast<float*>(smem) : a.partial + ((size_t)(ks * gridDim.x + rb) * 16) * RPC;
  if (a.cluster) __syncthreads();      // the staged inputs are not read any more
#pragma unroll
  for (int r = 0; r < REC; ++r)
#pragma unroll
    for (int n = 0; n < NB; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        int rl = r * 128 + warp * 16 + g + 8 * (i >> 1);
        int b = n * 8 + 2 * t + (i & 1);
        if (b < a.B) part[(size_t)b * RPC + rl] = acc[r][n][i];
      }
  if (a.cluster) {
    // every block of the cluster sums a share of the outputs over all S splits, in the same order
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
    const uint32_t mine = (uint32_t)__cvta_generic_to_shared(smem);
    for (int idx = ks * (int)blockDim.x + threadIdx.x; idx < a.B * RPC; idx += a.S * (int)blockDim.x) {
      float sum = 0.f;
      for (int s = 0; s < a.S; ++s) {
        uint32_t addr;
        float v;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(mine + 4u * (uint32_t)idx), "r"(s));
        asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
        sum += v;
      }
      const int b = idx / RPC, row = rb * RPC + idx % RPC;
      if (row < a.oc) store_y(a.y, a.y_dtype, (size_t)b * a.oc + row, sum);
    }
    // no block leaves while others may read its partial sums
    asm volatile("barrier.cluster.arrive.relaxed.aligned;\n barrier.cluster.wait.aligned;" ::: "memory");
    return;
  }
  __threadfence();
  __syncthreads();
  __shared__ unsigned s_last;
  if (threadIdx.x == 0) s_last = (atomicAdd(&a.counters[rb], 1u) == (unsigned)(a.S - 1));
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  for (int idx = threadIdx.x; idx < a.B * RPC; idx += blockDim.x) {
    int b = idx / RPC, rl = idx % RPC;
    float sum = 0.f;
    for (int s = 0; s < a.S; ++s)  // fixed order: the result does not depend on arrival order
      sum += __ldcg(a.partial + ((size_t)(s * gridDim.x + rb) * 16 + b) * RPC + rl);
    int row = rb * RPC + rl;
    if (row < a.oc) store_y(a.y, a.y_dtype, (size_t)b * a.oc + row, sum);
  }
  if (threadIdx.x == 0) a.counters[rb] = 0u;  // leave the workspace zero-filled for the next call
}

// ---------------------------------------------------------------------------------------------
// Dequantisation probe: one warp per record, same unpack routines as the products.
// ---------------------------------------------------------------------------------------------
// With `ref` (the fp16 matrix the image was made from) nothing is stored: each warp instead adds up
// (w - w_hat)^2 over its record in fp64 and writes the sum to sse_partial[record].
template <int FMT>
__global__ void dequant_kernel(const uint8_t* payload, const uint8_t* aux, int oc, int ic, int KT,
                               int entries, void* out, int dtype, int n_records, const __half* ref = nullptr,
                               double* sse_partial = nullptr) {
  const int lane = threadIdx.x & 31;
  const int recid = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (recid >= n_records) return;
  const int rt = recid & 7, chunk = recid >> 3;
  const int mb = chunk / KT, kt = chunk % KT;
  const int g = lane >> 2, t = lane & 3;
  const int r0 = mb * 128 + rt * 16, c0 = kt * 256;
  double sse = 0.0;
  if constexpr (FMT == FMT_SQ3) {
    SqRecord rec;
    rec.load(payload + (size_t)recid * RWKVQ_SQ_RECORD_BYTES, lane);
    uint32_t w[12];
    rec.words(w);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      uint32_t r[16];
      sq_unpack_triple(w[3 * i], w[3 * i + 1], w[3 * i + 2], r);
#pragma unroll
      for (int e = 0; e < 16; ++e) {
        const int m = e >> 2, R = e & 3;
        const int row = r0 + g + 8 * (R & 1);
        const int col = c0 + 64 * i + 16 * m + 4 * t + 2 * (R >> 1);
        const uint32_t szw = rec.sz_word((R & 1) * 2 + (i >> 1));
        const float s = __half2float(__ushort_as_half((unsigned short)(szw & 0xFFFF)));
        const float z = __half2float(__ushort_as_half((unsigned short)(szw >> 16)));
        const __half2 biased = *reinterpret_cast<const __half2*>(&r[e]);
        const float bias = (float)(1024 >> rwkvq_sq_pos(e));
        const float q0 = __half2float(__low2half(biased)) - bias;   // exact: integers below 2048
        const float q1 = __half2float(__high2half(biased)) - bias;
        const float v0 = __fmul_rn(s, __fsub_rn(q0, z));
        const float v1 = __fmul_rn(s, __fsub_rn(q1, z));
        if (row < oc && col < ic) {
          if (ref) {
            const float2 wv = __half22float2(*reinterpret_cast<const __half2*>(ref + (size_t)row * ic + col));
            const double d0 = (double)wv.x - (double)v0, d1 = (double)wv.y - (double)v1;
            sse += d0 * d0 + d1 * d1;
          } else {
            store_w(out, dtype, (size_t)row * ic + col, v0);
            store_w(out, dtype, (size_t)row * ic + col + 1, v1);
          }
        }
      }
    }
  } else {
    constexpr int BITS = (FMT == FMT_VQ6) ? 6 : 8;
    VqRecord<BITS> rec;
    rec.load(payload + (size_t)recid * (64 * 32 * BITS / 8), lane);
    const uint32_t* cb = reinterpret_cast<const uint32_t*>(aux) + (size_t)((mb >> 1) * KT + kt) * entries;
#pragma unroll
    for (int n = 0; n < 64; ++n) {
      const int j = n >> 2, R = n & 3;
      const int row = r0 + g + 8 * (R & 1);
      const int col = c0 + 16 * j + 4 * t + 2 * (R >> 1);
      const uint32_t v = cb[vq_index<BITS, VqRecord<BITS>::NW>(rec.w, n)];
      const __half2 h = *reinterpret_cast<const __half2*>(&v);
      if (ref) {
        const float2 wv = __half22float2(*reinterpret_cast<const __half2*>(ref + (size_t)row * ic + col));
        const double d0 = (double)wv.x - (double)__half2float(__low2half(h)), d1 = (double)wv.y - (double)__half2float(__high2half(h));
        sse += d0 * d0 + d1 * d1;
      } else {
        store_w(out, dtype, (size_t)row * ic + col, __half2float(__low2half(h)));
        store_w(out, dtype, (size_t)row * ic + col + 1, __half2float(__high2half(h)));
      }
    }
  }
  if (ref) {
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) sse += __shfl_xor_sync(0xFFFFFFFFu, sse, off);
    if (lane == 0) sse_partial[recid] = sse;
  }
}

// Sum of n doubles in a fixed order (one block): the result does not depend on scheduling.
__global__ void __launch_bounds__(1024) sum_fixed_kernel(const double* v, int n, double* out) {
  __shared__ double s_red[1024];
  double acc = 0.0;
  for (int i = threadIdx.x; i < n; i += 1024) acc += v[i];
  s_red[threadIdx.x] = acc;
  __syncthreads();
  for (int s = 512; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) s_red[threadIdx.x] += s_red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = s_red[0];
}

__global__ void dequant_vector_kernel(const uint8_t* payload, const uint8_t* aux, int ic, int bits,
                                      void* out, int dtype) {
  int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= ic / 2) return;
  uint32_t v = reinterpret_cast<const uint32_t*>(aux)[vector_index(payload, p, bits)];
  const __half2 h = *reinterpret_cast<const __half2*>(&v);
  store_w(out, dtype, 2 * (size_t)p, __half2float(__low2half(h)));
  store_w(out, dtype, 2 * (size_t)p + 1, __half2float(__high2half(h)));
}

// ---------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------
static int fmt_of(const rwkvq_desc* d) {
  if (d->method == RWKVQ_SQ) return FMT_SQ3;
  return d->bits == 6 ? FMT_VQ6 : FMT_VQ8;
}

struct GemvPlan {
  int fmt, NRB, KT, S, nkt;
  bool cluster, dependent;
  size_t smem, ws_bytes, counters_bytes;
};


static rwkvq_status plan_gemv(const rwkvq_desc* d, int B, bool has_mu, int mu_entries, GemvPlan* p) {
  if (!d || B < 1 || B > 16) return RWKVQ_EINVAL;
  if (d->oc == 1) return RWKVQ_ESHAPE;
  rwkvq_status st = check_matrix_desc(d);
  if (st != RWKVQ_OK) return st;
  p->fmt = fmt_of(d);
  const int rpc = p->fmt == FMT_SQ3 ? 128 : 256;
  p->NRB = d->oc_pad / rpc;
  p->KT = d->ic_pad / 256;
  const int entries = has_mu ? mu_entries : 0;
  auto smem_of = [&](int nkt) {
    return p->fmt == FMT_SQ3 ? smem_layout<FMT_SQ3>(nkt, B, entries, d->entries).total
         : p->fmt == FMT_VQ6 ? smem_layout<FMT_VQ6>(nkt, B, entries, d->entries).total
                             : smem_layout<FMT_VQ8>(nkt, B, entries, d->entries).total;
  };
  // Enough blocks for two per SM, bounded by the shared-memory footprint of the staged input.
  int want = (2 * 148 + p->NRB - 1) / p->NRB;
  int S = want < 1 ? 1 : (want > p->KT ? p->KT : want);
  while (S < p->KT && smem_of((p->KT + S - 1) / S) > 96 * 1024) ++S;
  // A contraction of a few tiles is done by one block: a tile costs it less than the sum over splits does.  Where eight splits
  // leave no block with many more tiles than that, the splits are a cluster (measured from 512 x 512 to 14336 x 4096).  A VQ tile is dearer, it
  // brings its codebook, and a sum through global memory is cheap for a few rows: tiles that a block takes more than without the cluster have to be
  // paid for by the batch (us through global memory / cluster, one tile more: 64 entries, 512 x 4096: B=1 6.4 / 7.6, B=4 8.9 / 7.8;
  // 4096 x 4096: B=4 9.8 / 10.2, B=6 11.2 / 10.8; 256 entries, 512 x 4096: B=8 15.5 / 17.0, B=12 18.8 / 18.5; 4096 x 4096: B=12 20.4 / 21.5, B=16
  // 23.4 / 22.1; two tiles more, 64 entries, 512 x 6144: B=1 7.2 / 10.5, B=8 14.6 / 11.5).
  const bool sq = p->fmt == FMT_SQ3, vq6 = p->fmt == FMT_VQ6;
  const int kTilesPerSum = sq ? 2 : 1, kClusterTiles = sq ? 4 : vq6 ? 3 : 2;
  const int kRowsPerTile = sq ? 0 : vq6 ? (p->NRB > 8 ? 6 : 4) : (p->NRB > 8 ? 16 : 12);
  const int per_cluster = (p->KT + 7) / 8, more = per_cluster - (p->KT + S - 1) / S;
  p->cluster = false;
  if (p->KT <= kTilesPerSum) {
    S = 1;
  } else if (S <= 8 || (per_cluster <= kClusterTiles && B >= more * kRowsPerTile && smem_of(per_cluster) <= 96 * 1024)) {
    S = S < 8 ? S : 8;
    p->cluster = true;
  }
  auto blocks_of = [&](int s) { const int nkt = (p->KT + s - 1) / s; return p->NRB * ((p->KT + nkt - 1) / nkt); };      // no empty splits
  // More blocks than surely fit at once (two per SM, whole clusters within a GPC): clusters would wait for room
  // together (14336 x 4096 VQ 28.7 us, through global memory 23.3; 9456 x 9600 SQ 22.0 and 18.4).
  if (blocks_of(S) == p->NRB || blocks_of(S) > 256) p->cluster = false;
  // A few blocks more than fit at once cost a second round.  64-entry products of up to eight rows, whose blocks take half an SM's registers each, avoid
  // it where that saves a tenth (beyond four rows, an eighth) by this estimate (in tiles; a block costs one besides its own; a round that leaves SMs
  // with a single block takes 0.55 of the time): 10240 x 10240, one row: 320 blocks of five tiles 37.1 us, 280 of six 29.0; 9216 x 9216: 29.0 and 22.8; 23040 x 3840: 26.8
  // and 22.8; 4096 x 14336: 20.5 and 19.1, eight rows 29.4 and 30.5; not 8192 x 14336 (30.3 and 31.8), whose second round is a short last split,
  // nor 14336 x 4096 (17.7 and 18.1).
  constexpr int kFit = 2 * 148;
  if (vq6 && B <= 8 && !p->cluster && blocks_of(S) > kFit) {
    auto estimate = [&](int s) {
      const int nkt = (p->KT + s - 1) / s, n = blocks_of(s) / p->NRB, last = p->KT - (n - 1) * nkt;
      double sum = 0.0;
      for (int left = n * p->NRB; left > 0; left -= kFit)       // blocks are dealt split by split
        sum += ((left <= p->NRB ? last : nkt) + 1) * (left <= kFit / 2 && n * p->NRB > kFit ? 0.55 : 1.0);
      return sum;
    };
    int best = S;
    for (int s = 1; s <= p->KT; ++s)
      if (estimate(s) < estimate(best) && smem_of((p->KT + s - 1) / s) <= 96 * 1024) best = s;
    if (estimate(best) <= (B <= 4 ? 0.9 : 0.88) * estimate(S)) S = best;
  }
  p->nkt = (p->KT + S - 1) / S;
  p->S = (p->KT + p->nkt - 1) / p->nkt;
  // A launch that starts early finds the SMs occupied by the product in front: up to a block per SM then double up on some (2048 x 4096, 64 entries, 128
  // blocks: 7.4 us a call, plainly launched 6.8; 64 blocks 6.8 and 6.7, 32 6.4 and 6.6, 195 8.3 and 8.7, 256 7.6 and 8.2).
  p->dependent = sq || p->cluster || p->NRB * p->S <= 74 || p->NRB * p->S > 148;
  p->smem = smem_of(p->nkt);
  if (p->cluster) p->smem = std::max(p->smem, (size_t)B * rpc * 4);
  p->counters_bytes = ((size_t)p->NRB * 4 + 255) / 256 * 256;
  p->ws_bytes = p->counters_bytes + (p->S > 1 && !p->cluster ? (size_t)p->S * p->NRB * 16 * rpc * 4 : 0);
  return RWKVQ_OK;
}

template <int FMT, int NB>
static cudaError_t launch_gemv_as(const GemvArgs& a, const GemvPlan& p, cudaStream_t s) {
  static SmemOptIn opt_in;
  if (p.smem > 48 * 1024) {
    const cudaError_t e = opt_in((const void*)gemv_kernel<FMT, NB>, 112 * 1024);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.NRB, p.S); cfg.blockDim = dim3(256); cfg.dynamicSmemBytes = p.smem; cfg.stream = s;
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (p.dependent) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (p.cluster) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = 1; attr[n].val.clusterDim.y = p.S; attr[n++].val.clusterDim.z = 1;
  }
  cfg.attrs = attr; cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, gemv_kernel<FMT, NB>, a);
}
template <int FMT>
static cudaError_t launch_gemv(const GemvArgs& a, const GemvPlan& p, cudaStream_t s) {
  return a.B <= 8 ? launch_gemv_as<FMT, 1>(a, p, s) : launch_gemv_as<FMT, 2>(a, p, s);
}

}  // namespace rwkvq

using namespace rwkvq;

extern "C" {

size_t rwkvq_gemv_workspace_bytes(const rwkvq_desc* d, int B) {
  // the call may come without a token shift or with one of either codebook, whose shared memory moves the splits
  size_t most = 0;
  for (const int mu_entries : {0, 64, 256}) {
    GemvPlan p;
    if (plan_gemv(d, B, mu_entries != 0, mu_entries, &p) != RWKVQ_OK) return 0;
    most = std::max(most, p.ws_bytes);
  }
  return most;
}

// Every argument check of the decode product, made on the host before anything is enqueued.
static rwkvq_status check_gemv_args(const rwkvq_desc* d, const void* W, const rwkvq_desc* mud, const void* mu, const void* x,
                                    const void* xprev, int B, const void* y, int y_dtype, GemvPlan* p) {
  if (!d || !W || !x || !y) return RWKVQ_EINVAL;
  if ((mu == nullptr) != (xprev == nullptr)) return RWKVQ_EINVAL;
  if (mu && !mud) return RWKVQ_EINVAL;
  if (y_dtype != RWKVQ_F32 && y_dtype != RWKVQ_F16) return RWKVQ_EINVAL;
  if (mu) {
    rwkvq_status st = check_vector_desc(mud, d->ic);
    if (st != RWKVQ_OK) return st;
  }
  rwkvq_status st = plan_gemv(d, B, mu != nullptr, mu ? mud->entries : 0, p);
  if (st != RWKVQ_OK) return st;
  if (!aligned16(W) || !aligned16(x) || !aligned16(y) || (mu && (!aligned16(mu) || !aligned16(xprev)))) return RWKVQ_EALIGN;
  return RWKVQ_OK;
}

static rwkvq_status run_gemv(const GemvPlan& p, const rwkvq_desc* d, const void* W, const rwkvq_desc* mud, const void* mu,
                             const void* x, const void* xprev, int B, void* y, int y_dtype, void* ws, void* stream) {
  GemvArgs a;
  fill_gemv_args(&a, d, W, mud, mu, x, xprev, B, y, y_dtype);
  a.KT = p.KT; a.S = p.S; a.nkt = p.nkt; a.cluster = p.cluster ? 1 : 0;
  a.counters = static_cast<unsigned*>(ws);
  a.partial = reinterpret_cast<float*>(static_cast<uint8_t*>(ws) + p.counters_bytes);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaError_t e = p.fmt == FMT_SQ3 ? launch_gemv<FMT_SQ3>(a, p, s)
                : p.fmt == FMT_VQ6 ? launch_gemv<FMT_VQ6>(a, p, s)
                                   : launch_gemv<FMT_VQ8>(a, p, s);
  return cuda_status(e);
}

rwkvq_status rwkvq_gemv(const rwkvq_desc* d, const void* W, const rwkvq_desc* mud, const void* mu,
                        const void* x, const void* xprev, int B, void* y, int y_dtype, void* ws,
                        size_t ws_bytes, void* stream) {
  GemvPlan p;
  rwkvq_status st = check_gemv_args(d, W, mud, mu, x, xprev, B, y, y_dtype, &p);
  if (st != RWKVQ_OK) return st;
  if (ws && !aligned16(ws)) return RWKVQ_EALIGN;
  if (!ws || ws_bytes < p.ws_bytes) return RWKVQ_ENOMEM;
  return run_gemv(p, d, W, mud, mu, x, xprev, B, y, y_dtype, ws, stream);
}

// ---------------------------------------------------------------------------------------------
// rwkvq_gemv for callers that cannot allocate device memory: the split-K scratch lives in a
// file-scope device array.  In host code the array's name is only a handle; its device address
// is looked up once per device and context (with that device current).
// ---------------------------------------------------------------------------------------------
#define RWKVQ_STATIC_SCRATCH_BYTES (8u << 20)
static __device__ __align__(256) unsigned char g_static_scratch[RWKVQ_STATIC_SCRATCH_BYTES];
static SymbolAddress g_static_scratch_address;

size_t rwkvq_gemv_static_max_scratch_bytes(void) { return RWKVQ_STATIC_SCRATCH_BYTES; }

rwkvq_status rwkvq_gemv_static(const rwkvq_desc* d, const void* W, const rwkvq_desc* mud, const void* mu,
                               const void* x, const void* xprev, int B, void* y, int y_dtype, void* stream) {
  // every argument error is reported before anything reaches the stream
  GemvPlan p;
  rwkvq_status st = check_gemv_args(d, W, mud, mu, x, xprev, B, y, y_dtype, &p);
  if (st != RWKVQ_OK) return st;
  if (p.ws_bytes > RWKVQ_STATIC_SCRATCH_BYTES) return RWKVQ_ENOMEM;   // this product needs more scratch than the built-in array holds
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_status(e);
  if (dev < 0 || dev >= kMaxDevices) return RWKVQ_EUNSUPPORTED;
  void* ws = nullptr;
  e = g_static_scratch_address((const void*)g_static_scratch, &ws);
  if (e != cudaSuccess) return cuda_status(e);
  // The array keeps whatever the previous call left: the arrival counters must start at zero.
  if (p.S > 1 && !p.cluster) {
    e = cudaMemsetAsync(ws, 0, p.counters_bytes, static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return cuda_status(e);
  }
  return run_gemv(p, d, W, mud, mu, x, xprev, B, y, y_dtype, ws, stream);
}

rwkvq_status rwkvq_dequant(const rwkvq_desc* d, const void* W, void* out, int dtype, void* stream) {
  if (!d || !W || !out) return RWKVQ_EINVAL;
  if (dtype != RWKVQ_F32 && dtype != RWKVQ_BF16) return RWKVQ_EINVAL;
  if (!aligned16(W) || !aligned16(out)) return RWKVQ_EALIGN;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const uint8_t* img = static_cast<const uint8_t*>(W);
  if (d->oc == 1) {
    rwkvq_status st = check_vector_desc(d, d->ic);
    if (st != RWKVQ_OK) return st;
    int n = d->ic / 2;
    dequant_vector_kernel<<<(n + 255) / 256, 256, 0, s>>>(img + RWKVQ_HEADER_BYTES, img + vector_aux_offset(d), d->ic, d->bits, out, dtype);
    return cuda_status(cudaGetLastError());
  }
  rwkvq_status st = check_matrix_desc(d);
  if (st != RWKVQ_OK) return st;
  const int KT = d->ic_pad / 256, nrec = (d->oc_pad / 128) * KT * 8;
  const uint8_t* payload = img + RWKVQ_HEADER_BYTES;
  const uint8_t* aux = img + matrix_aux_offset(d);
  const int fmt = fmt_of(d);
  dim3 grid((nrec + 3) / 4);
  if (fmt == FMT_SQ3) dequant_kernel<FMT_SQ3><<<grid, 128, 0, s>>>(payload, aux, d->oc, d->ic, KT, d->entries, out, dtype, nrec);
  else if (fmt == FMT_VQ6) dequant_kernel<FMT_VQ6><<<grid, 128, 0, s>>>(payload, aux, d->oc, d->ic, KT, d->entries, out, dtype, nrec);
  else dequant_kernel<FMT_VQ8><<<grid, 128, 0, s>>>(payload, aux, d->oc, d->ic, KT, d->entries, out, dtype, nrec);
  return cuda_status(cudaGetLastError());
}

size_t rwkvq_quant_error_workspace_bytes(const rwkvq_desc* d) {
  if (!d || d->oc == 1 || check_matrix_desc(d) != RWKVQ_OK) return 0;
  return (size_t)(d->oc_pad / 128) * (d->ic_pad / 256) * 8 * sizeof(double) + 256;
}

rwkvq_status rwkvq_quant_error(const void* w, const rwkvq_desc* d, const void* W, double* sse_host, void* ws,
                               size_t ws_bytes, void* stream) {
  if (!w || !d || !W || !sse_host || !ws) return RWKVQ_EINVAL;
  if (d->oc == 1) return RWKVQ_ESHAPE;
  rwkvq_status st = check_matrix_desc(d);
  if (st != RWKVQ_OK) return st;
  if (!aligned16(w) || !aligned16(W) || !aligned16(ws)) return RWKVQ_EALIGN;
  if (ws_bytes < rwkvq_quant_error_workspace_bytes(d)) return RWKVQ_ENOMEM;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const uint8_t* img = static_cast<const uint8_t*>(W);
  const int KT = d->ic_pad / 256, nrec = (d->oc_pad / 128) * KT * 8;
  const uint8_t* payload = img + RWKVQ_HEADER_BYTES;
  const uint8_t* aux = img + matrix_aux_offset(d);
  double* total = static_cast<double*>(ws);
  double* partial = reinterpret_cast<double*>(static_cast<uint8_t*>(ws) + 256);
  const __half* ref = static_cast<const __half*>(w);
  const int fmt = fmt_of(d);
  dim3 grid((nrec + 3) / 4);
  if (fmt == FMT_SQ3) dequant_kernel<FMT_SQ3><<<grid, 128, 0, s>>>(payload, aux, d->oc, d->ic, KT, d->entries, nullptr, 0, nrec, ref, partial);
  else if (fmt == FMT_VQ6) dequant_kernel<FMT_VQ6><<<grid, 128, 0, s>>>(payload, aux, d->oc, d->ic, KT, d->entries, nullptr, 0, nrec, ref, partial);
  else dequant_kernel<FMT_VQ8><<<grid, 128, 0, s>>>(payload, aux, d->oc, d->ic, KT, d->entries, nullptr, 0, nrec, ref, partial);
  sum_fixed_kernel<<<1, 1024, 0, s>>>(partial, nrec, total);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(sse_host, total, sizeof(double), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  return cuda_status(e);
}

}  // extern "C"
