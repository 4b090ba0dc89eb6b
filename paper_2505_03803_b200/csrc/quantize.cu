// Device quantizers: the round-to-nearest scalar quantizer of Section 3.2 Eq. 2, the k-means
// vector quantizer of Section 3.2 Eq. 3 (one codebook per 256 x 256 tile, or per token-shift
// vector), the X^2-weighted k-means of Section 4.2 Eq. 19 for token-shift vectors, and the
// percentile-clipped representative activation of Section 4.2.  Each writes the packed device
// image of format.h directly; nothing passes through the host.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "../../include/rwkvq.h"
#include "format.h"
#include "host_util.h"

namespace rwkvq {
namespace {

constexpr int kFlagNonFinite = 1, kFlagTimeout = 2;

// Every kernel here is launched while the one before it still runs, lets the next one be, and touches memory behind this: a call of short kernels
// otherwise waits 2 us for each to start (five vectors of 4096 with 128 samples, ten kernels: 303 -> 288 us; a layer of 512 columns 284 -> 270).
// What the kernel before may still write while this one is resident is not read through the read-only path, whose data has to stay as it is for the
// whole life of the reading kernel: __ldcg, or an ordinary load where it is read again.
__device__ __forceinline__ void after_the_kernel_before() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;");
}

// The first block of a quantizer kernel also writes the image's header and clears the alignment padding behind its last section
// (a launch and a memset of their own took as long as quantizing a small matrix).
__device__ __forceinline__ void write_header(const rwkvq_image_header& h, uint8_t* image) {
  const uint32_t* src = reinterpret_cast<const uint32_t*>(&h);
  if (threadIdx.x < RWKVQ_HEADER_BYTES / 4) reinterpret_cast<uint32_t*>(image)[threadIdx.x] = src[threadIdx.x];
  const uint64_t used = h.off_aux + h.aux_bytes;
  for (uint64_t i = used + threadIdx.x; i < h.image_bytes; i += blockDim.x) image[i] = 0;
}

// Two fp32 operations in one instruction, each rounded as the single one is.
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 r;
  asm("{\n .reg .b64 x, y, z;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n add.rn.f32x2 z, x, y;\n mov.b64 {%0, %1}, z;\n}" : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  float2 r;
  asm("{\n .reg .b64 x, y, z;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n mul.rn.f32x2 z, x, y;\n mov.b64 {%0, %1}, z;\n}" : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 r;
  asm("{\n .reg .b64 x, y, z, w;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n mov.b64 w, {%6, %7};\n fma.rn.f32x2 z, x, y, w;\n mov.b64 {%0, %1}, z;\n}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return r;
}

// ---- scalar quantizer ------------------------------------------------------------------------
//
// One warp per record (16 rows x 256 columns).  A lane keeps its eight columns of all sixteen
// rows in registers (lanes 0..15 have group 0, lanes 16..31 group 1), so that the matrix is read once, sixteen 16-byte loads in flight.
// The (row, group) minima and maxima are reduced sixteen rows at once: each step exchanges half of the rows that a lane still
// has, 15 shuffles in all, and lane r + 16 h ends with (row r, group h), whose (s, z) it derives
// in fp64 exactly as Eq. 2 prescribes.
//
// A code is clamp(round(w / s) + z, 0, 7), ties to even before z is added.  The quotient by Markstein's correction of w * (1/s) with fused
// multiply-adds ("Computation of elementary functions on the IBM RISC System/6000 processor", 1990): an m + 1/2 comes out exact, and any other
// quotient below 8 is at least 2^-13 away from one (w and s have 11 bits) while the correction leaves 2^-21.  Then (w / s + z) / 8, saturated
// to [0, 1], plus 1.5 * 2^20, whose last place is 1/8: the addition rounds, and the code is in the low bits.  An odd z would turn the ties; with
// one more in the constant they fall as they should, and the code is one more, too.  Eight, where the largest quotient rounds up,
// becomes seven for four codes at once.  These are multiply-adds beside the integer pipe, which holds this kernel (minima and maxima, codes, bit
// packing): choosing among seven exact thresholds by three packed comparisons kept it busy half as long again.  Twenty warps an SM in blocks of four: with
// sixteen in blocks of eight, 1792 chunks are seven rounds of 6.05, with sixteen in blocks of four 37.1 us, with twenty-four (spilled) 40.
// 14336 x 4096: 35.1 us (45.4 with the comparisons, 40.6 without them), 4096 x 4096: 14.6 (18.2).
constexpr int kSqWarps = 4;              // of a block; twenty on an SM
constexpr int kSqRowStride = 256 + 16;   // bytes per row of the code staging area: conflict-free lane reads

__device__ __forceinline__ float h2f_bits(uint32_t h) { return __half2float(__ushort_as_half((unsigned short)h)); }
__device__ __forceinline__ __half2 as_h2(uint32_t v) { return *reinterpret_cast<__half2*>(&v); }
__device__ __forceinline__ uint32_t as_u32(__half2 v) { return *reinterpret_cast<uint32_t*>(&v); }

__global__ void __launch_bounds__(32 * kSqWarps, 20 / kSqWarps) sq_quantize_kernel(const uint16_t* w, int oc, int ic, int KT,
                                                             uint8_t* __restrict__ payload, int* __restrict__ flags,
                                                             const __grid_constant__ rwkvq_image_header head, uint8_t* image) {
  __shared__ __align__(16) uint8_t codes_all[kSqWarps][16 * kSqRowStride];
  __shared__ float4 code_all[kSqWarps][2][16];                     // [warp][group][row]: -s, 1/s, z / 8, 1.5 * 2^20 (+ 1/8 for an odd z)
  after_the_kernel_before();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (blockIdx.x == 0) write_header(head, image);
  const unsigned record = blockIdx.x * kSqWarps + warp, chunk = record >> 3;
  const int mb = (int)(chunk / (unsigned)KT), kt = (int)(chunk % (unsigned)KT);
  const int r0 = mb * 128 + (int)(record & 7u) * 16, c0 = kt * 256;
  uint8_t* codes = codes_all[warp];
  const int half = lane >> 4;
  const int col = c0 + 8 * lane;
  const bool col_in = col < ic;            // ic is a multiple of 128: a whole group is inside or outside
  const uint16_t* src = w + (size_t)r0 * ic + col;
  uint32_t ext[16];                        // (minimum, -maximum) of the lane's columns of a row; a NaN stays
  uint4 v[16];
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    v[r] = make_uint4(0, 0, 0, 0);
    if (col_in && r0 + r < oc) v[r] = __ldcg(reinterpret_cast<const uint4*>(src + (size_t)r * ic));
  }
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    const uint32_t mn = as_u32(__hmin2_nan(__hmin2_nan(as_h2(v[r].x), as_h2(v[r].y)), __hmin2_nan(as_h2(v[r].z), as_h2(v[r].w))));
    const uint32_t mx = as_u32(__hmax2_nan(__hmax2_nan(as_h2(v[r].x), as_h2(v[r].y)), __hmax2_nan(as_h2(v[r].z), as_h2(v[r].w)))) ^ 0x80008000u;
    ext[r] = as_u32(__hmin2_nan(as_h2(__byte_perm(mn, mx, 0x5410u)), as_h2(__byte_perm(mn, mx, 0x7632u))));
  }
#pragma unroll
  for (int half_rows = 8; half_rows >= 1; half_rows >>= 1) {
    const bool upper = (lane & half_rows) != 0;
#pragma unroll
    for (int r = 0; r < half_rows; ++r) {
      const uint32_t keep = upper ? ext[r + half_rows] : ext[r], give = upper ? ext[r] : ext[r + half_rows];
      ext[r] = as_u32(__hmin2_nan(as_h2(keep), as_h2(__shfl_xor_sync(0xFFFFFFFFu, give, half_rows))));
    }
  }
  const float my_mn = __low2float(as_h2(ext[0])), my_mx = -__high2float(as_h2(ext[0]));
  // an all-ones exponent carries into bit 15 of its half
  if (((ext[0] & 0x7C007C00u) + 0x04000400u) & 0x80008000u) atomicOr(flags, kFlagNonFinite);
  // (s, z) of (row lane & 15, group half), Eq. 2; a constant group c is coded exactly:
  // c == 0 -> (1, 0, q 0), c > 0 -> (c, 0, q 1), c < 0 -> (|c|, 1, q 0).
  float my_s, my_z;
  {
    const double mn = (double)my_mn, mx = (double)my_mx;
    const __half s16 = __double2half((mx - mn) / 7.0);
    const double s = (double)__half2float(s16);
    float inv, add;
    if (mx == mn || s == 0.0) {
      my_s = mn == 0.0 ? 1.f : fabsf(my_mn);
      my_z = mn < 0.0 ? 1.f : 0.f;
      inv = 0.f;                                   // the same code for all
      add = mn > 0.0 ? 1.f : 0.f;
    } else {
      my_s = (float)s;
      my_z = (float)fmin(7.0, fmax(0.0, rint(-mn / s)));
      inv = 1.f / my_s;
      add = my_z;
    }
    code_all[warp][half][lane & 15] = make_float4(-my_s, inv, add * 0.125f, 1572864.f + (((int)add & 1) ? 0.125f : 0.f));
  }
  __syncwarp();
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    const bool inside = col_in && (r0 + r) < oc;
    const float4 c = code_all[warp][half][r];
    const float2 neg_s = make_float2(c.x, c.x), inv = make_float2(c.y, c.y), magic = make_float2(c.w, c.w);
    const uint32_t odd = (__float_as_uint(c.w) & 1u) * 0x01010101u;
    const uint32_t words[4] = {v[r].x, v[r].y, v[r].z, v[r].w};
    uint32_t bits[8];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2 x = __half22float2(as_h2(words[k]));
      const float2 q0 = mul2(x, inv), q1 = fma2(fma2(q0, neg_s, x), inv, q0);
      const float2 sum = add2(make_float2(__saturatef(fmaf(q1.x, 0.125f, c.z)), __saturatef(fmaf(q1.y, 0.125f, c.z))), magic);
      bits[2 * k] = __float_as_uint(sum.x); bits[2 * k + 1] = __float_as_uint(sum.y);
    }
    uint2 out;
    out.x = __byte_perm(__byte_perm(bits[0], bits[1], 0x0040u), __byte_perm(bits[2], bits[3], 0x0040u), 0x5410u) - odd;
    out.y = __byte_perm(__byte_perm(bits[4], bits[5], 0x0040u), __byte_perm(bits[6], bits[7], 0x0040u), 0x5410u) - odd;
    out.x -= (out.x >> 3) & 0x01010101u;
    out.y -= (out.y >> 3) & 0x01010101u;
    *reinterpret_cast<uint2*>(codes + r * kSqRowStride + 8 * lane) = inside ? out : make_uint2(0u, 0u);
  }
  __syncwarp();
  // Bit packing of format.h: lane (g, t) owns rows g and g + 8 and, in every tensor-core step,
  // the four columns 4t .. 4t+3 (one 32-bit read of the staging area = registers R and R + 2).
  const int g = lane >> 2, t = lane & 3;
  uint8_t* rec = payload + (size_t)record * RWKVQ_SQ_RECORD_BYTES;
  uint32_t wd[12];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    uint32_t w3[3] = {0u, 0u, 0u};
#pragma unroll
    for (int m = 0; m < 4; ++m) {
#pragma unroll
      for (int hrow = 0; hrow < 2; ++hrow) {
        const uint32_t four = *reinterpret_cast<const uint32_t*>(codes + (g + 8 * hrow) * kSqRowStride + 64 * i + 16 * m + 4 * t);
#pragma unroll
        for (int cp = 0; cp < 2; ++cp) {
          const int e = 4 * m + 2 * cp + hrow;             // register R = 2 * cp + hrow of step m
          const uint32_t pair = __byte_perm(four, 0u, cp ? 0x4342u : 0x4140u);   // (even column) | (odd column) << 16
          if (e < 15) {
            w3[e / 5] |= pair << (3 * (e % 5));
          } else {
#pragma unroll
            for (int b = 0; b < 3; ++b) w3[b] |= ((pair >> b) & 0x00010001u) << 15;
          }
        }
      }
    }
    wd[3 * i] = w3[0]; wd[3 * i + 1] = w3[1]; wd[3 * i + 2] = w3[2];
  }
#pragma unroll
  for (int p = 0; p < 3; ++p)
    *reinterpret_cast<uint4*>(rec + p * 512 + lane * 16) = make_uint4(wd[4 * p], wd[4 * p + 1], wd[4 * p + 2], wd[4 * p + 3]);
  // plane 3: for g = 0..7 the (s, z) pairs of (row g, group 0), (row g, group 1), (row g+8, group 0), (row g+8, group 1)
  {
    const int r = lane & 15;
    const bool inside = (r0 + r) < oc && (c0 + 128 * half) < ic;
    const uint32_t s_bits = inside ? (uint32_t)__half_as_ushort(__float2half_rn(my_s)) : 0u;
    const uint32_t z_bits = inside ? (uint32_t)__half_as_ushort(__float2half_rn(my_z)) : 0u;
    *reinterpret_cast<uint32_t*>(rec + RWKVQ_SQ_CODE_BYTES + (r & 7) * 16 + ((r >> 3) * 2 + half) * 4) = s_bits | (z_bits << 16);
  }
}

// ---- vector quantizer ------------------------------------------------------------------------
//
// k-means++ seeding and Lloyd iterations in fp32 with exact integer cluster sums, one cluster of blocks per codebook.  Two kinds:
// a 256 x 256 tile (32 768 two-element vectors, vector i = 128 * row + pair) and a token-shift vector (ic / 2 vectors,
// optionally weighted).  Both draw the same seeds: the distances are summed over runs of 64 consecutive vectors in
// order, the run sums by a scan over the lanes of a warp and then warp by warp, all in fp32, and a draw falls on
// the last vector whose running sum begins at or below the target.
constexpr int kVqThreads = 512;
constexpr int kVqPerThread = 64;
constexpr int kVqMaxVec = kVqThreads * kVqPerThread;   // 32768
constexpr int kVqMaxE = 256;

// Draw number k (0-based) of the generator of Steele, Lea, Flood: "Fast splittable pseudorandom number generators" (2014).
__device__ __forceinline__ uint64_t splitmix(uint64_t seed, int k) {
  uint64_t z = seed + (uint64_t)(k + 1) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
__device__ __forceinline__ double unit_of(uint64_t r) { return (double)(r >> 11) * (1.0 / 9007199254740992.0); }
__device__ __forceinline__ int below(uint64_t r, int n) {
  return (int)((unsigned long long)(unit_of(r) * (double)n) % (unsigned long long)n);
}

constexpr uint32_t kDefaultPollLimit = 1u << 20, kNoBlock = ~0u;      // a try takes up to 4 us
struct VqArgs {
  const uint16_t* w;        // matrix [oc][ic] or vector [ic]
  const float* elem_w;      // vector mode: X^2 per element, or NULL
  int ic;                   // row length of w
  int TC;                   // tiles per row of tiles (matrix mode)
  int n_vec;                // vectors per codebook
  int E, iters;
  uint32_t poll_limit;      // tries of a wait between the blocks of a cluster
  uint32_t mute;            // block of each cluster that sends nothing, for a test; kNoBlock: none
  uint64_t seed;
  uint8_t* payload;         // matrix: chunk grid; vector: bit stream
  uint32_t* aux;            // codebooks, E half2 each
  int* flags;
};

// fp16 value times 2^24 as an exact integer (|v| < 2^16, multiples of 2^-24)
__device__ __forceinline__ long long half_fixed(uint32_t h) {
  const int e = (h >> 10) & 31, m = h & 1023;
  const long long mag = e ? ((long long)(m + 1024) << (e - 1)) : (long long)m;
  return (h & 0x8000u) ? -mag : mag;
}

__device__ __forceinline__ float d2f(float x, float y, float2 c) {
  const float dx = x - c.x, dy = y - c.y;
  return fmaf(dx, dx, dy * dy);
}
__device__ __forceinline__ float2 vec_of(uint32_t v) { return make_float2(h2f_bits(v & 0xFFFFu), h2f_bits(v >> 16)); }
// Exact cluster sums with native 32-bit shared-memory atomics (a 64-bit one is a compare-and-swap loop): the fixed-point
// value is added as signed pieces of 13, 13 and 14 bits; 32 768 of them stay below 2^29.  The last piece is zero for
// |w| < 4 and then skipped.  Layout [piece][centre].
template <int E>
struct ClusterSums {
  int x[3][E], y[3][E], cnt[E];
};
template <int E>
__device__ __forceinline__ void add_sum(int (*sum)[E], int e, long long v) {
  const int sg = v < 0 ? -1 : 1;
  const unsigned long long m = (unsigned long long)(v < 0 ? -v : v);
  atomicAdd(&sum[0][e], sg * (int)(m & 0x1FFFu));
  const int p1 = (int)((m >> 13) & 0x1FFFu), p2 = (int)(m >> 26);
  if (p1) atomicAdd(&sum[1][e], sg * p1);
  if (p2) atomicAdd(&sum[2][e], sg * p2);
}
__device__ __forceinline__ double mean_of_pieces(int p0, int p1, int p2, int cnt) {
  const long long s = (long long)p0 + ((long long)p1 << 13) + ((long long)p2 << 26);
  return (double)s * (1.0 / 16777216.0) / (double)cnt;
}
// Numbers below 4 in magnitude are 26-bit integers times 2^-24: two pieces, without 64-bit arithmetic.
constexpr float kTwoPieces = 4.f;
struct Pieces { int lo, hi; };
__device__ __forceinline__ Pieces two_pieces(float v) {
  const int q = __float2int_rn(v * 16777216.f);
  return Pieces{q & 0x1FFF, q >> 13};
}
// A vector leaves centre `from` and joins `to`.
template <int E>
__device__ __forceinline__ void move_member(ClusterSums<E>& s, uint32_t bits, int from, int to) {
  const float2 f = vec_of(bits);
  if (fmaxf(fabsf(f.x), fabsf(f.y)) < kTwoPieces) {
    const Pieces x = two_pieces(f.x), y = two_pieces(f.y);
    atomicAdd(&s.x[0][from], -x.lo); atomicAdd(&s.x[1][from], -x.hi); atomicAdd(&s.y[0][from], -y.lo); atomicAdd(&s.y[1][from], -y.hi);
    atomicAdd(&s.x[0][to], x.lo); atomicAdd(&s.x[1][to], x.hi); atomicAdd(&s.y[0][to], y.lo); atomicAdd(&s.y[1][to], y.hi);
  } else {
    const long long x = half_fixed(bits & 0xFFFFu), y = half_fixed(bits >> 16);
    add_sum(s.x, from, -x); add_sum(s.y, from, -y);
    add_sum(s.x, to, x); add_sum(s.y, to, y);
  }
  atomicAdd(&s.cnt[from], -1);
  atomicAdd(&s.cnt[to], 1);
}

// All 64 vectors of a group (two a lane) join one centre.
template <int E>
__device__ __forceinline__ void join_group(ClusterSums<E>& s, uint32_t v0, uint32_t v1, int e) {
  const float2 f0 = vec_of(v0), f1 = vec_of(v1);
  const bool small = fmaxf(fmaxf(fabsf(f0.x), fabsf(f0.y)), fmaxf(fabsf(f1.x), fabsf(f1.y))) < kTwoPieces;
  if (__all_sync(0xFFFFFFFFu, small)) {
    const Pieces x0 = two_pieces(f0.x), y0 = two_pieces(f0.y), x1 = two_pieces(f1.x), y1 = two_pieces(f1.y);
    const int xl = __reduce_add_sync(0xFFFFFFFFu, x0.lo + x1.lo), xh = __reduce_add_sync(0xFFFFFFFFu, x0.hi + x1.hi);
    const int yl = __reduce_add_sync(0xFFFFFFFFu, y0.lo + y1.lo), yh = __reduce_add_sync(0xFFFFFFFFu, y0.hi + y1.hi);
    if ((threadIdx.x & 31) == 0) { atomicAdd(&s.x[0][e], xl); atomicAdd(&s.x[1][e], xh); atomicAdd(&s.y[0][e], yl); atomicAdd(&s.y[1][e], yh); }
  } else {
    add_sum(s.x, e, half_fixed(v0 & 0xFFFFu)); add_sum(s.y, e, half_fixed(v0 >> 16));
    add_sum(s.x, e, half_fixed(v1 & 0xFFFFu)); add_sum(s.y, e, half_fixed(v1 >> 16));
  }
  if ((threadIdx.x & 31) == 0) atomicAdd(&s.cnt[e], 64);
}

// Clusters: barrier, and accesses to the shared memory of a block at the address that `local` has here.
__device__ __forceinline__ uint32_t cluster_rank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ void cluster_arrive() { __syncwarp(); asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { __syncwarp(); asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t peer_address(uint32_t local, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
  return r;
}
// A store to a block of the cluster that its barrier `bar` counts.
__device__ __forceinline__ void peer_send(uint32_t at, ulonglong2 v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(at), "l"(v.x), "l"(v.y), "r"(bar) : "memory");
}
__device__ __forceinline__ void peer_send(uint32_t at, unsigned long long v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(at), "l"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ uint32_t shared_address(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void expect_sent(uint32_t bar, int bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void peer_send(uint32_t at, uint32_t v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(at), "r"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ void peer_store(uint32_t at, uint32_t v0, uint32_t v1) { asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(at), "r"(v0), "r"(v1) : "memory"); }
__device__ __forceinline__ uint32_t peer_load(uint32_t at) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(at) : "memory");
  return v;
}
__device__ __forceinline__ uint4 peer_load4(uint32_t at) {
  uint4 v;
  asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(at) : "memory");
  return v;
}
// Waits for a phase of a barrier of this block that stores of the cluster complete; gives up after `limit` tries.
__device__ __forceinline__ bool wait_sent(uint32_t bar, uint32_t parity, uint32_t limit) {
  for (uint32_t i = 0; i < limit; ++i) {
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}" : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    if (ok) return true;
  }
  return false;
}
// A block that has given up stays for some milliseconds after all others have sent what they will: what is still on its way to it lands.
__device__ __forceinline__ void stay_behind() {
  for (int i = 0; i < 8; ++i) __nanosleep(1000000);
}

// ---- seeds ----
//
// A thread has the distances of 64 consecutive vectors in registers; the vectors stay in shared memory as fp16 pairs (read 16 bytes at a time,
// the pieces of a thread's row rotated against bank conflicts).  Seeds are vectors of the tile, so the codebook area of the image holds them
// exactly until the centres are final.
__device__ __forceinline__ int vq_slot(int i) { return (i & ~63) | ((((i >> 2) ^ (i >> 6)) & 7) << 2) | (i & 35); }

// v - c with the fp16 pair v widened and each difference rounded once.
__device__ __forceinline__ void sub_pair(uint32_t v, float cx, float cy, float& dx, float& dy) {
  asm("{\n .reg .b16 x, y;\n mov.b32 {x, y}, %2;\n sub.rn.f32.f16 %0, x, %3;\n sub.rn.f32.f16 %1, y, %4;\n}" : "=f"(dx), "=f"(dy) : "r"(v), "f"(cx), "f"(cy));
}
// Distances to one more centre for a thread's 64 vectors; their sum in order.
__device__ __forceinline__ float nearer(float (&dist)[kVqPerThread], const uint32_t* vec, int base, uint32_t centre) {
  const float2 c = vec_of(centre);
  float local = 0.f;
#pragma unroll
  for (int k = 0; k < kVqPerThread; k += 4) {
    const uint4 q = *reinterpret_cast<const uint4*>(vec + vq_slot(base + k));
    float2 dxa, dya, dxb, dyb;
    sub_pair(q.x, c.x, c.y, dxa.x, dya.x); sub_pair(q.y, c.x, c.y, dxa.y, dya.y);
    sub_pair(q.z, c.x, c.y, dxb.x, dyb.x); sub_pair(q.w, c.x, c.y, dxb.y, dyb.y);
    const float2 da = fma2(dxa, dxa, mul2(dya, dya)), db = fma2(dxb, dxb, mul2(dyb, dyb));
    dist[k] = fminf(dist[k], da.x); dist[k + 1] = fminf(dist[k + 1], da.y);
    dist[k + 2] = fminf(dist[k + 2], db.x); dist[k + 3] = fminf(dist[k + 3], db.y);
    local += dist[k]; local += dist[k + 1]; local += dist[k + 2]; local += dist[k + 3];
  }
  return local;
}
// Sums over the lanes of a warp up to and including this one.
__device__ __forceinline__ float sum_to_lane(float v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const float o = __shfl_up_sync(0xFFFFFFFFu, v, off);
    if (lane >= off) v += o;
  }
  return v;
}
// Sums of all warps, and of those in front of number `warp`.
__device__ __forceinline__ void warp_sums(const float* tot, int warp, float& before, float& total) {
  before = total = 0.f;
#pragma unroll
  for (int w4 = 0; w4 < kVqMaxVec / 2048 / 4; ++w4) {
    const float4 t4 = *reinterpret_cast<const float4*>(tot + 4 * w4);
    const float tt[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (4 * w4 + k == warp) before = total;
      total += tt[k];
    }
  }
}
// Last vector of a thread's run whose running sum, from `acc` on, begins at or below the target.
__device__ __forceinline__ int last_at_or_below(const float (&dist)[kVqPerThread], float acc, float target, int base, int n) {
  int pick = base;
#pragma unroll
  for (int k = 0; k < kVqPerThread; ++k) {
    if (acc <= target && base + k < n) pick = base + k;
    acc += dist[k];
  }
  return pick;
}

// Rows of a tile to their slots; a warp reads 512 contiguous bytes, one row.
__device__ __forceinline__ void load_rows(uint32_t* vec, const uint16_t* src, int ic, int rows, int warps, int* flags) {
  const int lane = threadIdx.x & 31;
  bool bad = false;
#pragma unroll 4
  for (int r = threadIdx.x >> 5; r < rows; r += warps) {
    const uint4 q = __ldcg(reinterpret_cast<const uint4*>(src + (size_t)r * ic) + lane);
    const uint32_t v[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) bad |= ((v[k] & 0x7C00u) == 0x7C00u) | ((v[k] & 0x7C000000u) == 0x7C000000u);
    *reinterpret_cast<uint4*>(vec + vq_slot(r * 128 + lane * 4)) = q;
  }
  if (bad) atomicOr(flags, kFlagNonFinite);
}
__device__ __forceinline__ uint64_t tile_seed(uint64_t seed, int tile) { return seed * 0x9E3779B97F4A7C15ull + (uint64_t)tile + 1ull; }

// Few tiles: a cluster of four blocks each, 64 rows (four warps) a block.  A draw hands over twice: every warp's sum goes to all blocks, and the
// drawn vector from the block that has it.  Bound by the latency of a draw (0.97 us: half of it the two trips, a quarter the distances).  64 entries: 62 us
// for up to 33 tiles, 79 for 64, 95 for 100; a block a tile, bound by the instructions of the distances (six a vector), 92 in every case (117 with the
// fp16 numbers converted before the difference was taken).
constexpr int kTileBlocks = 4, kPartVec = kVqMaxVec / kTileBlocks, kSeedThreads = kPartVec / kVqPerThread;
struct TileSeeds {
  uint32_t vec[kPartVec];
  float tot[2][kVqMaxVec / 2048];                // sums of the tile's warps, for every other draw
  float u01[kVqMaxE];
  uint64_t tot_here[2], pick_here;
  uint32_t pick;
};
__global__ void __launch_bounds__(kSeedThreads, 4) vq_tile_seed_kernel(const VqArgs a) {
  after_the_kernel_before();
  extern __shared__ __align__(16) uint8_t smem[];
  TileSeeds& sh = *reinterpret_cast<TileSeeds*>(smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, E = a.E;
  const uint32_t rank = cluster_rank();
  const int tile = blockIdx.x / kTileBlocks, tr = tile / a.TC, tc = tile % a.TC;
  const uint32_t tot_here = shared_address(&sh.tot_here[0]), pick_here = shared_address(&sh.pick_here);
  if (tid == 0)
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n mbarrier.init.shared::cta.b64 [%1], 1;\n mbarrier.init.shared::cta.b64 [%2], 1;\n fence.mbarrier_init.release.cluster;"
                 ::"r"(tot_here), "r"(tot_here + 8), "r"(pick_here) : "memory");
  load_rows(sh.vec, a.w + (size_t)(tr * 256 + (int)rank * (256 / kTileBlocks)) * a.ic + tc * 256, a.ic, 256 / kTileBlocks, kSeedThreads / 32, a.flags);
  const uint64_t seed = tile_seed(a.seed, tile);
  for (int e = tid; e < E; e += kSeedThreads) sh.u01[e] = (float)unit_of(splitmix(seed, e));
  __syncthreads();
  cluster_arrive();
  cluster_wait();
  const int base = tid * kVqPerThread, tile_warp = (int)rank * (kSeedThreads / 32) + warp;
  float dist[kVqPerThread];
#pragma unroll
  for (int k = 0; k < kVqPerThread; ++k) dist[k] = INFINITY;
  uint32_t* aux = a.aux + (size_t)tile * E;
  bool lost = false;
  // the block with vector `at` sends it to all
  const bool mute = rank == a.mute;
  auto send = [&](int at) {
    if (mute) return;
    const uint32_t v = sh.vec[vq_slot(at)];
#pragma unroll
    for (uint32_t r = 0; r < kTileBlocks; ++r) peer_send(peer_address(shared_address(&sh.pick), r), v, peer_address(pick_here, r));
  };
  // a warp whose wait has run out leaves: it neither sends nor expects any more, and the others' waits run out in turn
  auto wait = [&](uint32_t bar, uint32_t parity) { lost = !__all_sync(0xFFFFFFFFu, wait_sent(bar, parity, a.poll_limit)); };
  const int first = below(splitmix(seed, 0), kVqMaxVec);
  if (tid == 0 && first / kPartVec == (int)rank) send(first % kPartVec);
  for (int e = 0;; ++e) {
    // A block sends its next draw when it has the next sums of all warps, and a warp its next sums when it has this draw; the sums of two draws
    // are under way at once, to places and barriers of their own.
    if (tid == 0) expect_sent(pick_here, 4);
    wait(pick_here, (uint32_t)e & 1u);
    if (lost) break;
    const uint32_t cv = sh.pick;
    if (tid == 0 && rank == 0u) aux[e] = cv;
    if (e + 1 == E) break;
    const float local = nearer(dist, sh.vec, base, cv);
    const float incl = sum_to_lane(local);
    const uint32_t bar = tot_here + 8 * (e & 1);
    if (tid == 0) expect_sent(bar, (int)sizeof(sh.tot[0]));
    if (lane == 31 && !mute) {
#pragma unroll
      for (uint32_t r = 0; r < kTileBlocks; ++r)
        peer_send(peer_address(shared_address(&sh.tot[e & 1][tile_warp]), r), __float_as_uint(incl), peer_address(bar, r));
    }
    float excl = __shfl_up_sync(0xFFFFFFFFu, incl, 1);
    if (lane == 0) excl = 0.f;
    wait(bar, (uint32_t)(e >> 1) & 1u);
    if (lost) break;
    float before, total;
    warp_sums(sh.tot[e & 1], tile_warp, before, total);
    const float target = sh.u01[e + 1] * total;
    if (!(total > 0.f) || !(target < total)) {       // no distance left, or nothing behind the target
      const int at = total > 0.f ? kVqMaxVec - 1 : below(splitmix(seed, e + 1), kVqMaxVec);
      if (tid == 0 && at / kPartVec == (int)rank) send(at % kPartVec);
    } else if (before <= target && target < before + sh.tot[e & 1][tile_warp]) {      // one warp: the sums in front of the warps do not fall
      const uint32_t hit = __ballot_sync(0xFFFFFFFFu, before + excl <= target && target < before + incl);
      if (hit != 0u && lane == __ffs((int)hit) - 1) send(last_at_or_below(dist, before + excl, target, base, kPartVec));
    }
  }
  if (lost) atomicOr(a.flags, kFlagTimeout);
  cluster_arrive();
  cluster_wait();
  if (lost) stay_behind();
}

// One block: a tile, where there are enough of them for every SM (hand-overs cost less inside a block), or a token-shift vector of n vectors, more
// than kVecSeeds, with n / 2048 warps.
constexpr int kVqWarps = kVqThreads / 32;
struct SeedShared {
  float warp_tot[kVqWarps];
  float u01[kVqMaxE];
  int pick[kVqMaxE];
};
template <bool kVector>
__global__ void __launch_bounds__(kVqThreads, 1) vq_seed_kernel(const VqArgs a) {
  after_the_kernel_before();
  extern __shared__ __align__(16) uint8_t smem[];
  uint32_t* vec = reinterpret_cast<uint32_t*>(smem);
  const int n = kVector ? a.n_vec : kVqMaxVec, E = a.E, threads = kVector ? (int)blockDim.x : kVqThreads;
  SeedShared& sh = *reinterpret_cast<SeedShared*>(smem + (size_t)threads * kVqPerThread * 4);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tile = blockIdx.x, tr = tile / a.TC, tc = tile % a.TC;
  if (kVector) {
    const uint32_t* src = reinterpret_cast<const uint32_t*>(a.w);
    bool bad = false;
    for (int i = tid; i < threads * kVqPerThread; i += threads) {
      const uint32_t v = i < n ? __ldcg(src + i) : 0u;
      bad |= ((v & 0x7C00u) == 0x7C00u) | ((v & 0x7C000000u) == 0x7C000000u);
      vec[vq_slot(i)] = v;
    }
    if (bad) atomicOr(a.flags, kFlagNonFinite);
    if (tid < kVqWarps) sh.warp_tot[tid] = 0.f;
  } else {
    load_rows(vec, a.w + (size_t)(tr * 256) * a.ic + tc * 256, a.ic, 256, kVqWarps, a.flags);
  }
  const uint64_t seed = kVector ? a.seed : tile_seed(a.seed, tile);
  for (int e = tid; e < E; e += threads) {
    sh.u01[e] = (float)unit_of(splitmix(seed, e));
    sh.pick[e] = n - 1;
  }
  __syncthreads();
  uint32_t* aux = a.aux + (size_t)tile * E;
  const int base = tid * kVqPerThread;
  float dist[kVqPerThread];
#pragma unroll
  for (int k = 0; k < kVqPerThread; ++k) dist[k] = !kVector || base + k < n ? INFINITY : 0.f;
  int at = below(splitmix(seed, 0), n);
  for (int e = 0; e < E; ++e) {
    const uint32_t cv = vec[vq_slot(at)];
    if (tid == 0) aux[e] = cv;
    if (e + 1 == E) break;
    const float local = nearer(dist, vec, base, cv);
    float incl = sum_to_lane(local);
    if (lane == 31) sh.warp_tot[warp] = incl;
    float excl = __shfl_up_sync(0xFFFFFFFFu, incl, 1);
    if (lane == 0) excl = 0.f;
    __syncthreads();
    float before, total;
    warp_sums(sh.warp_tot, warp, before, total);
    excl = before + excl;
    incl = before + incl;
    const float target = sh.u01[e + 1] * total;
    if (total > 0.f && excl <= target && target < incl) sh.pick[e + 1] = last_at_or_below(dist, excl, target, base, n);
    __syncthreads();
    at = total > 0.f ? sh.pick[e + 1] : below(splitmix(seed, e + 1), n);
  }
}

// ---- tiles ----
//
// Lloyd iterations.  The assignment takes the nearest centre of all E, but looks at a few: the vectors are sorted once along
// a Hilbert curve over 64 x 64 cells and every 64 neighbours form a group with a box around them.  In every iteration two threads
// strike out, for one group, the centres that cannot be nearest to any point of its box: those the box lies wholly on the
// far side of, at their bisector with one centre near the box, by a margin far above the rounding of the fp32 (and fp64)
// distances.  The assignment found among the others, lowest index first, is therefore the one that all E centres would give,
// bit for bit.  Then the groups are dealt over the warps in turn (the long lists lie together, in the tails), all lanes of a
// warp testing the same candidates for two neighbours each, two to an instruction: nothing diverges and no two lanes read different centres.  (Candidate lists per
// cell of a grid, read by vectors in any order, took three times as long an iteration for bank conflicts and divergence; lists built
// from a warp's common shortlist waited for the warps in the tails, whose shortlists were all E centres.)  A group that lay
// and still lies wholly with one centre is passed over; cluster sums change only by the vectors that moved.
// A tile is one block's, or a cluster of four sorts it together, deals its groups out and adds up all blocks' sums after an iteration (`LloydOf`).
// Bound by instructions (190 a group, iteration and warp; 55 % of the issue slots).  A block with 144 tiles, ten iterations: 281 us (283 with
// groups of 32 dealt out beforehand and the first members added up by one thread a group; seeds 93 us instead of 117).
constexpr int kCells = 64, kMoveQueue = 64, kGroupVec = 64, kListMax = 15;
template <int kBlocks>
struct LloydOf {
  static constexpr int kVec = kVqMaxVec / kBlocks, kThreads = kVec / 32, kWarps = kThreads / 32, kGroups = kVec / kGroupVec, kTurns = kGroups / kWarps;
  static constexpr int kRows = 256 / kBlocks;      // of the matrix
  static_assert(2 * kGroups == kThreads && kTurns <= 32, "two threads a group, a turn a lane");
};
constexpr uint32_t kListAll = 255u, kListSame = 0u;
// Vectors and their numbers as the sort leaves them, sent from all blocks; before that the cells' counts and the curve.
template <int kBlocks>
struct SortedVectors { uint2 both[LloydOf<kBlocks>::kVec]; };
template <>
struct SortedVectors<1> { uint32_t vec[kVqMaxVec]; uint16_t pos[kVqMaxVec]; };
template <int E, int kBlocks>
union LloydShared {
  using L = LloydOf<kBlocks>;
  struct {
    SortedVectors<kBlocks> to;
    uint32_t place[kCells * kCells / 2];          // next place of a cell, two to a word
    float red[2][L::kWarps], mean[2];
    int tot[L::kWarps];
  } sort;
  struct {
    uint32_t vec[L::kVec];                        // at last the indices in the order of the matrix, those of the whole tile
    uint8_t idx[L::kVec];                         // at last those of the block's rows
    uint4 list[L::kGroups];                       // up to fifteen candidates in ascending order, padded with the last one to an even number; last byte: their
                                                  // number, kListAll (more: take every centre), kListSame (nothing to do)
    double cx[E], cy[E];                          // centres
    float4 cf[E + 1];                             // x, y rounded to fp32; their squared length less a margin, and as it is; see cf_slot
    float4 neg[E];                                // -x, -x, -y, -y for the assignment
    ClusterSums<E> sums;                          // of the block's members
    uint32_t moves[L::kWarps][kMoveQueue];        // vector << 16 | old centre << 8 | new centre
    int moved, next[2];                           // group to be taken next, for every other iteration
    // a place of padding between the halves: the two threads of a group read different banks
    static __device__ __forceinline__ int cf_slot(int e) { return e + (e >= E / 2 ? 1 : 0); }
    __device__ __forceinline__ void set_centre(int e, float x, float y) {
      const float l = fmaf(x, x, y * y);
      cf[cf_slot(e)] = make_float4(x, y, l - 1e-5f * l, l);
      neg[e] = make_float4(-x, -x, -y, -y);
    }
    __device__ __forceinline__ float2 centre(int e) const { return *reinterpret_cast<const float2*>(cf + cf_slot(e)); }
  } it;
};
static_assert(3 * (sizeof(LloydShared<256, 4>) + 1024) <= 233472 && sizeof(LloydShared<256, 1>) <= 232448, "three blocks an SM, or one");

// Cell of a coordinate: eight per doubling of |x| + mean for the first two octaves, then four, so that a heavy-tailed tile is resolved as well as
// a Gaussian one.  Only the sorting order depends on it.
__device__ __forceinline__ int axis_cell(float x, float mean) {
  const uint32_t eighth = (__float_as_uint(fabsf(x) + mean) - __float_as_uint(mean)) >> 20;
  const int m = (int)min(min(eighth, (eighth >> 1) + kCells / 8), (uint32_t)(kCells / 2 - 1));
  return kCells / 2 + (m ^ ((int)__float_as_uint(x) >> 31));
}
// Position of cell (x, y) along the Hilbert curve of the 64 x 64 grid: quadrant by quadrant, each turned so that the curve joins up.
__device__ __forceinline__ int hilbert(int x, int y) {
  int d = 0;
#pragma unroll
  for (int s = kCells / 2; s > 0; s >>= 1) {
    const int rx = (x & s) != 0, ry = (y & s) != 0;
    d += s * s * ((3 * rx) ^ ry);
    if (!ry) {
      if (rx) { x = kCells - 1 - x; y = kCells - 1 - y; }
      const int t = x; x = y; y = t;
    }
  }
  return d;
}

// Box as middle and half extents, widened beyond the rounding of either.
struct Box {
  float mx, my, hx, hy;
  __device__ __forceinline__ void set(float x0, float x1, float y0, float y1) {
    mx = 0.5f * (x0 + x1); hx = 0.5005f * (x1 - x0) + 1e-6f * (fabsf(x0) + fabsf(x1));
    my = 0.5f * (y0 + y1); hy = 0.5005f * (y1 - y0) + 1e-6f * (fabsf(y0) + fabsf(y1));
  }
};

// The list of a group, by two neighbouring threads with half of the centres each (`half`: 0 or 1); they have the same box, `near` and
// `owner`.  `near`: a centre near the middle of the box (-1: to be looked for), the one that strikes others out;
// replaced by the nearest for the next time.  `owner`: the only centre of the group in the iteration before, -1 if it had
// several; `skip_same` writes kListSame where that has not changed.
//   |p - c|^2 - |p - b|^2 is linear in p: over the box its minimum is  |c|^2 - 2 m c - (|b|^2 - 2 m b) - 2 |c - b| h  per dimension,
// six operations a centre; what it has to exceed is a margin of 1e-5 (|c|^2 + |b|^2 + |m|^2 + |h|^2).
template <int EW, int kBlocks>
__device__ __forceinline__ void build_list(LloydShared<EW * 32, kBlocks>& sh, const Box& box, int group, int half, int& near, int& owner, bool skip_same) {
  auto& s = sh.it;
  constexpr int W = EW / 2;                      // words of a half
  const int first = half * W * 32;
  auto nearer_of_both = [&](float best, int at) -> int {
    const float other = __shfl_xor_sync(0xFFFFFFFFu, best, 1);
    const int other_at = __shfl_xor_sync(0xFFFFFFFFu, at, 1);
    return other < best || (other == best && other_at < at) ? other_at : at;
  };
  if (__any_sync(0xFFFFFFFFu, near < 0)) {
    float best = INFINITY;
    int at = first;
#pragma unroll 8
    for (int e = first; e < first + W * 32; ++e) {
      const float d = d2f(box.mx, box.my, s.centre(e));
      if (d < best) { best = d; at = e; }
    }
    at = nearer_of_both(best, at);
    if (near < 0) near = at;
  }
  const float4 b = s.cf[s.cf_slot(near)];
  const float mx2 = -2.f * box.mx, my2 = -2.f * box.my, hx2 = -2.f * box.hx, hy2 = -2.f * box.hy;
  const float limit = fmaf(mx2, b.x, fmaf(my2, b.y, b.w)) + 1e-5f * (b.w + box.mx * box.mx + box.my * box.my + box.hx * box.hx + box.hy * box.hy);
  uint32_t mask[W];
  int count = 0;
#pragma unroll
  for (int i = 0; i < W; ++i) {
    uint32_t m = 0u;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      const float4 c = s.cf[first + half + i * 32 + k];
      float t = fmaf(mx2, c.x, fmaf(my2, c.y, c.z));
      t = fmaf(hx2, fabsf(c.x - b.x), t);
      t = fmaf(hy2, fabsf(c.y - b.y), t);
      if (!(t > limit)) m |= 1u << k;
    }
    if (((near - first) >> 5) == i) m |= 1u << (near & 31);
    mask[i] = m;
    count += __popc(m);
  }
  const int others = __shfl_xor_sync(0xFFFFFFFFu, count, 1), all = count + others;
  uint8_t* list = reinterpret_cast<uint8_t*>(s.list + group);
  int now = -1;
  if (__any_sync(0xFFFFFFFFu, all <= kListMax)) {
    float best = INFINITY;
    int nearest = near, n = half ? others : 0, last = -1;
    if (all <= kListMax) {
#pragma unroll
      for (int i = 0; i < W; ++i)
        for (uint32_t m = mask[i]; m; m &= m - 1u) {
          last = first + i * 32 + __ffs((int)m) - 1;
          list[n++] = (uint8_t)last;
          const float d = d2f(box.mx, box.my, s.centre(last));
          if (d < best) { best = d; nearest = last; }
        }
    }
    nearest = nearer_of_both(best, nearest);
    last = max(last, __shfl_xor_sync(0xFFFFFFFFu, last, 1));
    if (all <= kListMax) {
      if ((all & 1) && half == 0) list[all] = (uint8_t)last;          // at fifteen: overwritten below, and over_list repeats the last one
      near = nearest;
      if (all == 1) now = last;
    } else {
      near = -1;
    }
  } else {
    near = -1;
  }
  __syncwarp();
  if (half == 0) list[15] = (uint8_t)(skip_same && now >= 0 && now == owner ? kListSame : all <= kListMax ? (uint32_t)all : kListAll);
  owner = now;
}

// take(a, b) over the list of a group, two candidates at a time.
template <int E, class F>
__device__ __forceinline__ void over_list(uint4 entry, F take) {
  const uint32_t n = entry.w >> 24;
  if (n != kListAll) {
    take(entry.x & 0xFFu, entry.x >> 8 & 0xFFu);
    if (n > 2u) take(entry.x >> 16 & 0xFFu, entry.x >> 24);
    if (n > 4u) take(entry.y & 0xFFu, entry.y >> 8 & 0xFFu);
    if (n > 6u) {
      take(entry.y >> 16 & 0xFFu, entry.y >> 24);
      if (n > 8u) take(entry.z & 0xFFu, entry.z >> 8 & 0xFFu);
      if (n > 10u) take(entry.z >> 16 & 0xFFu, entry.z >> 24);
      if (n > 12u) take(entry.w & 0xFFu, entry.w >> 8 & 0xFFu);
      if (n > 14u) take(entry.w >> 16 & 0xFFu, entry.w >> 16 & 0xFFu);
    }
  } else {
#pragma unroll 2
    for (uint32_t e = 0; e < (uint32_t)E; e += 2u) take(e, e + 1u);
  }
}

// The 64 indices of lane (g, t) of record `rec` of the tile as its little-endian bit stream.
template <int BITS>
__device__ __forceinline__ void vq_pack_lane(const uint8_t* idx, int rec, int g, int t, int L, uint8_t* out) {
  uint32_t words[2 * BITS + 1];
#pragma unroll
  for (int k = 0; k < 2 * BITS + 1; ++k) words[k] = 0u;
#pragma unroll
  for (int nn = 0; nn < 64; ++nn) {
    const int j = nn >> 2, R = nn & 3;
    const int row = rec * 16 + g + 8 * (R & 1);
    const int pair = 8 * j + 2 * t + (R >> 1);
    const uint32_t v = idx[row * 128 + pair];
    const int bitpos = BITS * nn, wi = bitpos >> 5, shft = bitpos & 31;
    words[wi] |= v << shft;
    if (shft + BITS > 32) words[wi + 1] |= v >> (32 - shft);
  }
#pragma unroll
  for (int p = 0; p < BITS / 2; ++p)
    *reinterpret_cast<uint4*>(out + p * 512 + L * 16) = make_uint4(words[4 * p], words[4 * p + 1], words[4 * p + 2], words[4 * p + 3]);
}

template <int EW, int kBlocks>
__global__ void __launch_bounds__(LloydOf<kBlocks>::kThreads, kBlocks == 1 ? 1 : 3) vq_lloyd_kernel(const VqArgs a, const __grid_constant__ rwkvq_image_header head, uint8_t* image) {
  extern __shared__ __align__(16) uint8_t smem[];
  using L = LloydOf<kBlocks>;
  constexpr int E = EW * 32, kThreads = L::kThreads, kVec = L::kVec;
  LloydShared<E, kBlocks>& sh = *reinterpret_cast<LloydShared<E, kBlocks>*>(smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t rank = cluster_rank();
  const int tile = blockIdx.x / kBlocks, tr = tile / a.TC, tc = tile % a.TC;
  asm volatile("griddepcontrol.launch_dependents;");      // the kernel of the seeds has seen the one before it end: weights and image may be touched
  if (blockIdx.x == 0) write_header(head, image);
  uint32_t pos[kVec / kThreads / 2];         // numbers of the vectors tid, tid + kThreads, ..., two to a word
  {
    constexpr int kRows = L::kRows / L::kWarps, kCounts = kCells * kCells / 2;
    uint32_t* const counts = reinterpret_cast<uint32_t*>(&sh.sort.to);      // of the cells, two to a word
    uint16_t* const curve = reinterpret_cast<uint16_t*>(counts + kCounts);
    uint4 q[kRows];
    const uint16_t* src = a.w + (size_t)(tr * 256 + (int)rank * L::kRows) * a.ic + tc * 256;
#pragma unroll
    for (int j = 0; j < kRows; ++j) q[j] = __ldg(reinterpret_cast<const uint4*>(src + (size_t)(warp + j * L::kWarps) * a.ic) + lane);
    float ax = 0.f, ay = 0.f;
#pragma unroll
    for (int j = 0; j < kRows; ++j) {
      const float2 f0 = vec_of(q[j].x), f1 = vec_of(q[j].y), f2 = vec_of(q[j].z), f3 = vec_of(q[j].w);
      ax += fabsf(f0.x) + fabsf(f1.x) + fabsf(f2.x) + fabsf(f3.x);
      ay += fabsf(f0.y) + fabsf(f1.y) + fabsf(f2.y) + fabsf(f3.y);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) { ax += __shfl_xor_sync(0xFFFFFFFFu, ax, off); ay += __shfl_xor_sync(0xFFFFFFFFu, ay, off); }
    if (lane == 0) { sh.sort.red[0][warp] = ax; sh.sort.red[1][warp] = ay; }
    for (int i = tid; i < kCounts; i += kThreads) counts[i] = 0u;
    for (int i = tid; i < kCells * kCells; i += kThreads) curve[i] = (uint16_t)hilbert(i % kCells, i / kCells);
    __syncthreads();
    if (tid < 2) {
      float sum = 0.f;
      for (int w = 0; w < L::kWarps; ++w) sum += sh.sort.red[tid][w];
      sh.sort.mean[tid] = sum;
    }
    cluster_arrive();
    cluster_wait();
    ax = ay = 0.f;
#pragma unroll
    for (uint32_t r = 0; r < kBlocks; ++r) {
      ax += __uint_as_float(peer_load(peer_address(shared_address(&sh.sort.mean[0]), r)));
      ay += __uint_as_float(peer_load(peer_address(shared_address(&sh.sort.mean[1]), r)));
    }
    ax = ax > 1e-25f && ax < 1e25f ? ax * (1.f / kVqMaxVec) : 1.f;
    ay = ay > 1e-25f && ay < 1e25f ? ay * (1.f / kVqMaxVec) : 1.f;
    auto cell_of = [&](uint32_t v) -> uint32_t {
      const float2 f = vec_of(v);
      return curve[axis_cell(f.y, ay) * kCells + axis_cell(f.x, ax)];
    };
    uint32_t cells[kRows][2];                         // of a row's four vectors, two to a word
#pragma unroll
    for (int j = 0; j < kRows; ++j) {
      cells[j][0] = cell_of(q[j].x) | cell_of(q[j].y) << 16;
      cells[j][1] = cell_of(q[j].z) | cell_of(q[j].w) << 16;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t c = (cells[j][k / 2] >> (16 * (k & 1))) & 0xFFFFu;
        atomicAdd(counts + (c >> 1), c & 1u ? 0x10000u : 1u);      // 32 768 at most: no carry into the other half
      }
    }
    cluster_arrive();
    cluster_wait();
    {
      // a thread's cells: their counts in all blocks, and in the blocks in front
      constexpr int kPer = kCounts / kThreads;
      static_assert(kPer % 2 == 0, "cells per thread");
      uint32_t all[kPer], front[kPer];
#pragma unroll
      for (int i = 0; i < kPer; ++i) all[i] = front[i] = 0u;
#pragma unroll
      for (uint32_t r = 0; r < kBlocks; ++r) {
        const uint32_t at = peer_address(shared_address(counts + tid * kPer), r);
        uint32_t c[kPer];
        if constexpr (kPer % 4 == 0) {
#pragma unroll
          for (int i = 0; i < kPer; i += 4) {
            const uint4 v = peer_load4(at + 4 * i);
            c[i] = v.x; c[i + 1] = v.y; c[i + 2] = v.z; c[i + 3] = v.w;
          }
        } else {
#pragma unroll
          for (int i = 0; i < kPer; ++i) c[i] = peer_load(at + 4 * i);
        }
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
          if (r < rank) front[i] += c[i];
          all[i] += c[i];
        }
      }
      int sum = 0;
#pragma unroll
      for (int i = 0; i < kPer; ++i) sum += (int)(all[i] & 0xFFFFu) + (int)(all[i] >> 16);
      int incl = sum;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int v = __shfl_up_sync(0xFFFFFFFFu, incl, off);
        if (lane >= off) incl += v;
      }
      if (lane == 31) sh.sort.tot[warp] = incl;
      __syncthreads();
      int at = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? sh.sort.tot[lane] : 0) + incl - sum;
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        const int lo = (int)(all[i] & 0xFFFFu), hi = (int)(all[i] >> 16);
        sh.sort.place[tid * kPer + i] = (uint32_t)at + (uint32_t)(at + lo) * 0x10000u + front[i];
        at += lo + hi;
      }
    }
    cluster_arrive();                                 // the counts have been read, the curve has been used: their place may be written
    cluster_wait();
#pragma unroll
    for (int j = 0; j < kRows; ++j) {
      const uint32_t v[4] = {q[j].x, q[j].y, q[j].z, q[j].w};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t c = (cells[j][k / 2] >> (16 * (k & 1))) & 0xFFFFu;
        const uint32_t old = atomicAdd(sh.sort.place + (c >> 1), c & 1u ? 0x10000u : 1u);      // the order within a cell does not matter: sums are exact
        const uint32_t p = c & 1u ? old >> 16 : old & 0xFFFFu, number = (uint32_t)(((int)rank * L::kRows + warp + j * L::kWarps) * 128 + lane * 4 + k);
        if constexpr (kBlocks == 1) {
          sh.sort.to.vec[p] = v[k];
          sh.sort.to.pos[p] = (uint16_t)number;
        } else {
          // the groups go to the blocks in turn: their lists are longest at either end of the curve
          const uint32_t group = p / kGroupVec;
          peer_store(peer_address(shared_address(sh.sort.to.both + group / kBlocks * kGroupVec + p % kGroupVec), group % kBlocks), v[k], number);
        }
      }
    }
    cluster_arrive();
    cluster_wait();
    // `vec` lies over the first half of `both`
    constexpr int kStep = 8;
#pragma unroll
    for (int i0 = 0; i0 < kVec / kThreads; i0 += kStep) {
      uint2 t[kStep];
#pragma unroll
      for (int i = 0; i < kStep; ++i) {
        if constexpr (kBlocks == 1) t[i].y = sh.sort.to.pos[(i0 + i) * kThreads + tid];
        else t[i] = sh.sort.to.both[(i0 + i) * kThreads + tid];
      }
      if (kBlocks > 1) __syncthreads();
#pragma unroll
      for (int i = 0; i < kStep; ++i) {
        if (kBlocks > 1) sh.it.vec[(i0 + i) * kThreads + tid] = t[i].x;
        if (i & 1) pos[(i0 + i) / 2] |= t[i].y << 16; else pos[(i0 + i) / 2] = t[i].y;
      }
    }
    __syncthreads();
  }
  const int my_group = tid >> 1, my_half = tid & 1;
  Box box;                                       // of this thread's group
  {
    float x0 = INFINITY, x1 = -INFINITY, y0 = INFINITY, y1 = -INFINITY;
#pragma unroll 8
    for (int k = 0; k < 32; ++k) {
      const float2 f = vec_of(sh.it.vec[tid * 32 + ((k + lane) & 31)]);
      x0 = fminf(x0, f.x); x1 = fmaxf(x1, f.x); y0 = fminf(y0, f.y); y1 = fmaxf(y1, f.y);
    }
    x0 = fminf(x0, __shfl_xor_sync(0xFFFFFFFFu, x0, 1)); x1 = fmaxf(x1, __shfl_xor_sync(0xFFFFFFFFu, x1, 1));
    y0 = fminf(y0, __shfl_xor_sync(0xFFFFFFFFu, y0, 1)); y1 = fmaxf(y1, __shfl_xor_sync(0xFFFFFFFFu, y1, 1));
    box.set(x0, x1, y0, y1);
  }
  uint32_t* aux = a.aux + (size_t)tile * E;
  auto& s = sh.it;
  asm volatile("griddepcontrol.wait;" ::: "memory");      // the seeds
  for (int e = tid; e < E; e += kThreads) {
#pragma unroll
    for (int p = 0; p < 3; ++p) s.sums.x[p][e] = s.sums.y[p][e] = 0;
    s.sums.cnt[e] = 0;
    const float2 c = vec_of(__ldcg(aux + e));
    s.cx[e] = (double)c.x; s.cy[e] = (double)c.y;
    s.set_centre(e, c.x, c.y);
  }
  if (tid == 0) s.moved = s.next[0] = s.next[1] = 0;
  __syncthreads();
  int near = -1, owner = -1;
  for (int it = 0; it < a.iters; ++it) {
    build_list<EW, kBlocks>(sh, box, my_group, my_half, near, owner, it > 0);
    __syncthreads();
    if (it > 0) cluster_wait();                  // the sums have been read
    bool moved = it == 0;
    int queued = 0;                              // moves of this warp not yet in the sums
    uint32_t* queue = s.moves[warp];
    auto flush = [&](int count) {
      __syncwarp();
      if (lane < count) {
        const uint32_t m = queue[lane];
        const uint32_t v = s.vec[m >> 16];
        move_member(s.sums, v, (int)((m >> 8) & 0xFFu), (int)(m & 0xFFu));
      }
      __syncwarp();
    };
    // the vectors that moved are queued and taken 32 at a time: a few lanes of every warp would otherwise walk
    // the whole update for every group
    auto move = [&](int p, uint32_t was, uint32_t now) {
      const uint32_t who = __ballot_sync(0xFFFFFFFFu, now != was);
      if (who == 0u) return;
      moved = true;
      if (now != was) {
        s.idx[p] = (uint8_t)now;
        queue[queued + __popc(who & ((1u << lane) - 1u))] = (uint32_t)p << 16 | was << 8 | now;
      }
      queued += __popc(who);
      if (queued >= 32) {
        flush(32);
        queued -= 32;
        const uint32_t m = queue[32 + lane];
        __syncwarp();
        if (lane < queued) queue[lane] = m;
      }
    };
    // a warp takes the next group when it is done with one: their lists differ
    auto take = [&]() -> int { return lane == 0 ? atomicAdd(&s.next[it & 1], 1) : 0; };
    int ahead = take();
    for (;;) {
      const int g = __shfl_sync(0xFFFFFFFFu, ahead, 0), p = g * kGroupVec + lane;
      if (g >= L::kGroups) break;
      ahead = take();
      const uint4 entry = s.list[g];
      if ((entry.w >> 24) == kListSame) continue;
      const uint32_t v0 = s.vec[p], v1 = s.vec[p + 32];
      const float2 f0 = vec_of(v0), f1 = vec_of(v1);
      const float2 x = make_float2(f0.x, f1.x), y = make_float2(f0.y, f1.y);
      float best0 = INFINITY, best1 = INFINITY;
      uint32_t at0 = 0u, at1 = 0u;
      auto compare = [&](uint32_t e) {
        const float4 c = s.neg[e];
        const float2 dx = add2(x, make_float2(c.x, c.y)), dy = add2(y, make_float2(c.z, c.w)), d = fma2(dx, dx, mul2(dy, dy));
        if (d.x < best0) { best0 = d.x; at0 = e; }
        if (d.y < best1) { best1 = d.y; at1 = e; }
      };
      over_list<E>(entry, [&](uint32_t e0, uint32_t e1) { compare(e0); compare(e1); });
      uint32_t was0, was1;
      if (it == 0) {
        // all join the centre of one of them, and most others' centres: the rest moves on
        const uint32_t a8 = __shfl_sync(0xFFFFFFFFu, at0, 8), a24 = __shfl_sync(0xFFFFFFFFu, at1, 24);
        const int n8 = __popc(__ballot_sync(0xFFFFFFFFu, at0 == a8)) + __popc(__ballot_sync(0xFFFFFFFFu, at1 == a8));
        const int n24 = __popc(__ballot_sync(0xFFFFFFFFu, at0 == a24)) + __popc(__ballot_sync(0xFFFFFFFFu, at1 == a24));
        was0 = was1 = n8 >= n24 ? a8 : a24;
        s.idx[p] = s.idx[p + 32] = (uint8_t)was0;
        join_group(s.sums, v0, v1, (int)was0);
      } else {
        was0 = s.idx[p]; was1 = s.idx[p + 32];
      }
      move(p, was0, at0);
      move(p + 32, was1, at1);
    }
    flush(queued);
    if (tid == 0) s.next[(it + 1) & 1] = 0;
    if (moved && lane == 0) s.moved = it + 1;
    cluster_arrive();
    cluster_wait();
    bool any = false;
#pragma unroll
    for (uint32_t r = 0; r < kBlocks; ++r) any |= (int)peer_load(peer_address(shared_address(&s.moved), r)) == it + 1;
    if (any) {
      // four neighbouring lanes a centre, one for each block's sums
#pragma unroll
      for (int k = tid; k < kBlocks * E; k += kThreads) {
        const int e = k / kBlocks;
        const uint32_t from = (uint32_t)(k % kBlocks);
        int v[7];
#pragma unroll
        for (int p = 0; p < 3; ++p) {
          v[p] = (int)peer_load(peer_address(shared_address(&s.sums.x[p][e]), from));
          v[3 + p] = (int)peer_load(peer_address(shared_address(&s.sums.y[p][e]), from));
        }
        v[6] = (int)peer_load(peer_address(shared_address(&s.sums.cnt[e]), from));
#pragma unroll
        for (int p = 0; p < 7; ++p) {
#pragma unroll
          for (int off = 1; off < kBlocks; off <<= 1) v[p] += __shfl_xor_sync(0xFFFFFFFFu, v[p], off);
        }
        if (from == 0u && v[6]) {
          const double x = mean_of_pieces(v[0], v[1], v[2], v[6]), y = mean_of_pieces(v[3], v[4], v[5], v[6]);
          s.cx[e] = x; s.cy[e] = y;
          s.set_centre(e, (float)x, (float)y);
        }
      }
    }
    cluster_arrive();
    if (!any) {                                  // the centres would stay as they are in every further iteration
      cluster_wait();
      break;
    }
    if (it + 1 == a.iters) cluster_wait();
    __syncthreads();
  }
  // ---- centres to fp16; final assignment against the rounded centres in fp64 (exact differences,
  // products and sum each rounded once, in this order; the lowest index wins ties)
  for (int e = tid; e < E; e += kThreads) {
    const __half hx = __double2half(s.cx[e]), hy = __double2half(s.cy[e]);
    s.cx[e] = (double)__half2float(hx); s.cy[e] = (double)__half2float(hy);
    s.set_centre(e, __half2float(hx), __half2float(hy));
    if (rank == 0u) aux[e] = (uint32_t)__half_as_ushort(hx) | ((uint32_t)__half_as_ushort(hy) << 16);
  }
  __syncthreads();
  build_list<EW, kBlocks>(sh, box, my_group, my_half, near, owner, false);
  __syncthreads();
  // In fp32 first: a distance is wrong by less than seven roundings there, so a centre whose distance is smallest by more than 2^-20 of it is
  // the nearest in fp64 too, and so is one that the vector equals.  The others (and distances near the end of fp32's range) are taken in fp64.
  for (int g = warp; g < L::kGroups; g += L::kWarps) {
    const uint4 entry = s.list[g];
    const int p = g * kGroupVec + lane;
    const float2 f[2] = {vec_of(s.vec[p]), vec_of(s.vec[p + 32])};
    const float2 x = make_float2(f[0].x, f[1].x), y = make_float2(f[0].y, f[1].y);
    float best[2] = {INFINITY, INFINITY}, next[2] = {INFINITY, INFINITY};
    uint32_t at[2] = {entry.x & 0xFFu, entry.x & 0xFFu}, last = kListAll + 1u;
    if ((entry.w >> 24) != 1u) {
      auto compare = [&](uint32_t e) {
        if (e == last) return;                   // the padding of a list is no second centre
        last = e;
        const float4 c = s.neg[e];
        const float2 dx = add2(x, make_float2(c.x, c.y)), dy = add2(y, make_float2(c.z, c.w)), d = fma2(dx, dx, mul2(dy, dy));
        next[0] = fminf(next[0], fmaxf(best[0], d.x)); next[1] = fminf(next[1], fmaxf(best[1], d.y));
        if (d.x < best[0]) { best[0] = d.x; at[0] = e; }
        if (d.y < best[1]) { best[1] = d.y; at[1] = e; }
      };
      over_list<E>(entry, [&](uint32_t e0, uint32_t e1) { compare(e0); compare(e1); });
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const float4 c = s.neg[at[k]];
        const bool equal = f[k].x + c.x == 0.f && f[k].y + c.z == 0.f;
        if (next[k] > best[k] * (1.f + 1.f / 1048576.f) && (equal || (best[k] > 1e-30f && best[k] < 1e30f))) continue;
        const double dx = (double)f[k].x, dy = (double)f[k].y;
        double nearest = INFINITY;
        over_list<E>(entry, [&](uint32_t e0, uint32_t e1) {
          const double dx0 = dx - s.cx[e0], dy0 = dy - s.cy[e0], dx1 = dx - s.cx[e1], dy1 = dy - s.cy[e1];
          const double d0 = __dadd_rn(__dmul_rn(dx0, dx0), __dmul_rn(dy0, dy0)), d1 = __dadd_rn(__dmul_rn(dx1, dx1), __dmul_rn(dy1, dy1));
          if (d0 < nearest) { nearest = d0; at[k] = e0; }
          if (d1 < nearest) { nearest = d1; at[k] = e1; }
        });
      }
    }
    s.idx[p] = (uint8_t)at[0]; s.idx[p + 32] = (uint8_t)at[1];
  }
  __syncthreads();
  // back to the order of the matrix; the vectors are not needed any more.  A block writes its indices into an empty tile, and takes its rows
  // of all blocks' tiles.  (Bytes stored to the block that has the row took 16 000 cycles instead of 8 000.)
  uint8_t* const tile_idx = reinterpret_cast<uint8_t*>(s.vec);
  if (kBlocks > 1) {
#pragma unroll
    for (int i = 0; i < kVqMaxVec / 16 / kThreads; ++i) reinterpret_cast<uint4*>(tile_idx)[i * kThreads + tid] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < kVec / kThreads; ++i) tile_idx[(pos[i / 2] >> (16 * (i & 1))) & 0xFFFFu] = s.idx[i * kThreads + tid];
  if constexpr (kBlocks > 1) {
    cluster_arrive();
    cluster_wait();
#pragma unroll
    for (int i = 0; i < kVec / 16 / kThreads; ++i) {
      const int at = i * kThreads + tid;
      uint4 all = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
      for (uint32_t r = 0; r < kBlocks; ++r) {
        const uint4 v = peer_load4(peer_address(shared_address(tile_idx + rank * kVec + at * 16), r));
        all.x |= v.x; all.y |= v.y; all.z |= v.z; all.w |= v.w;
      }
      reinterpret_cast<uint4*>(s.idx)[at] = all;
    }
    cluster_arrive();                            // the others have read this block's tile
  }
  __syncthreads();
  // ---- bit packing (format.h)
  constexpr int kRecords = 16 / kBlocks;
  if (warp < kRecords) {
    const int gr = lane >> 2, t = lane & 3, rec = (int)rank * kRecords + warp;
    constexpr int kBits = EW == 2 ? 6 : 8;
    const int mb = tr * 2 + (rec >> 3), rt = rec & 7;
    uint8_t* out = a.payload + (((size_t)mb * a.TC + tc) * 8 + rt) * rwkvq_vq_record_bytes(kBits);
    vq_pack_lane<kBits>(kBlocks > 1 ? s.idx : tile_idx, warp, gr, t, lane, out);
  }
  if (kBlocks > 1) cluster_wait();
}

// ---- token-shift vectors ----
//
// One cluster a call.  Every block draws all the seeds (up to kVecSeeds vectors: sixteen a thread in registers; a longer vector is
// seeded by vq_seed_kernel) and then keeps a part of the vectors.  An iteration: four lanes a vector, each against a quarter of the
// centres; the members of a centre become bit masks, from which four sums a centre (of w * v and of w in either dimension; exact integers
// without weights) are added in a fixed order; every block sends its sums to the block that has the centre, which adds up those of all blocks and sends
// the new centre to all.  (Every block sending its sums to all saved that second trip, and took longer for the bytes.)  Bound by latency: two barriers
// a draw (0.42 us), two barriers and two trips through the cluster an iteration (1.65 us).  2048 weighted vectors, 64 centres, ten iterations:
// 47.6 us; 139 with one warp drawing all seeds by the chains, one block sorting the members by centre and adding them up, and a barrier of the
// cluster at either end of it.  256 centres, 2560 vectors: 166 us, 418 then.
constexpr int kVecThreads = 512;
constexpr int kVecCluster = 16;                  // blocks
constexpr int kSeedPer = 16, kVecSeeds = 4096, kSeedWarps = kVecSeeds / (32 * kSeedPer);
constexpr int kVecParts = 4;                     // lanes a vector
constexpr int kVecRound = kVecThreads / kVecParts;      // vectors a block compares at a time
constexpr int kVecGroups = 32;                   // groups of 32 vectors whose members a block adds up at a time
// The search for the nearest centre takes the minimum over groups of eight centres, less than one instruction a distance, and looks for the
// centre only in the group that wins.
constexpr int kCentreGroup = 8;
struct VecSeeds {
  float tot[kSeedWarps], run_tot[kVecSeeds / 2048];
  float u01[kVqMaxE];
  int pick[kVqMaxE];                             // -1: not decided
  float dist[kVecSeeds / 64 * 65];               // runs of 64, each in banks of its own
  __align__(16) uint32_t vec[kVecSeeds];
};
constexpr int kGroupSlots = kCentreGroup / 2 + 1;      // one of padding: lanes that look in different groups read different banks
template <int E>
struct VecShared {
  double c[2][E];                                // centres
  float4 neg[E / kCentreGroup * kGroupSlots];    // (-x, -x', -y, -y') of two neighbouring centres, rounded to fp32, in groups
  uint64_t sums_here, centres_here;              // barriers of what the other blocks send
  double sent[E][2];                             // centres, from the block that has them
  ulonglong2 part[kVecCluster][E / kVecCluster][2];    // (of w * v, of w) of this block's centres in either dimension, from every block
  uint32_t seed[E];
  __align__(16) uint32_t mask[2][E][kVecGroups + 4];   // members of a centre in each group of 32; one is cleared while the other is filled
  uint8_t idx[kVqMaxVec / kVecCluster];
  VecSeeds s;
  ulonglong2 table[kVecGroups * 32][2];          // (w * v, w) in either dimension of the block's vectors, if there are no more
};
static_assert(sizeof(VecShared<256>) <= 232448, "shared memory of a block");

// Draws E seeds; a draw is defined as in vq_seed_kernel: distances summed in fp32 over runs of 64 vectors in order, run sums by a scan over the lanes
// of a warp, and the last vector whose running sum begins at or below the target.  Those chains are 64 additions long, twice a draw.  So the
// sums are taken in a tree first: with u = 2^-24, the chains' running sums are off by at most 148 u of themselves and their target by 84 u, the
// tree's by 23 u and 20 u (its differences from the target by three more), and the sum in front of a thread, the scan less the thread's own sum, by five u of
// the scan besides, which may be thousands of times the target.  So a vector whose running sums begin and end at least 320 u of the target and 8 u of the
// scan away from the target (and on either side) is the one that the chains give.  Otherwise (one draw in 25 for 2048 vectors) the chains are
// walked.  (The sum in front by a shuffle from the neighbour needs no second term, and took 2 us longer for a vector of 4096.)
// Called by the first `threads` threads, which hold sixteen vectors each.
__device__ __forceinline__ void draw_seeds(VecSeeds& sh, uint32_t* seeds, int n, int E, uint64_t seed, int threads) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, base = kSeedPer * tid;
  auto sync = [&]() { asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory"); };
  float2 x[kSeedPer / 2], y[kSeedPer / 2];
  float dist[kSeedPer];
#pragma unroll
  for (int k = 0; k < kSeedPer; k += 4) {
    const uint4 q = *reinterpret_cast<const uint4*>(sh.vec + base + k);
    const float2 a = vec_of(q.x), b = vec_of(q.y), c = vec_of(q.z), d = vec_of(q.w);
    x[k / 2] = make_float2(a.x, b.x); x[k / 2 + 1] = make_float2(c.x, d.x);
    y[k / 2] = make_float2(a.y, b.y); y[k / 2 + 1] = make_float2(c.y, d.y);
  }
#pragma unroll
  for (int k = 0; k < kSeedPer; ++k) dist[k] = base + k < n ? INFINITY : 0.f;
  uint32_t cv = sh.vec[below(splitmix(seed, 0), n)];
  for (int e = 0;; ++e) {
    if (tid == 0) seeds[e] = cv;
    if (e + 1 == E) break;
    const float u01 = sh.u01[e + 1];
    const float2 c = vec_of(cv);
    const float2 ncx = make_float2(-c.x, -c.x), ncy = make_float2(-c.y, -c.y);
#pragma unroll
    for (int k = 0; k < kSeedPer / 2; ++k) {
      const float2 dx = add2(x[k], ncx), dy = add2(y[k], ncy), d = fma2(dx, dx, mul2(dy, dy));
      dist[2 * k] = fminf(dist[2 * k], d.x); dist[2 * k + 1] = fminf(dist[2 * k + 1], d.y);
    }
    float sum[kSeedPer + 1];                       // sum[k]: of the first k
    sum[0] = 0.f;
    {
      float two[kSeedPer / 2], four[kSeedPer / 4];
#pragma unroll
      for (int k = 0; k < kSeedPer / 2; ++k) two[k] = dist[2 * k] + dist[2 * k + 1];
#pragma unroll
      for (int k = 0; k < kSeedPer / 4; ++k) four[k] = two[2 * k] + two[2 * k + 1];
      sum[4] = four[0]; sum[8] = four[0] + four[1]; sum[16] = sum[8] + (four[2] + four[3]); sum[12] = sum[8] + four[2];
#pragma unroll
      for (int k = 0; k < kSeedPer; k += 4) {
        sum[k + 1] = sum[k] + dist[k];
        sum[k + 2] = sum[k] + two[k / 2];
        sum[k + 3] = sum[k + 2] + dist[k + 2];
      }
      static_assert(kSeedPer == 16, "sums of a thread");
    }
    float incl = sum[kSeedPer];
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const float v = __shfl_up_sync(0xFFFFFFFFu, incl, off);
      if (lane >= off) incl += v;
    }
    if (lane == 31) sh.tot[warp] = incl;
    sync();
    float t[kSeedWarps];                           // zeros behind the last warp
#pragma unroll
    for (int w = 0; w < kSeedWarps; w += 4) {
      const float4 t4 = *reinterpret_cast<const float4*>(sh.tot + w);
      t[w] = t4.x; t[w + 1] = t4.y; t[w + 2] = t4.z; t[w + 3] = t4.w;
    }
    float before[kSeedWarps];
#pragma unroll
    for (int w = 0; w < kSeedWarps; ++w) before[w] = w < warp ? t[w] : 0.f;
#pragma unroll
    for (int h = kSeedWarps / 2; h > 0; h >>= 1)
#pragma unroll
      for (int w = 0; w < h; ++w) { t[w] += t[w + h]; before[w] += before[w + h]; }
    const float target = u01 * t[0], margin = fmaf(incl, 8.f / 16777216.f, target * (320.f / 16777216.f));
    const float rest = target - (before[0] + (incl - sum[kSeedPer]));
    const float under = rest - margin, over = rest + margin;
    if (sum[0] <= under && sum[kSeedPer] > over) {
      // the last that begins at or below, by halves
      int at = base;
      float win[kSeedPer + 1];
#pragma unroll
      for (int k = 0; k <= kSeedPer; ++k) win[k] = sum[k];
#pragma unroll
      for (int h = kSeedPer / 2; h > 0; h >>= 1) {
        const bool upper = win[h] <= under;
        at += upper ? h : 0;
#pragma unroll
        for (int k = 0; k <= h; ++k) win[k] = upper ? win[k + h] : win[k];
      }
      if (win[1] > over) sh.pick[e + 1] = at;
    }
    sync();
    const int pick = sh.pick[e + 1];
    cv = sh.vec[max(pick, 0)];
    if (pick >= 0) continue;
    // the chains; thread t < n / 64 has run t
#pragma unroll
    for (int k = 0; k < kSeedPer; ++k) sh.dist[base + k + (base >> 6)] = dist[k];
    sync();
    const int runs = (n + 2047) / 2048 * 32;
    const float* run = sh.dist + 65 * tid;
    const bool holds = tid < runs && 64 * tid < kSeedPer * threads;        // `threads` is a multiple of 32: whole runs
    float excl = 0.f;
    if (tid < runs) {
      float chain = 0.f;
      if (holds) {
#pragma unroll 16
        for (int k = 0; k < 64; ++k) chain += run[k];
      }
      incl = chain;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const float v = __shfl_up_sync(0xFFFFFFFFu, incl, off);
        if (lane >= off) incl += v;
      }
      if (lane == 31) sh.run_tot[warp] = incl;
      excl = __shfl_up_sync(0xFFFFFFFFu, incl, 1);
      if (lane == 0) excl = 0.f;
    }
    if (tid == 0) sh.pick[e + 1] = n - 1;
    sync();
    const float first = warp == 1 ? sh.run_tot[0] : 0.f, total = sh.run_tot[0] + (runs > 32 ? sh.run_tot[1] : 0.f);
    excl = first + excl;
    incl = first + incl;
    if (!(total > 0.f)) {
      if (tid == 0) sh.pick[e + 1] = below(splitmix(seed, e + 1), n);
    } else if (holds && excl <= u01 * total && u01 * total < incl) {
      int last = 64 * tid;
#pragma unroll 16
      for (int k = 0; k < 64; ++k) {
        if (excl <= u01 * total && 64 * tid + k < n) last = 64 * tid + k;
        excl += run[k];
      }
      sh.pick[e + 1] = last;
    }
    sync();
    cv = sh.vec[sh.pick[e + 1]];
  }
}

// Distances of a vector to two centres, each rounded as d = w.x * (dx * dx) + (w.y * (dy * dy)) with the last product and sum in one
// rounding (unweighted: dx * dx + (dy * dy), likewise).
template <bool kWeighted>
__device__ __forceinline__ float2 pair_distance(float2 f, float2 w, float4 c) {
  const float2 dx = add2(make_float2(f.x, f.x), make_float2(c.x, c.y)), dy = add2(make_float2(f.y, f.y), make_float2(c.z, c.w)), yy = mul2(dy, dy);
  return kWeighted ? fma2(make_float2(w.x, w.x), mul2(dx, dx), mul2(make_float2(w.y, w.y), yy)) : fma2(dx, dx, yy);
}

__device__ __forceinline__ constexpr int neg_slot(int e) { return e / kCentreGroup * kGroupSlots + e % kCentreGroup / 2; }
template <class T> struct alignas(16) VecSums { T wv, w; };
template <int E, bool kWeighted>
__global__ void __launch_bounds__(kVecThreads, 1) vq_vector_kernel(const VqArgs a, const __grid_constant__ rwkvq_image_header head, uint8_t* image) {
  extern __shared__ __align__(16) uint8_t smem[];
  VecShared<E>& sh = *reinterpret_cast<VecShared<E>*>(smem);
  using Sums = VecSums<typename std::conditional<kWeighted, double, long long>::type>;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = a.n_vec;
  const uint32_t* vec = reinterpret_cast<const uint32_t*>(a.w);
  const float2* wgt = reinterpret_cast<const float2*>(a.elem_w);
  const uint32_t rank = cluster_rank();
  const bool lead = rank == 0u;
  if (n <= kVecSeeds) asm volatile("griddepcontrol.wait;" ::: "memory");      // else the kernel of the seeds has waited
  asm volatile("griddepcontrol.launch_dependents;");
  if (lead) write_header(head, image);
  // this block's vectors: [begin, begin + 32 * groups), those below n
  const int groups = (n + 32 * kVecCluster - 1) / (32 * kVecCluster), begin = (int)rank * groups * 32;
  const int pass_groups = min(groups, kVecGroups);
  const bool one_pass = groups <= kVecGroups;
  const uint32_t sums_here = shared_address(&sh.sums_here), centres_here = shared_address(&sh.centres_here);
  // summands of vector i in one dimension
  auto summands = [&](int i, int dim) -> Sums {
    const uint32_t v = a.w[2 * i + dim];
    if constexpr (kWeighted) {
      const double w = (double)__ldcg(a.elem_w + 2 * i + dim);        // written by the kernel before, which this one need not have started behind
      return Sums{w * (double)h2f_bits(v), w};                     // the product of 24 and 11 bits is exact
    } else {
      return Sums{half_fixed(v), 1};
    }
  };
  Sums* const table = reinterpret_cast<Sums*>(sh.table);
  if (one_pass)
    for (int k = tid; k < groups * 64; k += kVecThreads)
      if (begin + (k >> 1) < n) table[k] = summands(begin + (k >> 1), k & 1);
  // neighbouring lanes compare one vector
  const int in_four = lane & (kVecParts - 1), in_round = warp * (32 / kVecParts) + lane / kVecParts;
  float2 f, w = make_float2(1.f, 1.f);
  auto fetch = [&](int i0) {
    const int i = min(i0 + in_round, n - 1);
    f = vec_of(vec[i]);
    if (kWeighted) w = __ldcg(wgt + i);
  };
  fetch(begin);
  if (tid == 0)
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n mbarrier.init.shared::cta.b64 [%1], 1;\n fence.mbarrier_init.release.cluster;" ::"r"(sums_here), "r"(centres_here) : "memory");
  if (n <= kVecSeeds) {
    const int warps = (n + 32 * kSeedPer - 1) / (32 * kSeedPer);
    bool bad = false;
    for (int i = tid; i < warps * 32 * kSeedPer; i += kVecThreads) {
      const uint32_t v = i < n ? __ldcg(vec + i) : 0u;
      bad |= ((v & 0x7C00u) == 0x7C00u) | ((v & 0x7C000000u) == 0x7C000000u);
      sh.s.vec[i] = v;
    }
    if (bad && lead) atomicOr(a.flags, kFlagNonFinite);
    if (tid < kSeedWarps) sh.s.tot[tid] = 0.f;
    if (tid < E) { sh.s.u01[tid] = (float)unit_of(splitmix(a.seed, tid)); sh.s.pick[tid] = -1; }
    __syncthreads();
    if (warp < warps) draw_seeds(sh.s, sh.seed, n, E, a.seed, 32 * warps);
  } else {
    // the seeds lie where the codebook will
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (tid < E) sh.seed[tid] = __ldcg(a.aux + tid);
  }
  __syncthreads();
  auto set_centre = [&](int e, int dim, double c) {
    sh.c[dim][e] = c;
    reinterpret_cast<float*>(sh.neg + neg_slot(e))[2 * dim + (e & 1)] = -(float)c;
  };
  if (tid < 2 * E) set_centre(tid >> 1, tid & 1, (double)h2f_bits((sh.seed[tid >> 1] >> (16 * (tid & 1))) & 0xFFFFu));
  auto clear_masks = [&](int which) {
    for (int k = tid; k < E * 8; k += kVecThreads) *reinterpret_cast<uint4*>(&sh.mask[which][k >> 3][4 * (k & 7)]) = make_uint4(0u, 0u, 0u, 0u);
  };
  clear_masks(0);
  cluster_arrive();                                // every block runs and has its seeds: sums may be sent
  cluster_wait();
  // The nearest centre of this lane's vector, the first of equally near ones, known to all four lanes.  `alone`: no other centre is within 2^-20
  // of its distance, which is `best`.
  auto nearest = [&](float& best, bool* alone) -> int {
    int group = 0;
    best = INFINITY;
    float next = INFINITY;                         // smallest minimum of another group
#pragma unroll 2
    for (int g = in_four; g < E / kCentreGroup; g += kVecParts) {
      float d[kCentreGroup];
#pragma unroll
      for (int k = 0; k < kCentreGroup / 2; ++k) {
        const float2 two = pair_distance<kWeighted>(f, w, sh.neg[g * kGroupSlots + k]);
        d[2 * k] = two.x; d[2 * k + 1] = two.y;
      }
      const float m = fminf(fminf(fminf(d[0], d[1]), fminf(d[2], d[3])), fminf(fminf(d[4], d[5]), fminf(d[6], d[7])));
      if (alone) next = fminf(next, fmaxf(best, m));
      if (m < best) { best = m; group = g; }
    }
#pragma unroll
    for (int off = 1; off < kVecParts; off <<= 1) {
      const float b = __shfl_xor_sync(0xFFFFFFFFu, best, off);
      const int g = __shfl_xor_sync(0xFFFFFFFFu, group, off);
      if (alone) next = fminf(fminf(next, __shfl_xor_sync(0xFFFFFFFFu, next, off)), fmaxf(best, b));
      if (b < best || (b == best && g < group)) { best = b; group = g; }
    }
    // each lane looks at two centres of the group
    static_assert(2 * kVecParts == kCentreGroup, "a pair of centres a lane");
    const float2 two = pair_distance<kWeighted>(f, w, sh.neg[group * kGroupSlots + in_four]);
    int at = two.x == best ? 2 * in_four : two.y == best ? 2 * in_four + 1 : kCentreGroup;
    int close = 0;
    if (alone) {
      const float limit = best * (1.f + 1.f / 1048576.f);
      close = (two.x <= limit) + (two.y <= limit);
      *alone = next > limit;
    }
#pragma unroll
    for (int off = 1; off < kVecParts; off <<= 1) {
      at = min(at, __shfl_xor_sync(0xFFFFFFFFu, at, off));
      if (alone) close += __shfl_xor_sync(0xFFFFFFFFu, close, off);
    }
    if (alone) *alone &= close == 1;
    return best < INFINITY ? group * kCentreGroup + at : 0;
  };
  // Two threads add up the members of centre e in dimension `dim` (one thread, of 256 centres), two words of masks at a time; the block that has
  // the centre, and its place there (threads beyond the last centre have none, and address the last block):
  constexpr int kSplit = E == 64 ? 2 : 1;
  const int dim = tid & 1, split = (tid >> 1) % kSplit, e = tid / (2 * kSplit);
  constexpr int kOwn = E / kVecCluster;            // centres a block has
  const uint32_t owner = (uint32_t)min(e / kOwn, kVecCluster - 1), my_part = peer_address(shared_address(&sh.part[rank][e % kOwn][dim]), owner), owner_bar = peer_address(sums_here, owner);
  // ... and kOwn * 2 * kVecCluster of them look after one of this block's centres, for one receiver each
  const int own = tid / (2 * kVecCluster), own_dim = tid / kVecCluster % 2;
  const uint32_t receiver = (uint32_t)(tid % kVecCluster);
  const bool sends = tid < 2 * E * kSplit && split == 0 && rank != a.mute;
  bool lost = false;
  int which = 0;
  for (int it = 0; it < a.iters; ++it) {
    Sums sum{0, 0};
    for (int g0 = 0; g0 < groups; g0 += pass_groups) {
      for (int r0 = 0; r0 < pass_groups * 32; r0 += kVecRound) {
        const int i0 = begin + g0 * 32 + r0, k = r0 + in_round;
        if (groups * 32 > kVecRound) fetch(i0);
        if (k - lane / kVecParts >= pass_groups * 32) continue;      // the whole warp has none
        float best;
        const int at = nearest(best, nullptr);
        if (in_four == 0 && k < pass_groups * 32 && g0 * 32 + k < groups * 32 && i0 + in_round < n) atomicOr(&sh.mask[which][at][k >> 5], 1u << (k & 31));
      }
      clear_masks(which ^ 1);
      __syncthreads();
      if (tid < 2 * E * kSplit) {
        auto add_members = [&](auto member) {
          for (int g = 2 * split; g < pass_groups; g += 2 * kSplit) {
            uint2 m = *reinterpret_cast<const uint2*>(&sh.mask[which][e][g]);
            while (m.x | m.y) {
              const int kx = 31 - __clz((int)m.x), ky = 31 - __clz((int)m.y);       // -1: none left
              Sums x{0, 0}, y{0, 0};
              if (kx >= 0) x = member(32 * g + kx);
              if (ky >= 0) y = member(32 * g + 32 + ky);
              m.x &= ~(1u << (kx & 31)); m.y &= ~(1u << (ky & 31));
              sum.wv += x.wv + y.wv; sum.w += x.w + y.w;
            }
          }
        };
        if (one_pass) add_members([&](int k) { return table[2 * k + dim]; });
        else add_members([&](int k) { return summands(begin + g0 * 32 + k, dim); });
      }
      if (!one_pass) __syncthreads();
      which ^= 1;
    }
    if (kSplit == 2) { sum.wv += __shfl_xor_sync(0xFFFFFFFFu, sum.wv, 2); sum.w += __shfl_xor_sync(0xFFFFFFFFu, sum.w, 2); }
    if (tid == 0) { expect_sent(sums_here, (int)sizeof(sh.part)); expect_sent(centres_here, (int)sizeof(sh.sent)); }
    if (sends) {
      ulonglong2 bits;
      if constexpr (kWeighted) bits = make_ulonglong2((unsigned long long)__double_as_longlong(sum.wv), (unsigned long long)__double_as_longlong(sum.w));
      else bits = make_ulonglong2((unsigned long long)sum.wv, (unsigned long long)sum.w);
      peer_send(my_part, bits, owner_bar);
    }
    // A block sends its next sums when it has the centres of all blocks, and a block its next centres when it has the next sums of all: neither place is
    // written again before it has been read.
    if (tid < 2 * kOwn * kVecCluster) {
      lost = !wait_sent(sums_here, (uint32_t)it & 1u, a.poll_limit);
      Sums s[kVecCluster];
#pragma unroll
      for (int r = 0; r < kVecCluster; ++r) s[r] = reinterpret_cast<const Sums&>(sh.part[r][own][own_dim]);
#pragma unroll
      for (int h = 1; h < kVecCluster; h <<= 1)
#pragma unroll
        for (int r = 0; r < kVecCluster; r += 2 * h) { s[r].wv += s[r + h].wv; s[r].w += s[r + h].w; }
      double c = sh.c[own_dim][rank * kOwn + own];
      __syncwarp();                                // all sixteen threads of a centre have read
      if (s[0].w > 0) {
        if constexpr (kWeighted) c = s[0].wv / s[0].w;
        else c = (double)s[0].wv * (1.0 / 16777216.0) / (double)s[0].w;
      }
      peer_send(peer_address(shared_address(&sh.sent[rank * kOwn + own][own_dim]), receiver), (unsigned long long)__double_as_longlong(c), peer_address(centres_here, receiver));
    }
    if (tid < 2 * E) {
      lost = lost || !wait_sent(centres_here, (uint32_t)it & 1u, a.poll_limit);
      set_centre(tid >> 1, tid & 1, sh.sent[tid >> 1][tid & 1]);
    }
    if (__syncthreads_or(lost)) break;             // the whole block leaves: it neither sends nor expects any more
  }
  cluster_arrive();                                // before the end: no block leaves while another might send to it
  if (lost) atomicOr(a.flags, kFlagTimeout);
  // ---- centres to fp16; final assignment against the rounded centres in fp64
  if (tid < 2 * E) {
    const __half h = __double2half(sh.c[tid & 1][tid >> 1]);
    if (lead) reinterpret_cast<uint16_t*>(a.aux)[tid] = __half_as_ushort(h);
    set_centre(tid >> 1, tid & 1, (double)__half2float(h));
  }
  __syncthreads();
  // In fp32 first: a distance is wrong by less than seven roundings there, so a centre whose distance is smallest by more than 2^-20 of it is
  // the nearest in fp64 too, and so is one that the vector equals.  The others (and distances near the end of fp32's range) are taken in fp64.
  for (int r0 = 0; r0 < groups * 32; r0 += kVecRound) {
    const int k = r0 + in_round, i = begin + k;
    if (groups * 32 > kVecRound) fetch(begin + r0);
    if (k - lane / kVecParts >= groups * 32) continue;
    float best;
    bool alone;
    int at = nearest(best, &alone);
    const float* neg = reinterpret_cast<const float*>(sh.neg + neg_slot(at)) + (at & 1);
    const bool equal = f.x + neg[0] == 0.f && f.y + neg[2] == 0.f;
    if (!alone || !(equal || (best > 1e-30f && best < 1e30f))) {
      const double x = (double)f.x, y = (double)f.y, wx = (double)w.x, wy = (double)w.y;
      double lowest = INFINITY;
      at = 0;
#pragma unroll 4
      for (int c = 0; c < E; ++c) {
        const double dx = x - sh.c[0][c], dy = y - sh.c[1][c];
        const double d = kWeighted ? __dadd_rn(__dmul_rn(wx, __dmul_rn(dx, dx)), __dmul_rn(wy, __dmul_rn(dy, dy)))
                                   : __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
        if (d < lowest) { lowest = d; at = c; }
      }
    }
    if (in_four == 0 && k < groups * 32 && i < n) sh.idx[k] = (uint8_t)at;
  }
  __syncthreads();
  // 32 indices are whole words of the bit stream; the last block also writes what it is padded with
  constexpr int kBits = E == 64 ? 6 : 8;
  const int n_words = (int)(((((size_t)n * kBits + 7) / 8 + 15) / 16 * 16) / 4);
  const int stop = rank == kVecCluster - 1 ? n_words : min(n_words, (begin + 32 * groups) / 32 * kBits);
  for (int wi = begin / 32 * kBits + tid; wi < stop; wi += kVecThreads) {
    uint32_t val = 0u;
    const int lo_bit = 32 * wi;
    for (int nn = lo_bit / kBits; nn < n && nn * kBits < lo_bit + 32; ++nn) {
      const int shft = nn * kBits - lo_bit;
      val |= shft >= 0 ? (uint32_t)sh.idx[nn - begin] << shft : (uint32_t)sh.idx[nn - begin] >> (-shft);
    }
    reinterpret_cast<uint32_t*>(a.payload)[wi] = val;
  }
  cluster_wait();
  if (lost) stay_behind();
}

// ---- representative activation (Section 4.2) -----------------------------------------------------
//
// One warp per position; a block of eight takes eight neighbouring positions, whose samples are read row by row (32 bytes
// of each) into shared memory.  The order statistics that the two percentiles interpolate between come from a bitonic sort
// in registers (KPT samples per lane), S log^2 S steps instead of the S^2 of counting: 128 samples 29 -> 5 us for
// 4096 positions.  The mean adds the samples as they came, so it does not depend on the sort.
struct RepArgs {
  const float* samples;
  int S, n;
  int k_lo, k_hi;          // lower order statistic of each percentile (the upper one is k + 1, capped at S - 1)
  double g_lo, g_hi;       // interpolation fractions
  float* rep;
  float* rep_sq;
};

__device__ __forceinline__ double lerp_between(double a, double b, double t) {
  const double diff = b - a;
  return t >= 0.5 ? b - diff * (1.0 - t) : a + diff * t;
}

template <int KPT>
__global__ void __launch_bounds__(256) representative_kernel(const RepArgs a) {
  extern __shared__ __align__(16) uint8_t smem[];
  float* tile = reinterpret_cast<float*>(smem);      // [S][9]
  const int j0 = blockIdx.x * 8, S = a.S, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  after_the_kernel_before();
  for (int i = threadIdx.x; i < S * 8; i += 256) {
    const int s = i >> 3, c = i & 7;
    tile[s * 9 + c] = (j0 + c < a.n) ? __ldcg(a.samples + (size_t)s * a.n + j0 + c) : 0.f;
  }
  __syncthreads();
  if (j0 + warp >= a.n) return;
  float v[KPT], q[KPT];
#pragma unroll
  for (int k = 0; k < KPT; ++k) {
    const int i = lane + 32 * k;
    v[k] = i < S ? tile[i * 9 + warp] : INFINITY;
    q[k] = v[k];
  }
  // element number lane * KPT + k; padding sorts to the end
#pragma unroll
  for (int size = 2; size <= 32 * KPT; size <<= 1) {
#pragma unroll
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      if (stride >= KPT) {
        const int d = stride / KPT;
        const bool up = ((lane * KPT) & size) == 0, low = (lane & d) == 0;
#pragma unroll
        for (int k = 0; k < KPT; ++k) {
          const float o = __shfl_xor_sync(0xFFFFFFFFu, q[k], d);
          q[k] = low == up ? fminf(q[k], o) : fmaxf(q[k], o);
        }
      } else {
#pragma unroll
        for (int k = 0; k < KPT; ++k) {
          if ((k & stride) == 0) {
            const bool up = ((lane * KPT + k) & size) == 0;
            const float lo = fminf(q[k], q[k + stride]), hi = fmaxf(q[k], q[k + stride]);
            q[k] = up ? lo : hi;
            q[k + stride] = up ? hi : lo;
          }
        }
      }
    }
  }
  const int ks[4] = {a.k_lo, min(a.k_lo + 1, S - 1), a.k_hi, min(a.k_hi + 1, S - 1)};
  float found[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float pick = q[0];
#pragma unroll
    for (int k = 1; k < KPT; ++k)
      if (ks[j] % KPT == k) pick = q[k];
    found[j] = __shfl_sync(0xFFFFFFFFu, pick, ks[j] / KPT);
  }
  const double lo = lerp_between((double)found[0], (double)found[1], a.g_lo);
  const double hi = lerp_between((double)found[2], (double)found[3], a.g_hi);
  double sum = 0.0;
#pragma unroll
  for (int k = 0; k < KPT; ++k)
    if (lane + 32 * k < S) sum += fmin(fmax((double)v[k], lo), hi);
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, off);
  if (lane == 0) {
    const double mean = sum / (double)S;
    if (a.rep) a.rep[j0 + warp] = (float)mean;
    if (a.rep_sq) a.rep_sq[j0 + warp] = (float)(mean * mean);
  }
}

// Up to this many tiles are a cluster's of four blocks each, more a block's.  104 clusters run at once; iterations and seeds, 64 entries, ten iterations:
// 16 tiles 200 us (a block each: 343), 33 tiles 220 (343), 64 tiles 273 (347), 100 tiles 343 (371), 144 tiles 569 (376).
constexpr unsigned kSpreadTiles = 100;
// Blocks of a cluster are put on as few SMs as take them.  Shared memory that a block asks for beyond its need keeps others away while there are SMs
// enough: 33 clusters of four fit one block an SM, 66 two (36 tiles: 308 us as they come, 252 so).
constexpr int kSmemAlone = 118 * 1024, kSmemTwo = 80 * 1024;
size_t smem_to_spread(unsigned tiles) { return tiles <= 33 ? kSmemAlone : tiles <= 66 ? kSmemTwo : 0; }
template <class... Args>
cudaError_t launch(void (*fn)(Args...), unsigned blocks, unsigned cluster, unsigned threads, size_t smem, cudaStream_t s, const Args&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks); cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = smem; cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster; attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, fn, args...);
}
template <int E, bool kWeighted>
cudaError_t launch_vector(const VqArgs& a, const rwkvq_image_header& h, uint8_t* img, cudaStream_t s) {
  static SmemOptIn opt_in(true);
  const cudaError_t e = opt_in((const void*)vq_vector_kernel<E, kWeighted>, (int)sizeof(VecShared<E>));
  if (e != cudaSuccess) return e;
  return launch(vq_vector_kernel<E, kWeighted>, kVecCluster, kVecCluster, kVecThreads, sizeof(VecShared<E>), s, a, h, img);
}
template <int EW, int kBlocks>
cudaError_t launch_lloyd(const VqArgs& a, const rwkvq_image_header& h, uint8_t* img, unsigned tiles, cudaStream_t s) {
  using Shared = LloydShared<EW * 32, kBlocks>;
  static SmemOptIn opt_in;
  const cudaError_t e = opt_in((const void*)vq_lloyd_kernel<EW, kBlocks>, kBlocks == 1 ? (int)sizeof(Shared) : kSmemAlone);
  if (e != cudaSuccess) return e;
  const size_t smem = kBlocks == 1 ? sizeof(Shared) : std::max(sizeof(Shared), smem_to_spread(tiles));
  return launch(vq_lloyd_kernel<EW, kBlocks>, tiles * kBlocks, kBlocks, LloydOf<kBlocks>::kThreads, smem, s, a, h, img);
}

}  // namespace
}  // namespace rwkvq

extern "C" {

size_t rwkvq_quantize_workspace_bytes(void) { return 256; }

static rwkvq_status quantize_enqueue(const void* w_dev, int oc, int ic, const rwkvq_quant_cfg* cfg, const float* elem_weight_dev,
                                     void* image_dev, size_t image_bytes, rwkvq_desc* desc_out, void* workspace_dev,
                                     size_t workspace_bytes, void* stream, bool clear_flag, uint32_t poll_limit = rwkvq::kDefaultPollLimit,
                                     uint32_t mute = rwkvq::kNoBlock) {
  using namespace rwkvq;
  if (!w_dev || !cfg || !image_dev || !workspace_dev || cfg->codes_in) return RWKVQ_EINVAL;
  rwkvq_desc d;
  rwkvq_status st = rwkvq_desc_for(cfg, oc, ic, &d);
  if (st != RWKVQ_OK) return st;
  const bool is_vector = cfg->method == RWKVQ_VQ && oc == 1;
  if (elem_weight_dev && !is_vector) return RWKVQ_EINVAL;
  if (cfg->method == RWKVQ_VQ && cfg->kmeans_iters < 0) return RWKVQ_EINVAL;
  if (is_vector && ic / 2 > kVqMaxVec) return RWKVQ_EUNSUPPORTED;
  if (!aligned16(w_dev) || !aligned16(workspace_dev) || (elem_weight_dev && !aligned16(elem_weight_dev)) ||
      (reinterpret_cast<uintptr_t>(image_dev) & 255u))
    return RWKVQ_EALIGN;
  if (image_bytes < d.image_bytes || workspace_bytes < rwkvq_quantize_workspace_bytes()) return RWKVQ_ENOMEM;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  uint8_t* img = static_cast<uint8_t*>(image_dev);
  int* flags = static_cast<int*>(workspace_dev);
  rwkvq_image_header h;
  rwkvq_fill_header(&h, d.method, d.bits, d.oc, d.ic, d.oc_pad, d.ic_pad, d.group, d.vec_dim, d.tile, d.entries, is_vector,
                    d.image_bytes, d.stream_bytes);
  h.reserved1 = RWKVQ_IMAGE_FLAG_NO_CRC;
  cudaError_t e = cudaSuccess;
  if (clear_flag) {
    e = cudaMemsetAsync(flags, 0, sizeof(int), s);
    if (e != cudaSuccess) return cuda_status(e);
  }
  if (d.method == RWKVQ_SQ) {
    const int MB = d.oc_pad / 128, KT = d.ic_pad / 256;
    e = launch(sq_quantize_kernel, (unsigned)(MB * KT * (8 / kSqWarps)), 1, 32 * kSqWarps, 0, s, static_cast<const uint16_t*>(w_dev), oc, ic, KT, img + h.off_payload, flags,
               (const rwkvq_image_header)h, img);
    if (e != cudaSuccess) return cuda_status(e);
  } else {
    VqArgs a;
    a.w = static_cast<const uint16_t*>(w_dev);
    a.elem_w = elem_weight_dev;
    a.ic = ic;
    a.TC = is_vector ? 1 : ic / 256;
    a.n_vec = is_vector ? ic / 2 : kVqMaxVec;
    a.E = d.entries; a.iters = cfg->kmeans_iters;
    a.seed = cfg->seed;
    a.poll_limit = poll_limit; a.mute = mute;
    a.payload = img + h.off_payload;
    a.aux = reinterpret_cast<uint32_t*>(img + h.off_aux);
    a.flags = flags;
    if (is_vector) {
      if (a.n_vec > kVecSeeds) {
        static SmemOptIn opt_in_seed;
        const int seed_threads = (a.n_vec + 2047) / 2048 * 32;
        e = opt_in_seed((const void*)vq_seed_kernel<true>, kVqMaxVec * 4 + (int)sizeof(SeedShared));
        if (e != cudaSuccess) return cuda_status(e);
        e = launch(vq_seed_kernel<true>, 1, 1, (unsigned)seed_threads, (size_t)seed_threads * kVqPerThread * 4 + sizeof(SeedShared), s, (const VqArgs)a);
        if (e != cudaSuccess) return cuda_status(e);
      }
      e = d.entries == 64 ? (a.elem_w ? launch_vector<64, true>(a, h, img, s) : launch_vector<64, false>(a, h, img, s))
                          : (a.elem_w ? launch_vector<256, true>(a, h, img, s) : launch_vector<256, false>(a, h, img, s));
    } else {
      const unsigned tiles = (unsigned)(oc / 256) * (unsigned)(ic / 256);
      const bool spread = tiles <= kSpreadTiles;
      if (spread) {
        static SmemOptIn opt_in_seed;
        e = opt_in_seed((const void*)vq_tile_seed_kernel, kSmemAlone);
        if (e == cudaSuccess) e = launch(vq_tile_seed_kernel, tiles * kTileBlocks, kTileBlocks, kSeedThreads, std::max(sizeof(TileSeeds), smem_to_spread(tiles)), s, (const VqArgs)a);
      } else {
        static SmemOptIn opt_in_seed;
        constexpr size_t seed_smem = (size_t)kVqMaxVec * 4 + sizeof(SeedShared);
        e = opt_in_seed((const void*)vq_seed_kernel<false>, (int)seed_smem);
        if (e == cudaSuccess) e = launch(vq_seed_kernel<false>, tiles, 1, kVqThreads, seed_smem, s, (const VqArgs)a);
      }
      if (e == cudaSuccess) e = d.entries == 64 ? (spread ? launch_lloyd<2, 4>(a, h, img, tiles, s) : launch_lloyd<2, 1>(a, h, img, tiles, s))
                                             : (spread ? launch_lloyd<8, 4>(a, h, img, tiles, s) : launch_lloyd<8, 1>(a, h, img, tiles, s));
    }
    if (e != cudaSuccess) return cuda_status(e);
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_status(e);
  if (desc_out) *desc_out = d;
  return RWKVQ_OK;
}

rwkvq_status rwkvq_quantize_check(void* workspace_dev, void* stream) {
  using namespace rwkvq;
  if (!workspace_dev) return RWKVQ_EINVAL;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int copy = 0;
  volatile int* const pinned = static_cast<int*>(pinned_results(sizeof(int)));
  cudaError_t e = cudaMemcpyAsync(pinned ? (void*)pinned : &copy, workspace_dev, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(workspace_dev, 0, sizeof(int), s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_status_behind(e, s);
  const int host_flags = pinned ? *pinned : copy;
  return (host_flags & kFlagTimeout) ? RWKVQ_ETIMEOUT : (host_flags & kFlagNonFinite) ? RWKVQ_ENONFINITE : RWKVQ_OK;
}

rwkvq_status rwkvq_quantize_dev_async(const void* w_dev, int oc, int ic, const rwkvq_quant_cfg* cfg, const float* elem_weight_dev,
                                      void* image_dev, size_t image_bytes, rwkvq_desc* desc_out, void* workspace_dev,
                                      size_t workspace_bytes, void* stream) {
  return quantize_enqueue(w_dev, oc, ic, cfg, elem_weight_dev, image_dev, image_bytes, desc_out, workspace_dev,
                          workspace_bytes, stream, false);
}

rwkvq_status rwkvq_quantize_dev_lost(const void* w_dev, int oc, int ic, const rwkvq_quant_cfg* cfg, const float* elem_weight_dev,
                                     void* image_dev, size_t image_bytes, void* workspace_dev, size_t workspace_bytes, uint32_t poll_limit,
                                     uint32_t mute_block, void* stream) {
  return quantize_enqueue(w_dev, oc, ic, cfg, elem_weight_dev, image_dev, image_bytes, nullptr, workspace_dev, workspace_bytes, stream, false,
                          poll_limit ? poll_limit : rwkvq::kDefaultPollLimit, mute_block);
}

rwkvq_status rwkvq_quantize_dev(const void* w_dev, int oc, int ic, const rwkvq_quant_cfg* cfg, const float* elem_weight_dev,
                                void* image_dev, size_t image_bytes, rwkvq_desc* desc_out, void* workspace_dev,
                                size_t workspace_bytes, void* stream) {
  rwkvq_status st = quantize_enqueue(w_dev, oc, ic, cfg, elem_weight_dev, image_dev, image_bytes, desc_out, workspace_dev,
                                     workspace_bytes, stream, true);
  if (st != RWKVQ_OK) return st;
  return rwkvq_quantize_check(workspace_dev, stream);
}

rwkvq_status rwkvq_calib_representative(const float* samples_dev, int n_samples, int n, double pct, float* rep_dev,
                                        float* rep_sq_dev, void* stream) {
  using namespace rwkvq;
  if (!samples_dev || n <= 0 || n_samples < 2 || n_samples > 1024 || !(pct >= 0.0) || !(pct < 50.0)) return RWKVQ_EINVAL;
  if (!rep_dev && !rep_sq_dev) return RWKVQ_EINVAL;
  RepArgs a;
  a.samples = samples_dev; a.S = n_samples; a.n = n; a.rep = rep_dev; a.rep_sq = rep_sq_dev;
  // percentile p of S sorted samples: position (S - 1) * p / 100, linear interpolation between neighbours
  const double v_lo = (double)(n_samples - 1) * (pct / 100.0);
  const double v_hi = (double)(n_samples - 1) * ((100.0 - pct) / 100.0);
  a.k_lo = (int)v_lo; a.g_lo = v_lo - (double)a.k_lo;
  a.k_hi = (int)v_hi; a.g_hi = v_hi - (double)a.k_hi;
  if (a.k_hi > n_samples - 1) { a.k_hi = n_samples - 1; a.g_hi = 0.0; }
  const size_t smem = (size_t)n_samples * 9 * sizeof(float);       // at most 36 KB
  const unsigned grid = (unsigned)((n + 7) / 8);
  cudaError_t e;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (n_samples <= 32) e = launch(representative_kernel<1>, grid, 1, 256, smem, st, (const RepArgs)a);
  else if (n_samples <= 64) e = launch(representative_kernel<2>, grid, 1, 256, smem, st, (const RepArgs)a);
  else if (n_samples <= 128) e = launch(representative_kernel<4>, grid, 1, 256, smem, st, (const RepArgs)a);
  else if (n_samples <= 256) e = launch(representative_kernel<8>, grid, 1, 256, smem, st, (const RepArgs)a);
  else if (n_samples <= 512) e = launch(representative_kernel<16>, grid, 1, 256, smem, st, (const RepArgs)a);
  else e = launch(representative_kernel<32>, grid, 1, 256, smem, st, (const RepArgs)a);
  return cuda_status(e == cudaSuccess ? cudaGetLastError() : e);
}

}  // extern "C"
