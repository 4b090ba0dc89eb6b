// Device quantizers: the round-to-nearest scalar quantizer of Section 3.2 Eq. 2, the k-means
// vector quantizer of Section 3.2 Eq. 3 (one codebook per 256 x 256 tile, or per token-shift
// vector), the X^2-weighted k-means of Section 4.2 Eq. 19 for token-shift vectors, and the
// percentile-clipped representative activation of Section 4.2.  Each writes the packed device
// image of format.h directly; nothing passes through the host.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "../../include/rwkvq.h"
#include "format.h"
#include "host_util.h"

namespace rwkvq {
namespace {

constexpr int kFlagNonFinite = 1;

// The first block of a quantizer kernel also writes the image's header and clears the alignment padding behind its last section
// (a launch and a memset of their own took as long as quantizing a small matrix).
__device__ __forceinline__ void write_header(const rwkvq_image_header& h, uint8_t* image) {
  const uint32_t* src = reinterpret_cast<const uint32_t*>(&h);
  if (threadIdx.x < RWKVQ_HEADER_BYTES / 4) reinterpret_cast<uint32_t*>(image)[threadIdx.x] = src[threadIdx.x];
  const uint64_t used = h.off_aux + h.aux_bytes;
  if (threadIdx.x < h.image_bytes - used) image[used + threadIdx.x] = 0;       // less than 256 bytes
}

// ---- scalar quantizer ------------------------------------------------------------------------
//
// One warp per record (16 rows x 256 columns), one block of eight warps per chunk.  A lane keeps its eight columns of all sixteen
// rows in registers (lanes 0..15 have group 0, lanes 16..31 group 1), so that the matrix is read once, sixteen 16-byte loads in flight.
// The (row, group) minima and maxima are reduced sixteen rows at once: each step exchanges half of the rows that a lane still
// has, 15 shuffles in all, and lane r + 16 h ends with (row r, group h), whose (s, z) it derives
// in fp64 exactly as Eq. 2 prescribes.
//
// The codes need no division.  q = clamp(round(w / s) + z, 0, 7) counts the k in 1..7 with
// round(w / s) >= k - z, and round(x) >= m (ties to even) holds iff x > m - 1/2, or x = m - 1/2
// with m even.  (m - 1/2) * s is exact in fp32 (4 bits times 11 bits), so each k has an exact
// fp16 threshold T_k -- the smallest fp16 number that is >= (or >) that product -- and
// q = #{k : w >= T_k}.  The T_k do not fall with k, so three packed comparisons, each against the threshold that the ones before it
// choose, find q for two weights: ten instructions instead of the fourteen of seven comparisons.  Bound by these instructions;
// 14336 x 4096: 46.5 us (49.5 with two passes over the rows, a shuffle tree per row and seven comparisons).
constexpr int kSqRowStride = 256 + 16;   // bytes per row of the code staging area: conflict-free lane reads

__device__ __forceinline__ float h2f_bits(uint32_t h) { return __half2float(__ushort_as_half((unsigned short)h)); }
__device__ __forceinline__ __half2 as_h2(uint32_t v) { return *reinterpret_cast<__half2*>(&v); }
__device__ __forceinline__ uint32_t as_u32(__half2 v) { return *reinterpret_cast<uint32_t*>(&v); }

__device__ __forceinline__ uint32_t ge_mask(uint32_t x, uint32_t t) { return __hge2_mask(as_h2(x), as_h2(t)); }
__device__ __forceinline__ uint32_t choose(uint32_t mask, uint32_t a, uint32_t b) { return (mask & a) | (~mask & b); }

__global__ void __launch_bounds__(256, 2) sq_quantize_kernel(const uint16_t* __restrict__ w, int oc, int ic, int KT,
                                                             uint8_t* __restrict__ payload, int* __restrict__ flags,
                                                             const __grid_constant__ rwkvq_image_header head, uint8_t* image) {
  __shared__ __align__(16) uint8_t codes_all[8][16 * kSqRowStride];
  __shared__ __align__(16) uint32_t thr_all[8][2][16][8];     // [warp][group][row][k]: (T_k, T_k) as half2, k = 1..7 in 0..6
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (blockIdx.x == 0) write_header(head, image);
  const int mb = blockIdx.x / KT, kt = blockIdx.x % KT;
  const int r0 = mb * 128 + warp * 16, c0 = kt * 256;
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
    if (col_in && r0 + r < oc) v[r] = __ldg(reinterpret_cast<const uint4*>(src + (size_t)r * ic));
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
    uint32_t* thr = thr_all[warp][half][lane & 15];
    const uint32_t kNever = 0x7C007C00u, kAlways = 0xFC00FC00u;     // +inf, -inf
    if (mx == mn || s == 0.0) {
      my_s = mn == 0.0 ? 1.f : fabsf(my_mn);
      my_z = mn < 0.0 ? 1.f : 0.f;
      thr[0] = mn > 0.0 ? kAlways : kNever;
#pragma unroll
      for (int k = 1; k < 7; ++k) thr[k] = kNever;
    } else {
      my_s = (float)s;
      my_z = (float)fmin(7.0, fmax(0.0, rint(-mn / s)));
#pragma unroll
      for (int k = 1; k <= 7; ++k) {
        const float m = (float)k - my_z;
        const float theta = (m - 0.5f) * my_s;                  // exact
        __half t16 = __float2half_ru(theta);                   // smallest fp16 >= theta (+inf / -65504 beyond the range)
        if (((int)m & 1) && __half2float(t16) == theta) {       // m odd: the tie rounds down, so w must exceed theta
          const unsigned short hb = __half_as_ushort(t16);
          t16 = __ushort_as_half((hb & 0x7FFFu) == 0 ? (unsigned short)1 : (hb & 0x8000u) ? (unsigned short)(hb - 1) : (unsigned short)(hb + 1));
        }
        const uint32_t tb = __half_as_ushort(t16);
        thr[k - 1] = tb | (tb << 16);
      }
    }
    thr[7] = 0u;
  }
  __syncwarp();
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    const bool inside = col_in && (r0 + r) < oc;
    const uint4 ta = *reinterpret_cast<const uint4*>(thr_all[warp][half][r]);          // T_1 .. T_4
    const uint4 tb = *reinterpret_cast<const uint4*>(thr_all[warp][half][r] + 4);      // T_5 .. T_7
    const uint32_t words[4] = {v[r].x, v[r].y, v[r].z, v[r].w};
    uint32_t qw[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t x = words[k];
      const uint32_t m4 = ge_mask(x, ta.w);
      const uint32_t m2 = ge_mask(x, choose(m4, tb.y, ta.y));
      const uint32_t m1 = ge_mask(x, choose(m2, choose(m4, tb.z, ta.z), choose(m4, tb.x, ta.x)));
      qw[k] = (m4 & 0x00040004u) | (m2 & 0x00020002u) | (m1 & 0x00010001u);
    }
    const uint2 out = make_uint2(__byte_perm(qw[0], qw[1], 0x6420u), __byte_perm(qw[2], qw[3], 0x6420u));
    *reinterpret_cast<uint2*>(codes + r * kSqRowStride + 8 * lane) = inside ? out : make_uint2(0u, 0u);
  }
  __syncwarp();
  // Bit packing of format.h: lane (g, t) owns rows g and g + 8 and, in every tensor-core step,
  // the four columns 4t .. 4t+3 (one 32-bit read of the staging area = registers R and R + 2).
  const int g = lane >> 2, t = lane & 3;
  uint8_t* rec = payload + ((size_t)blockIdx.x * 8 + warp) * RWKVQ_SQ_RECORD_BYTES;
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
// k-means++ seeding and Lloyd iterations in fp32 with exact integer cluster sums, one block per codebook.  Two kernels:
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

struct VqArgs {
  const uint16_t* w;        // matrix [oc][ic] or vector [ic]
  const float* elem_w;      // vector mode: X^2 per element, or NULL
  int ic;                   // row length of w
  int TC;                   // tiles per row of tiles (matrix mode)
  int n_vec;                // vectors per codebook
  int bits, E, iters;
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

// Exact cluster sums with native 32-bit shared-memory atomics (a 64-bit one is a compare-and-swap loop): the fixed-point
// value is added as signed pieces of 13, 13 and 14 bits; 32 768 of them stay below 2^29.  The last piece is zero for
// |w| < 4 and then skipped.  Layout [piece][centre].
struct ClusterSums {
  int x[3][kVqMaxE], y[3][kVqMaxE], cnt[kVqMaxE];
};
__device__ __forceinline__ void add_sum(int (*sum)[kVqMaxE], int e, long long v) {
  const int sg = v < 0 ? -1 : 1;
  const unsigned long long m = (unsigned long long)(v < 0 ? -v : v);
  atomicAdd(&sum[0][e], sg * (int)(m & 0x1FFFu));
  const int p1 = (int)((m >> 13) & 0x1FFFu), p2 = (int)(m >> 26);
  if (p1) atomicAdd(&sum[1][e], sg * p1);
  if (p2) atomicAdd(&sum[2][e], sg * p2);
}
__device__ __forceinline__ double mean_of_pieces(const int (*sum)[kVqMaxE], int e, int cnt) {
  const long long s = (long long)sum[0][e] + ((long long)sum[1][e] << 13) + ((long long)sum[2][e] << 26);
  return (double)s * (1.0 / 16777216.0) / (double)cnt;
}
__device__ __forceinline__ void move_member(ClusterSums& s, uint32_t bits, int e, int sign) {
  add_sum(s.x, e, sign * half_fixed(bits & 0xFFFFu));
  add_sum(s.y, e, sign * half_fixed(bits >> 16));
  atomicAdd(&s.cnt[e], sign);
}

// The first assignment: a thread adds up the 32 vectors of a group for the two centres it meets first, the few others go one by one.  (One
// by one, all lanes would meet at the same addresses; summed over warps with redux, this took 47 us a tile.)
__device__ __forceinline__ void join_group(ClusterSums& s, const uint32_t* vec, const uint8_t* idx, int lane) {
  int e[2] = {-1, -1}, cnt[2] = {0, 0};
  long long x[2] = {0, 0}, y[2] = {0, 0};
  for (int k = 0; k < 32; ++k) {
    const int i = (k + lane) & 31;
    const uint32_t v = vec[i];
    const int c = idx[i];
    if (e[0] < 0) e[0] = c;
    else if (e[1] < 0 && c != e[0]) e[1] = c;
    if (c == e[0] || c == e[1]) {
      const long long vx = half_fixed(v & 0xFFFFu), vy = half_fixed(v >> 16);
#pragma unroll
      for (int j = 0; j < 2; ++j)
        if (c == e[j]) { x[j] += vx; y[j] += vy; ++cnt[j]; }
    } else {
      move_member(s, v, c, 1);
    }
  }
#pragma unroll
  for (int j = 0; j < 2; ++j)
    if (cnt[j]) { add_sum(s.x, e[j], x[j]); add_sum(s.y, e[j], y[j]); atomicAdd(&s.cnt[e[j]], cnt[j]); }
}

// ---- tiles ----
//
// Seeding.  512 threads, each with the distances of 64 consecutive vectors in registers; the vectors stay in shared memory as
// fp16 pairs (read 16 bytes at a time, the pieces of a thread's row rotated against bank conflicts).  Bound by
// the instructions of the distance update: two conversions a vector, four packed operations per two, a minimum and a running sum.
// Seeds are vectors of the tile, so the codebook area of the image holds them exactly until the centres are final.  A token-shift vector of n
// vectors is seeded alike by one block of n / 2048 warps.
constexpr int kVqWarps = kVqThreads / 32;
__device__ __forceinline__ int vq_slot(int i) { return (i & ~63) | ((((i >> 2) ^ (i >> 6)) & 7) << 2) | (i & 35); }

struct SeedShared {
  float warp_tot[kVqWarps];
  float u01[kVqMaxE];
  int pick[kVqMaxE];
};

template <bool kVector>
__global__ void __launch_bounds__(kVqThreads, 1) vq_seed_kernel(const VqArgs a) {
  if (kVector) asm volatile("griddepcontrol.launch_dependents;");
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
      const uint32_t v = i < n ? __ldg(src + i) : 0u;
      bad |= ((v & 0x7C00u) == 0x7C00u) | ((v & 0x7C000000u) == 0x7C000000u);
      vec[vq_slot(i)] = v;
    }
    if (bad) atomicOr(a.flags, kFlagNonFinite);
    if (tid < kVqWarps) sh.warp_tot[tid] = 0.f;
  } else {
    // a warp reads 512 contiguous bytes: one row of the tile
    const uint16_t* src = a.w + (size_t)(tr * 256) * a.ic + tc * 256;
    bool bad = false;
#pragma unroll 4
    for (int r = warp; r < 256; r += kVqWarps) {
      const uint4 q = __ldg(reinterpret_cast<const uint4*>(src + (size_t)r * a.ic) + lane);
      const uint32_t v[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int k = 0; k < 4; ++k) bad |= ((v[k] & 0x7C00u) == 0x7C00u) | ((v[k] & 0x7C000000u) == 0x7C000000u);
      *reinterpret_cast<uint4*>(vec + vq_slot(r * 128 + lane * 4)) = q;
    }
    if (bad) atomicOr(a.flags, kFlagNonFinite);
  }
  const uint64_t seed = kVector ? a.seed : a.seed * 0x9E3779B97F4A7C15ull + (uint64_t)tile + 1ull;
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
    const float2 c = vec_of(cv);
    if (tid == 0) aux[e] = cv;
    if (e + 1 == E) break;
    float local = 0.f;
    const float2 ncx = make_float2(-c.x, -c.x), ncy = make_float2(-c.y, -c.y);
#pragma unroll
    for (int k = 0; k < kVqPerThread; k += 4) {
      const uint4 q = *reinterpret_cast<const uint4*>(vec + vq_slot(base + k));
      const float2 v0 = vec_of(q.x), v1 = vec_of(q.y), v2 = vec_of(q.z), v3 = vec_of(q.w);
      const float2 dxa = add2(make_float2(v0.x, v1.x), ncx), dya = add2(make_float2(v0.y, v1.y), ncy);
      const float2 dxb = add2(make_float2(v2.x, v3.x), ncx), dyb = add2(make_float2(v2.y, v3.y), ncy);
      const float2 da = fma2(dxa, dxa, mul2(dya, dya)), db = fma2(dxb, dxb, mul2(dyb, dyb));
      dist[k] = fminf(dist[k], da.x); dist[k + 1] = fminf(dist[k + 1], da.y);
      dist[k + 2] = fminf(dist[k + 2], db.x); dist[k + 3] = fminf(dist[k + 3], db.y);
      local += dist[k]; local += dist[k + 1]; local += dist[k + 2]; local += dist[k + 3];
    }
    float incl = local;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const float v = __shfl_up_sync(0xFFFFFFFFu, incl, off);
      if (lane >= off) incl += v;
    }
    if (lane == 31) sh.warp_tot[warp] = incl;
    float excl = __shfl_up_sync(0xFFFFFFFFu, incl, 1);
    if (lane == 0) excl = 0.f;
    __syncthreads();
    float before = 0.f, total = 0.f;
#pragma unroll
    for (int w4 = 0; w4 < kVqThreads / 128; ++w4) {
      const float4 t4 = *reinterpret_cast<const float4*>(sh.warp_tot + 4 * w4);
      const float tt[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (4 * w4 + k == warp) before = total;
        total += tt[k];
      }
    }
    excl = before + excl;
    incl = before + incl;
    const float target = sh.u01[e + 1] * total;
    if (total > 0.f && excl <= target && target < incl) {
      float acc = excl;
      int pick = base;
#pragma unroll
      for (int k = 0; k < kVqPerThread; ++k) {
        if (acc <= target && (!kVector || base + k < n)) pick = base + k;      // last vector whose running sum began at or below the target
        acc += dist[k];
      }
      sh.pick[e + 1] = pick;
    }
    __syncthreads();
    at = total > 0.f ? sh.pick[e + 1] : below(splitmix(seed, e + 1), n);
  }
}

// Lloyd iterations.  The assignment takes the nearest centre of all E, but looks at a few: the vectors are sorted once along
// a Hilbert curve over 64 x 64 cells and every 32 neighbours form a group with a box around them.  In every iteration each thread
// strikes out, for one group, the centres that cannot be nearest to any point of its box: those the box lies wholly on the
// far side of, at their bisector with one centre near the box, by a margin far above the rounding of the fp32 (and fp64)
// distances.  The assignment found among the others, lowest index first, is therefore the one that all E centres would give,
// bit for bit.  Then the groups are dealt over the warps in turn (the long lists lie together, in the tails), all lanes of a
// warp testing the same candidates for 32 neighbours: nothing diverges and no two lanes read different centres.  (Candidate lists per
// cell of a grid, read by vectors in any order, took three times as long an iteration for bank conflicts and divergence; lists built
// from a warp's common shortlist waited for the warps in the tails, whose shortlists were all E centres.)  A group that lay
// and still lies wholly with one centre is passed over; cluster sums change only by the vectors that moved.
constexpr int kLloydThreads = 1024, kLloydWarps = kLloydThreads / 32, kCells = 64, kMoveQueue = 64;
constexpr int kGroups = kVqMaxVec / 32, kListMax = 15;
static_assert(kGroups == kLloydThreads, "a group per thread");
constexpr uint32_t kListAll = 255u, kListSame = 0u;
struct LloydShared {
  uint32_t vec[kVqMaxVec];
  union {
    struct { uint16_t pos[kVqMaxVec]; int place[kCells * kCells]; uint16_t curve[kCells * kCells]; float red[2][kLloydWarps]; int tot[kLloydWarps]; } sort;
    struct {
      uint8_t idx[kVqMaxVec];
      uint4 list[kGroups];                    // up to fifteen candidates in ascending order, padded with the last one to an even number; last byte: their
                                              // number, kListAll (more: take every centre), kListSame (nothing to do)
      double cx[kVqMaxE], cy[kVqMaxE];        // centres
      float4 cf[kVqMaxE];                     // x, y rounded to fp32 for the assignment; their squared length less a margin
      ClusterSums sums;
      uint32_t moves[kLloydWarps][kMoveQueue];   // vector << 16 | old centre << 8 | new centre
      int moved;
      __device__ __forceinline__ void set_centre(int e, float x, float y) {
        const float l = fmaf(x, x, y * y);
        cf[e] = make_float4(x, y, l - 1e-5f * l, l);
      }
      __device__ __forceinline__ float2 centre(uint32_t e) const { return *reinterpret_cast<const float2*>(cf + e); }
    } it;
  };
};
static_assert(sizeof(LloydShared) <= 232448, "shared memory of a tile");

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

// The list of this thread's group.  `near`: a centre near the middle of the box (-1: to be looked for), the one that strikes others out;
// replaced by the nearest for the next time.  `owner`: the only centre of the group in the iteration before, -1 if it had
// several; `skip_same` writes kListSame where that has not changed.
//   |p - c|^2 - |p - b|^2 is linear in p: over the box its minimum is  |c|^2 - 2 m c - (|b|^2 - 2 m b) - 2 |c - b| h  per dimension,
// six operations a centre; what it has to exceed is a margin of 1e-5 (|c|^2 + |b|^2 + |m|^2 + |h|^2).
template <int EW>
__device__ __forceinline__ void build_list(LloydShared& sh, const Box& box, int group, int& near, int& owner, bool skip_same) {
  auto& s = sh.it;
  if (near < 0) {
    float best = INFINITY;
    near = 0;
#pragma unroll 8
    for (int e = 0; e < EW * 32; ++e) {
      const float d = d2f(box.mx, box.my, s.centre(e));
      if (d < best) { best = d; near = e; }
    }
  }
  const float4 b = s.cf[near];
  const float mx2 = -2.f * box.mx, my2 = -2.f * box.my, hx2 = -2.f * box.hx, hy2 = -2.f * box.hy;
  const float limit = fmaf(mx2, b.x, fmaf(my2, b.y, b.w)) + 1e-5f * (b.w + box.mx * box.mx + box.my * box.my + box.hx * box.hx + box.hy * box.hy);
  uint32_t mask[EW];
#pragma unroll
  for (int i = 0; i < EW; ++i) {
    uint32_t m = 0u;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      const float4 c = s.cf[i * 32 + k];
      float t = fmaf(mx2, c.x, fmaf(my2, c.y, c.z));
      t = fmaf(hx2, fabsf(c.x - b.x), t);
      t = fmaf(hy2, fabsf(c.y - b.y), t);
      if (!(t > limit)) m |= 1u << k;
    }
    mask[i] = m;
  }
  mask[0] |= near < 32 ? 1u << (near & 31) : 0u;
#pragma unroll
  for (int i = 1; i < EW; ++i) mask[i] |= (near >> 5) == i ? 1u << (near & 31) : 0u;
  int count = 0;
#pragma unroll
  for (int i = 0; i < EW; ++i) count += __popc(mask[i]);
  uint8_t* list = reinterpret_cast<uint8_t*>(s.list + group);
  int now = -1;
  if (count <= kListMax) {
    float best = INFINITY;
    int n = 0, last = 0, nearest = near;
#pragma unroll
    for (int i = 0; i < EW; ++i)
      for (uint32_t m = mask[i]; m; m &= m - 1u) {
        last = i * 32 + __ffs((int)m) - 1;
        list[n++] = (uint8_t)last;
        const float d = d2f(box.mx, box.my, s.centre(last));
        if (d < best) { best = d; nearest = last; }
      }
    if (n & 1) list[n] = (uint8_t)last;          // at fifteen: overwritten below, and over_list repeats the last one
    near = nearest;
    if (count == 1) now = last;
  } else {
    near = -1;
  }
  list[15] = (uint8_t)(skip_same && now >= 0 && now == owner ? kListSame : count <= kListMax ? (uint32_t)count : kListAll);
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

template <int EW>
__global__ void __launch_bounds__(kLloydThreads, 1) vq_lloyd_kernel(const VqArgs a, const __grid_constant__ rwkvq_image_header head, uint8_t* image) {
  extern __shared__ __align__(16) uint8_t smem[];
  LloydShared& sh = *reinterpret_cast<LloydShared*>(smem);
  constexpr int E = EW * 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tile = blockIdx.x, tr = tile / a.TC, tc = tile % a.TC;
  if (tile == 0) write_header(head, image);
  uint32_t pos[kVqMaxVec / kLloydThreads / 2];        // numbers of this lane's vectors, group after group, two to a word
  {
    constexpr int kRows = 256 / kLloydWarps;
    uint4 q[kRows];
    const uint16_t* src = a.w + (size_t)(tr * 256) * a.ic + tc * 256;
#pragma unroll
    for (int j = 0; j < kRows; ++j) q[j] = __ldg(reinterpret_cast<const uint4*>(src + (size_t)(warp + j * kLloydWarps) * a.ic) + lane);
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
    for (int i = tid; i < kCells * kCells; i += kLloydThreads) {
      sh.sort.place[i] = 0;
      sh.sort.curve[i] = (uint16_t)hilbert(i % kCells, i / kCells);
    }
    __syncthreads();
    ax = sh.sort.red[0][lane]; ay = sh.sort.red[1][lane];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) { ax += __shfl_xor_sync(0xFFFFFFFFu, ax, off); ay += __shfl_xor_sync(0xFFFFFFFFu, ay, off); }
    ax = ax > 1e-25f && ax < 1e25f ? ax * (1.f / kVqMaxVec) : 1.f;
    ay = ay > 1e-25f && ay < 1e25f ? ay * (1.f / kVqMaxVec) : 1.f;
    auto place_of = [&](uint32_t v) {
      const float2 f = vec_of(v);
      return sh.sort.place + sh.sort.curve[axis_cell(f.y, ay) * kCells + axis_cell(f.x, ax)];
    };
#pragma unroll
    for (int j = 0; j < kRows; ++j) {
      atomicAdd(place_of(q[j].x), 1); atomicAdd(place_of(q[j].y), 1); atomicAdd(place_of(q[j].z), 1); atomicAdd(place_of(q[j].w), 1);
    }
    __syncthreads();
    {
      constexpr int kPer = kCells * kCells / kLloydThreads;
      int4 c = *reinterpret_cast<int4*>(sh.sort.place + tid * kPer);
      static_assert(kPer == 4, "cells per thread");
      const int sum = c.x + c.y + c.z + c.w;
      int incl = sum;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int v = __shfl_up_sync(0xFFFFFFFFu, incl, off);
        if (lane >= off) incl += v;
      }
      if (lane == 31) sh.sort.tot[warp] = incl;
      __syncthreads();
      int before = sh.sort.tot[lane];
      before = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? before : 0);
      before += incl - sum;
      const int4 f = make_int4(before, before + c.x, before + c.x + c.y, before + c.x + c.y + c.z);
      *reinterpret_cast<int4*>(sh.sort.place + tid * kPer) = f;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kRows; ++j) {
      const uint32_t v[4] = {q[j].x, q[j].y, q[j].z, q[j].w};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int p = atomicAdd(place_of(v[k]), 1);      // the order within a cell does not matter: sums are exact
        sh.vec[p] = v[k];
        sh.sort.pos[p] = (uint16_t)((warp + j * kLloydWarps) * 128 + lane * 4 + k);
      }
    }
    __syncthreads();
#pragma unroll
    for (int g = 0; g < 32; g += 2) pos[g / 2] = sh.sort.pos[warp * 1024 + g * 32 + lane] | (uint32_t)sh.sort.pos[warp * 1024 + (g + 1) * 32 + lane] << 16;
    __syncthreads();
  }
  Box box;                                       // of group number tid
  {
    float x0 = INFINITY, x1 = -INFINITY, y0 = INFINITY, y1 = -INFINITY;
#pragma unroll 8
    for (int k = 0; k < 32; ++k) {
      const float2 f = vec_of(sh.vec[tid * 32 + ((k + lane) & 31)]);
      x0 = fminf(x0, f.x); x1 = fmaxf(x1, f.x); y0 = fminf(y0, f.y); y1 = fmaxf(y1, f.y);
    }
    box.set(x0, x1, y0, y1);
  }
  uint32_t* aux = a.aux + (size_t)tile * E;
  auto& s = sh.it;
  for (int e = tid; e < kVqMaxE; e += kLloydThreads) {
#pragma unroll
    for (int p = 0; p < 3; ++p) s.sums.x[p][e] = s.sums.y[p][e] = 0;
    s.sums.cnt[e] = 0;
    if (e < E) {
      const float2 c = vec_of(aux[e]);
      s.cx[e] = (double)c.x; s.cy[e] = (double)c.y;
      s.set_centre(e, c.x, c.y);
    }
  }
  if (tid == 0) s.moved = 0;
  __syncthreads();
  int near = -1, owner = -1;
  for (int it = 0; it < a.iters; ++it) {
    build_list<EW>(sh, box, tid, near, owner, it > 0);
    __syncthreads();
    // lane j holds the list of the j-th group of this warp's turn
    const uint4 entry = s.list[lane * kLloydWarps + warp];
    uint32_t todo = __ballot_sync(0xFFFFFFFFu, (entry.w >> 24) != kListSame);
    bool moved = it == 0;
    int queued = 0;                              // moves of this warp not yet in the sums
    uint32_t* queue = s.moves[warp];
    auto flush = [&](int count) {
      __syncwarp();
      if (lane < count) {
        const uint32_t m = queue[lane];
        const uint32_t v = sh.vec[m >> 16];
        move_member(s.sums, v, (int)((m >> 8) & 0xFFu), -1);
        move_member(s.sums, v, (int)(m & 0xFFu), 1);
      }
      __syncwarp();
    };
    for (; todo; todo &= todo - 1u) {
      const int j = __ffs((int)todo) - 1, g = j * kLloydWarps + warp, p = g * 32 + lane;
      const uint32_t q = sh.vec[p];
      const int was = it > 0 ? (int)s.idx[p] : 0;
      const float2 f = vec_of(q);
      float best = INFINITY;
      int bi = 0;
      const uint4 e16 = make_uint4(__shfl_sync(0xFFFFFFFFu, entry.x, j), __shfl_sync(0xFFFFFFFFu, entry.y, j), __shfl_sync(0xFFFFFFFFu, entry.z, j), __shfl_sync(0xFFFFFFFFu, entry.w, j));
      over_list<E>(e16, [&](uint32_t e0, uint32_t e1) {
        const float d0 = d2f(f.x, f.y, s.centre(e0)), d1 = d2f(f.x, f.y, s.centre(e1));
        if (d0 < best) { best = d0; bi = (int)e0; }
        if (d1 < best) { best = d1; bi = (int)e1; }
      });
      if (it == 0) {
        s.idx[p] = (uint8_t)bi;
        continue;
      }
      // the vectors that moved are queued and taken 32 at a time: a few lanes of every warp would otherwise walk
      // the whole update for every group
      const uint32_t who = __ballot_sync(0xFFFFFFFFu, bi != was);
      if (who == 0u) continue;
      moved = true;
      if (bi != was) {
        s.idx[p] = (uint8_t)bi;
        queue[queued + __popc(who & ((1u << lane) - 1u))] = (uint32_t)p << 16 | (uint32_t)was << 8 | (uint32_t)bi;
      }
      queued += __popc(who);
      if (queued >= 32) {
        flush(32);
        queued -= 32;
        const uint32_t m = queue[32 + lane];
        __syncwarp();
        if (lane < queued) queue[lane] = m;
      }
    }
    flush(queued);
    if (it == 0) {
      __syncthreads();
      join_group(s.sums, sh.vec + tid * 32, s.idx + tid * 32, lane);
    }
    if (moved && lane == 0) s.moved = it + 1;
    __syncthreads();
    if (s.moved != it + 1) break;                // the centres would stay as they are in every further iteration
    for (int e = tid; e < E; e += kLloydThreads) {
      const int cnt = s.sums.cnt[e];
      if (cnt) {
        s.cx[e] = mean_of_pieces(s.sums.x, e, cnt); s.cy[e] = mean_of_pieces(s.sums.y, e, cnt);
        s.set_centre(e, (float)s.cx[e], (float)s.cy[e]);
      }
    }
    __syncthreads();
  }
  // ---- centres to fp16; final assignment against the rounded centres in fp64 (exact differences,
  // products and sum each rounded once, in this order; the lowest index wins ties)
  for (int e = tid; e < E; e += kLloydThreads) {
    const __half hx = __double2half(s.cx[e]), hy = __double2half(s.cy[e]);
    s.cx[e] = (double)__half2float(hx); s.cy[e] = (double)__half2float(hy);
    s.set_centre(e, __half2float(hx), __half2float(hy));
    aux[e] = (uint32_t)__half_as_ushort(hx) | ((uint32_t)__half_as_ushort(hy) << 16);
  }
  __syncthreads();
  build_list<EW>(sh, box, tid, near, owner, false);
  __syncthreads();
  for (int g = warp; g < kGroups; g += kLloydWarps) {
    const int p = g * 32 + lane;
    const float2 f = vec_of(sh.vec[p]);
    const uint4 entry = s.list[g];
    int bi = (int)(entry.x & 0xFFu);
    if ((entry.w >> 24) != 1u) {
      const double x = (double)f.x, y = (double)f.y;
      double best = INFINITY;
      over_list<E>(entry, [&](uint32_t e0, uint32_t e1) {
        const double dx0 = x - s.cx[e0], dy0 = y - s.cy[e0], dx1 = x - s.cx[e1], dy1 = y - s.cy[e1];
        const double d0 = __dadd_rn(__dmul_rn(dx0, dx0), __dmul_rn(dy0, dy0)), d1 = __dadd_rn(__dmul_rn(dx1, dx1), __dmul_rn(dy1, dy1));
        if (d0 < best) { best = d0; bi = (int)e0; }
        if (d1 < best) { best = d1; bi = (int)e1; }
      });
    }
    s.idx[p] = (uint8_t)bi;
  }
  __syncthreads();
  // back to the order of the matrix; the vectors are not needed any more
  uint8_t* idx = reinterpret_cast<uint8_t*>(sh.vec);
#pragma unroll
  for (int g = 0; g < 32; ++g) idx[(pos[g / 2] >> (16 * (g & 1))) & 0xFFFFu] = s.idx[warp * 1024 + g * 32 + lane];
  __syncthreads();
  // ---- bit packing (format.h)
  if (warp < 16) {
    const int gr = lane >> 2, t = lane & 3;
    constexpr int kBits = EW == 2 ? 6 : 8;
    const int mb = tr * 2 + (warp >> 3), rt = warp & 7;
    uint8_t* out = a.payload + (((size_t)mb * a.TC + tc) * 8 + rt) * rwkvq_vq_record_bytes(kBits);
    vq_pack_lane<kBits>(idx, warp, gr, t, lane, out);
  }
}

// ---- token-shift vectors ----
//
// Weighted vectors are assigned by a cluster of kVecCluster, whose blocks take a part of the vectors each and
// write what they find into the first block's shared memory; that block sorts the members by centre (stable), and every centre
// adds its own in vector order.  Bound by the latency of the running sums: of the seeds' distances and of the longest
// centre's members.  2048 weighted vectors, 64 centres, ten iterations: 145 us with the seeds (237 before: one block for
// everything, seeds' distances in shared memory, two compare-and-selects for each distance, members counted and ranked
// twice by match, sums in chains of dependent loads and conversions, the final distances all in fp64).
constexpr int kVecThreads = 1024, kVecCluster = 8;
// The search for the nearest centre takes the minimum over groups of eight centres, one instruction a distance, and looks for the centre only
// in the group that wins.  One slot of padding per group: lanes that look in different groups read different banks.
constexpr int kCentreGroup = 8;
__host__ __device__ constexpr int centre_slot(int e) { return e + e / kCentreGroup; }
struct VecShared {
  double cx[kVqMaxE], cy[kVqMaxE];
  float4 neg[kVqMaxE + kVqMaxE / kCentreGroup];   // (-x, -x, -y, -y) of a centre, in groups, see centre_slot
  uint16_t hist[kVecThreads / 32][kVqMaxE + 2];   // members per warp's share and centre, then those of the shares before it; a column is read by a warp
  int first[kVqMaxE + 1];
  ClusterSums sums;
  float part_best[kVecCluster][64 * kVecThreads / 32 / kVecCluster];     // nearest centre of a part of them: distance, number
  uint8_t part_idx[kVecCluster][64 * kVecThreads / 32 / kVecCluster];
};
// Up to this many vectors the first block keeps, in fp64, w * v and w of either dimension: a conversion to fp64 takes four times a
// multiply-add's time, and a member of a centre is converted once instead of in each iteration.
constexpr int kVecTable = 4096;
__host__ __device__ constexpr size_t vec_smem_bytes(int n) {
  const size_t rows = ((size_t)n + 63) / 64;
  return (sizeof(VecShared) + 15) / 16 * 16 + rows * 320 + (n <= kVecTable ? (size_t)n * 32 : 0);
}

// The cluster: barrier, and stores to the shared memory of a block of it at the address that `local` has here.
__device__ __forceinline__ uint32_t cluster_rank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ uint32_t cluster_size() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ void cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t peer_address(const void* local, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(local)), "r"(rank));
  return r;
}
__device__ __forceinline__ void peer_store8(uint32_t at, uint32_t v) { asm volatile("st.shared::cluster.u8 [%0], %1;" ::"r"(at), "r"(v) : "memory"); }
__device__ __forceinline__ void peer_store16(uint32_t at, uint32_t v) { asm volatile("st.shared::cluster.u16 [%0], %1;" ::"r"(at), "h"((uint16_t)v) : "memory"); }
__device__ __forceinline__ void peer_store(uint32_t at, float4 v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(at), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void peer_store(uint32_t at, double v) { asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(at), "d"(v) : "memory"); }

// Two vectors against all centres, distances rounded as d = w.x * (dx * dx) + (w.y * (dy * dy)) with the last product and sum in one
// rounding (unweighted: dx * dx + (dy * dy), likewise).
struct Nearest {
  float best[2], second[2];     // smallest minimum of a group, and of the other groups
  int group[2];                 // first centre of the first group with that minimum
};
__device__ __forceinline__ float2 pair_distance(bool weighted, float2 x, float2 y, float2 wx, float2 wy, float4 c) {
  const float2 dx = add2(x, make_float2(c.x, c.y)), dy = add2(y, make_float2(c.z, c.w)), yy = mul2(dy, dy);
  return weighted ? fma2(wx, mul2(dx, dx), mul2(wy, yy)) : fma2(dx, dx, yy);
}
__device__ __forceinline__ Nearest nearest_group(const float4* neg, int E, bool weighted, float2 x, float2 y, float2 wx, float2 wy) {
  Nearest r;
#pragma unroll
  for (int q = 0; q < 2; ++q) { r.best[q] = r.second[q] = INFINITY; r.group[q] = 0; }
#pragma unroll 1
  for (int e = 0; e < E; e += kCentreGroup) {
    float2 m = make_float2(INFINITY, INFINITY);
#pragma unroll
    for (int k = 0; k < kCentreGroup; ++k) {
      const float2 d = pair_distance(weighted, x, y, wx, wy, neg[centre_slot(e) + k]);
      m = make_float2(fminf(m.x, d.x), fminf(m.y, d.y));
    }
    const float mm[2] = {m.x, m.y};
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      r.second[q] = fminf(r.second[q], fmaxf(r.best[q], mm[q]));
      if (mm[q] < r.best[q]) { r.best[q] = mm[q]; r.group[q] = e; }
    }
  }
  return r;
}
__device__ __forceinline__ float one_distance(bool weighted, float x, float y, float wx, float wy, float4 c) {
  const float dx = __fadd_rn(x, c.x), dy = __fadd_rn(y, c.z), yy = __fmul_rn(dy, dy);
  return weighted ? __fmaf_rn(wx, __fmul_rn(dx, dx), __fmul_rn(wy, yy)) : __fmaf_rn(dx, dx, yy);
}

__global__ void __launch_bounds__(kVecThreads, 1) vq_vector_kernel(const VqArgs a, const __grid_constant__ rwkvq_image_header head, uint8_t* image) {
  extern __shared__ __align__(16) uint8_t smem[];
  VecShared& sh = *reinterpret_cast<VecShared*>(smem);
  uint8_t* rest = smem + (sizeof(VecShared) + 15) / 16 * 16;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = a.n_vec, E = a.E, rows = (n + 63) / 64;
  const bool weighted = a.elem_w != nullptr;
  const uint32_t* vec = reinterpret_cast<const uint32_t*>(a.w);
  const float2* wgt = reinterpret_cast<const float2*>(a.elem_w);
  const uint32_t rank = cluster_rank(), peers = cluster_size();
  const bool lead = rank == 0u;
  if (lead) write_header(head, image);
  for (int e = E + tid; e < (E + kCentreGroup - 1) / kCentreGroup * kCentreGroup; e += kVecThreads)      // no centre is nearer than these
    sh.neg[centre_slot(e)] = make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
  // tables of the first block, behind the assignment (bytes), the ranks of the members and the members sorted by centre (16-bit numbers)
  const bool tables = n <= kVecTable;
  double2* const table_wv = reinterpret_cast<double2*>(rest + (size_t)rows * 320);      // [n] w * v
  double2* const table_w = table_wv + n;
  uint8_t* idx = rest;                                             // [rows * 64]
  if (lead) {
    if (tables && weighted) {
      for (int i = tid; i < n; i += kVecThreads) {
        const uint32_t v = __ldg(vec + i);
        const float2 wi = __ldg(wgt + i);
        const double wx = (double)wi.x, wy = (double)wi.y;
        table_w[i] = make_double2(wx, wy);
        table_wv[i] = make_double2(wx * (double)h2f_bits(v & 0xFFFFu), wy * (double)h2f_bits(v >> 16));      // exact: 24 and 11 bits
      }
    }
    // the seeds lie where the codebook will
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int e = tid; e < E; e += kVecThreads) {
      const float2 c = vec_of(__ldcg(a.aux + e));
      sh.cx[e] = (double)c.x; sh.cy[e] = (double)c.y;
    }
    __syncthreads();
  }
  uint16_t* ranks = reinterpret_cast<uint16_t*>(rest + rows * 64);   // [rows * 64]: members of the same centre before it in the warp's share
  uint16_t* sorted = ranks + rows * 64;                             // [rows * 64]
  // Negated centres, in fp32, to every block.
  auto publish = [&]() {
    for (int k = tid; k < E * (int)peers; k += kVecThreads) {
      const int e = k % E;
      const float cx = (float)sh.cx[e], cy = (float)sh.cy[e];
      peer_store(peer_address(&sh.neg[centre_slot(e)], (uint32_t)(k / E)), make_float4(-cx, -cx, -cy, -cy));
    }
  };
  // ---- Lloyd iterations.  Share k of the vectors is [k * share, (k + 1) * share), taken 64 at a time by the warps of block
  // k / shares that have this share, each with a part of the centres; the first of them goes on with the nearest of all.
  constexpr int kShares = kVecThreads / 32;
  const int share = ((n + kVecThreads - 1) / kVecThreads) * 32, shares = kShares / (int)peers, parts = (int)peers, part = warp / shares, mine = (int)rank * shares + warp % shares;
  const int part_e0 = E * part / parts, part_e1 = E * (part + 1) / parts;
  const uint32_t lead_idx = peer_address(idx, 0u), lead_ranks = peer_address(ranks, 0u);
  uint16_t* const hist = sh.hist[mine];
  uint32_t v[2];
  float2 wv[2] = {make_float2(1.f, 1.f), make_float2(1.f, 1.f)};
  auto fetch = [&](int i0) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int i = min(i0 + 32 * q + lane, n - 1);
      v[q] = __ldg(vec + i);
      if (weighted) wv[q] = __ldg(wgt + i);
    }
  };
  fetch(mine * share);                             // a share of 64 stays in registers
  cluster_sync();                                  // every block runs: their shared memory may be written
  if (lead) publish();
  for (int it = 0; it < a.iters; ++it) {
    if (!weighted) {
      for (int e = tid; e < E; e += kVecThreads) {
#pragma unroll
        for (int p = 0; p < 3; ++p) sh.sums.x[p][e] = sh.sums.y[p][e] = 0;
        sh.sums.cnt[e] = 0;
      }
    }
    if (part == 0) for (int e = lane; e < E; e += 32) hist[e] = 0;
    cluster_sync();
    for (int i0 = mine * share; i0 < min(n, (mine + 1) * share); i0 += 64) {
      // two vectors per lane: the packed operations take both
      const int i[2] = {i0 + lane, i0 + 32 + lane};
      const int stop = min(n, (mine + 1) * share);
      if (share > 64) fetch(i0);
      const float2 f0 = vec_of(v[0]), f1 = vec_of(v[1]);
      const float2 x = make_float2(f0.x, f1.x), y = make_float2(f0.y, f1.y), wx = make_float2(wv[0].x, wv[1].x), wy = make_float2(wv[0].y, wv[1].y);
      float best[2] = {INFINITY, INFINITY};
      int bi2[2] = {0, 0};
#pragma unroll 8
      for (int e = part_e0; e < part_e1; ++e) {
        const float2 d = pair_distance(weighted, x, y, wx, wy, sh.neg[centre_slot(e)]);
        if (d.x < best[0]) { best[0] = d.x; bi2[0] = e; }
        if (d.y < best[1]) { best[1] = d.y; bi2[1] = e; }
      }
      if (parts > 1) {
        const int at = (warp % shares) * 64 + lane;
#pragma unroll
        for (int q = 0; q < 2; ++q) { sh.part_best[part][at + 32 * q] = best[q]; sh.part_idx[part][at + 32 * q] = (uint8_t)bi2[q]; }
        asm volatile("bar.sync %0, %1;" ::"r"(2 + warp % shares), "r"(32 * parts) : "memory");
        if (part == 0) {
#pragma unroll
          for (int k = 1; k < kVecCluster; ++k)      // parts in the order of their centres: the first of equal distances stays
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              const float b = sh.part_best[k][at + 32 * q];
              const int e = sh.part_idx[k][at + 32 * q];
              if (b < best[q]) { best[q] = b; bi2[q] = e; }
            }
        }
        if (share > 64) asm volatile("bar.sync %0, %1;" ::"r"(2 + warp % shares), "r"(32 * parts) : "memory");
        if (part != 0) continue;
      }
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int bi = bi2[q];
        const bool in = i[q] < stop;
        if (in) peer_store8(lead_idx + (uint32_t)i[q], (uint32_t)bi);
        if (!weighted) {
          if (in) move_member(sh.sums, v[q], bi, 1);
        } else {
          const unsigned live = __ballot_sync(0xFFFFFFFFu, in);
          if (in) {
            const unsigned same = __match_any_sync(live, bi), below = same & ((1u << lane) - 1u);
            const int before = hist[bi];
            __syncwarp(live);
            peer_store16(lead_ranks + 2u * (uint32_t)i[q], (uint32_t)(before + __popc(below)));
            if (below == 0u) hist[bi] = (uint16_t)(before + __popc(same));
          }
          __syncwarp();
        }
      }
    }
    if (weighted && !lead && part == 0) {
      const uint32_t to = peer_address(hist, 0u);
      for (int e = lane; e < E; e += 32) peer_store16(to + 2u * (uint32_t)e, hist[e]);
    }
    cluster_sync();
    if (!lead) continue;
    if (!weighted) {
      for (int e = tid; e < E; e += kVecThreads) {
        const int cnt = sh.sums.cnt[e];
        if (cnt) { sh.cx[e] = mean_of_pieces(sh.sums.x, e, cnt); sh.cy[e] = mean_of_pieces(sh.sums.y, e, cnt); }
      }
    } else {
      // weighted means of Eq. 19, per dimension, members added in vector order: a stable sort by centre, then one thread
      // per centre and dimension
      for (int e = warp; e < E; e += kVecThreads / 32) {      // lane = share
        const int mine = sh.hist[lane][e];
        int s = mine;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const int o = __shfl_up_sync(0xFFFFFFFFu, s, off);
          if (lane >= off) s += o;
        }
        sh.hist[lane][e] = (uint16_t)(s - mine);
        if (lane == 31) sh.first[e + 1] = s;
      }
      __syncthreads();
      if (warp == 0) {
        int carry = 0;
        for (int e0 = 0; e0 < E; e0 += 32) {
          int s = e0 + lane < E ? sh.first[e0 + lane + 1] : 0;
#pragma unroll
          for (int off = 1; off < 32; off <<= 1) {
            const int o = __shfl_up_sync(0xFFFFFFFFu, s, off);
            if (lane >= off) s += o;
          }
          if (e0 + lane < E) sh.first[e0 + lane + 1] = carry + s;
          carry += __shfl_sync(0xFFFFFFFFu, s, 31);
        }
        if (lane == 0) sh.first[0] = 0;
      }
      __syncthreads();
      for (int i = warp * share + lane; i < min(n, (warp + 1) * share); i += 32) {
        const int e = idx[i];
        sorted[sh.first[e] + sh.hist[warp][e] + ranks[i]] = (uint16_t)i;
      }
      __syncthreads();
      // four threads a centre: the sums of w * v and of w, of either dimension
      for (int k = tid; k < 4 * E; k += kVecThreads) {
        const int e = k >> 2, dim = k & 1;
        const bool den = (k & 2) != 0;
        double sum = 0.0;
        const int stop = sh.first[e + 1];
        // eight members at a time; past the end the last one again, times zero
        if (tables) {
          const double* table = reinterpret_cast<const double*>(den ? table_w : table_wv) + dim;
          for (int j = sh.first[e]; j < stop; j += 8) {
            double v[8];
#pragma unroll
            for (int m = 0; m < 8; ++m) {
              v[m] = table[2 * sorted[min(j + m, stop - 1)]];
              if (j + m >= stop) v[m] = 0.0;
            }
#pragma unroll
            for (int m = 0; m < 8; ++m) sum += v[m];
          }
        } else {
          for (int j = sh.first[e]; j < stop; j += 8) {
            float wi[8], f[8];
#pragma unroll
            for (int m = 0; m < 8; ++m) {
              const int i = sorted[min(j + m, stop - 1)];
              wi[m] = j + m < stop ? __ldg(a.elem_w + 2 * i + dim) : 0.f;
              f[m] = den ? 1.f : h2f_bits(__ldg(a.w + 2 * i + dim));
            }
#pragma unroll
            for (int m = 0; m < 8; ++m) sum = fma((double)wi[m], (double)f[m], sum);      // the product of 24 and 11 bits is exact
          }
        }
        const unsigned four = 0xFu << (lane & 28);
        const double weight = __shfl_xor_sync(four, sum, 2);
        if (!den && weight > 0.0) (dim ? sh.cy : sh.cx)[e] = sum / weight;
      }
    }
    __syncthreads();
    publish();
  }
  // ---- centres to fp16; final assignment against the rounded centres in fp64
  cluster_sync();                                  // the last centres are no longer being written
  if (lead) {
    for (int e = tid; e < E; e += kVecThreads) {
      const __half hx = __double2half(sh.cx[e]), hy = __double2half(sh.cy[e]);
      const float cx = __half2float(hx), cy = __half2float(hy);
      a.aux[e] = (uint32_t)__half_as_ushort(hx) | ((uint32_t)__half_as_ushort(hy) << 16);
      for (uint32_t r = 0; r < peers; ++r) {
        peer_store(peer_address(&sh.neg[centre_slot(e)], r), make_float4(-cx, -cx, -cy, -cy));
        peer_store(peer_address(&sh.cx[e], r), (double)cx);
        peer_store(peer_address(&sh.cy[e], r), (double)cy);
      }
    }
  }
  cluster_sync();
  // In fp32 first: a distance is wrong by less than seven roundings there, so a centre whose distance is smallest by more than 2^-20 of it is
  // the nearest in fp64 too, and so is one that the vector equals.  The others (and distances near the end of fp32's range) are taken in fp64.
  const int stride = (int)peers * kVecThreads;
  for (int i0 = (int)rank * kVecThreads + tid; i0 < n; i0 += 2 * stride) {
    const int i[2] = {i0, i0 + stride};
    float2 f[2], wv[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      f[q] = vec_of(__ldg(vec + min(i[q], n - 1)));
      wv[q] = weighted ? __ldg(wgt + min(i[q], n - 1)) : make_float2(1.f, 1.f);
    }
    const Nearest nr = nearest_group(sh.neg, E, weighted, make_float2(f[0].x, f[1].x), make_float2(f[0].y, f[1].y), make_float2(wv[0].x, wv[1].x),
                                     make_float2(wv[0].y, wv[1].y));
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if (i[q] >= n) break;
      const float limit = nr.best[q] * (1.f + 1.f / 1048576.f);
      const float4* c = sh.neg + centre_slot(nr.group[q]);
      int k = 0, close = 0;
#pragma unroll
      for (int j = 0; j < kCentreGroup; ++j)
        if (one_distance(weighted, f[q].x, f[q].y, wv[q].x, wv[q].y, c[j]) <= limit) { k = j; ++close; }
      int bi = nr.group[q] + k;
      const bool equal = f[q].x + c[k].x == 0.f && f[q].y + c[k].z == 0.f;
      if (close != 1 || !(nr.second[q] > limit) || !(equal || (nr.best[q] > 1e-30f && nr.best[q] < 1e30f))) {
        const double x = (double)f[q].x, y = (double)f[q].y, wx = (double)wv[q].x, wy = (double)wv[q].y;
        double best = INFINITY;
        bi = 0;
#pragma unroll 4
        for (int e = 0; e < E; ++e) {
          const double dx = x - sh.cx[e], dy = y - sh.cy[e];
          const double d = weighted ? __dadd_rn(__dmul_rn(wx, __dmul_rn(dx, dx)), __dmul_rn(wy, __dmul_rn(dy, dy)))
                                    : __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
          if (d < best) { best = d; bi = e; }
        }
      }
      peer_store8(lead_idx + (uint32_t)i[q], (uint32_t)bi);
    }
  }
  cluster_sync();
  if (!lead) return;
  const int bits = a.bits, n_words = (int)(((((size_t)n * bits + 7) / 8 + 15) / 16 * 16) / 4);
  for (int wi = tid; wi < n_words; wi += kVecThreads) {
    uint32_t val = 0u;
    const int lo_bit = 32 * wi;
    for (int nn = lo_bit / bits; nn < n && nn * bits < lo_bit + 32; ++nn) {
      const int shft = nn * bits - lo_bit;
      val |= shft >= 0 ? (uint32_t)idx[nn] << shft : (uint32_t)idx[nn] >> (-shft);
    }
    reinterpret_cast<uint32_t*>(a.payload)[wi] = val;
  }
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
  for (int i = threadIdx.x; i < S * 8; i += 256) {
    const int s = i >> 3, c = i & 7;
    tile[s * 9 + c] = (j0 + c < a.n) ? __ldg(a.samples + (size_t)s * a.n + j0 + c) : 0.f;
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

}  // namespace
}  // namespace rwkvq

extern "C" {

size_t rwkvq_quantize_workspace_bytes(void) { return 256; }

static rwkvq_status quantize_enqueue(const void* w_dev, int oc, int ic, const rwkvq_quant_cfg* cfg, const float* elem_weight_dev,
                                     void* image_dev, size_t image_bytes, rwkvq_desc* desc_out, void* workspace_dev,
                                     size_t workspace_bytes, void* stream, bool clear_flag) {
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
    sq_quantize_kernel<<<MB * KT, 256, 0, s>>>(static_cast<const uint16_t*>(w_dev), oc, ic, KT, img + h.off_payload, flags, h, img);
  } else {
    VqArgs a;
    a.w = static_cast<const uint16_t*>(w_dev);
    a.elem_w = elem_weight_dev;
    a.ic = ic;
    a.TC = is_vector ? 1 : ic / 256;
    a.n_vec = is_vector ? ic / 2 : kVqMaxVec;
    a.bits = d.bits; a.E = d.entries; a.iters = cfg->kmeans_iters;
    a.seed = cfg->seed;
    a.payload = img + h.off_payload;
    a.aux = reinterpret_cast<uint32_t*>(img + h.off_aux);
    a.flags = flags;
    static SmemOptIn opt_in_seed, opt_in_64, opt_in_256, opt_in_vector, opt_in_vector_seed;
    if (is_vector) {
      const int seed_threads = (a.n_vec + 2047) / 2048 * 32;
      e = opt_in_vector_seed((const void*)vq_seed_kernel<true>, kVqMaxVec * 4 + (int)sizeof(SeedShared));
      if (e != cudaSuccess) return cuda_status(e);
      vq_seed_kernel<true><<<1, seed_threads, (size_t)seed_threads * kVqPerThread * 4 + sizeof(SeedShared), s>>>(a);
      e = opt_in_vector((const void*)vq_vector_kernel, (int)std::max(vec_smem_bytes(kVqMaxVec), vec_smem_bytes(kVecTable)));
      if (e != cudaSuccess) return cuda_status(e);
      // the exact sums of an unweighted vector are atomics in one block's shared memory
      cudaLaunchConfig_t cfg_v = {};
      cfg_v.gridDim = dim3(a.elem_w ? kVecCluster : 1); cfg_v.blockDim = dim3(kVecThreads); cfg_v.dynamicSmemBytes = vec_smem_bytes(a.n_vec); cfg_v.stream = s;
      cudaLaunchAttribute attr[2];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = cfg_v.gridDim.x; attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
      attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;      // starts while the seeds are drawn
      attr[1].val.programmaticStreamSerializationAllowed = 1;
      cfg_v.attrs = attr; cfg_v.numAttrs = 2;
      e = cudaLaunchKernelEx(&cfg_v, vq_vector_kernel, (const VqArgs)a, (const rwkvq_image_header)h, img);
      if (e != cudaSuccess) return cuda_status(e);
    } else {
      constexpr size_t seed_smem = (size_t)kVqMaxVec * 4 + sizeof(SeedShared);
      const int tiles = (oc / 256) * (ic / 256);
      e = opt_in_seed((const void*)vq_seed_kernel<false>, (int)seed_smem);
      if (e != cudaSuccess) return cuda_status(e);
      vq_seed_kernel<false><<<tiles, kVqThreads, seed_smem, s>>>(a);
      if (d.entries == 64) {
        e = opt_in_64((const void*)vq_lloyd_kernel<2>, (int)sizeof(LloydShared));
        if (e != cudaSuccess) return cuda_status(e);
        vq_lloyd_kernel<2><<<tiles, kLloydThreads, sizeof(LloydShared), s>>>(a, h, img);
      } else {
        e = opt_in_256((const void*)vq_lloyd_kernel<8>, (int)sizeof(LloydShared));
        if (e != cudaSuccess) return cuda_status(e);
        vq_lloyd_kernel<8><<<tiles, kLloydThreads, sizeof(LloydShared), s>>>(a, h, img);
      }
    }
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
  int host_flags = 0;
  cudaError_t e = cudaMemcpyAsync(&host_flags, workspace_dev, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(workspace_dev, 0, sizeof(int), s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_status(e);
  return (host_flags & kFlagNonFinite) ? RWKVQ_ENONFINITE : RWKVQ_OK;
}

rwkvq_status rwkvq_quantize_dev_async(const void* w_dev, int oc, int ic, const rwkvq_quant_cfg* cfg, const float* elem_weight_dev,
                                      void* image_dev, size_t image_bytes, rwkvq_desc* desc_out, void* workspace_dev,
                                      size_t workspace_bytes, void* stream) {
  return quantize_enqueue(w_dev, oc, ic, cfg, elem_weight_dev, image_dev, image_bytes, desc_out, workspace_dev,
                          workspace_bytes, stream, false);
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
  const dim3 grid((n + 7) / 8);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (n_samples <= 32) representative_kernel<1><<<grid, 256, smem, st>>>(a);
  else if (n_samples <= 64) representative_kernel<2><<<grid, 256, smem, st>>>(a);
  else if (n_samples <= 128) representative_kernel<4><<<grid, 256, smem, st>>>(a);
  else if (n_samples <= 256) representative_kernel<8><<<grid, 256, smem, st>>>(a);
  else if (n_samples <= 512) representative_kernel<16><<<grid, 256, smem, st>>>(a);
  else representative_kernel<32><<<grid, 256, smem, st>>>(a);
  return cuda_status(cudaGetLastError());
}

}  // extern "C"
