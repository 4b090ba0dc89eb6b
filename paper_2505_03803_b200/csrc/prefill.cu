// Prefill product Y[t][i] = sum_j bf16(w_hat[i][j]) * x_mix[t][j] on the tcgen05 tensor cores.
//
// (1) A pre-pass applies the token-shift mix of Appendix A.1 Eq. 20 along the
// sequence (x_mix[t] = X[t] + (X[t-1] - X[t]) (.) mu_hat, X[-1] = xprev0), rounds to bf16 and
// writes the result tile by tile in the shared-memory operand layout of the tensor core (tiles of
// NT tokens x 64 columns, 128-byte rows, 128-byte swizzle), so that the main kernel fetches an
// operand tile with ONE bulk asynchronous copy; products without a token shift skip it, their
// tiles are tensor-map copies straight from X.
// (2) ONE persistent launch, one CTA per SM, covers every product of the call
// (rwkvq_gemm_prefill_grouped; the single product is a group of one).  It starts while the
// pre-pass runs (programmatic dependent launch): the first weights are dequantised meanwhile.
// Output tiles of 128 weight rows (one chunk row of the packed image) x NT tokens, the tokens
// divided evenly over as many tiles of at most kTileTokens as they need, are handed out by an
// atomic ticket, longest contraction first, so tiles of different products balance:
//   * a producer thread draws the ticket, publishes the tile to the other roles through a small
//     queue, and streams the packed chunks (12-17 KB per 256 columns, as many slots as fit: two to
//     four) with cp.async.bulk + mbarrier transactions: it runs ahead of all others, so that the
//     ticket's trip and the first weights of the next tile are under way while this tile is worked
//     on (drawn by the activation producer they were not: 3 to 6 % of a call); a second producer
//     thread streams activation tiles (up to 26 KB per 64 columns, six stages) into shared memory;
//   * sixteen dequantisation warps in two groups (group g takes the 64-column blocks of parity g,
//     one warp per 16-row record) turn packed codes into bf16, exactly bf16_rne of the fp32
//     rounding of s * (q - z) or of the codebook entry, and store them in TENSOR MEMORY, a ring of
//     three blocks: the packed layout's registers are the fragments that tcgen05.st.16x256b takes,
//     so that a record's 64 columns are one instruction.  (In shared memory, written and read back
//     by the tensor core, the weights took a third of its 128 bytes per cycle: 960 cycles a block.)
//   * one warp issues tcgen05.mma (A = weights 128 x 16 from tensor memory, B = activations NT x 16,
//     fp32 accumulators in tensor memory: two stages of up to 208 columns) and commits to mbarriers;
//   * four epilogue warps read an accumulator stage with tcgen05.ld (lane = weight row, so a warp
//     writes 32 consecutive outputs of one token) while the tensor core fills the other stage
//     with the next tile.
// (3) Long contractions with few tiles are cut into slices, which leave their sums in the workspace;
// a third launch adds them up in order.
// What bounds it: with many tokens the instructions of the dequantisation warps beside the tensor core's 4 * NT / 2 cycles per
// 64-column block (about 500 cycles a block at NT = 208, where the tensor pipe needs 417: busy 72 % of prefill_kernel's time), and in a loop of
// seconds the power limit (1417 instead of 1965 MHz).  With few tokens the parts around the blocks: of d 2048, 203 tokens the pre-pass takes
// 5 us, prefill_kernel 30, of which its blocks would fill 11.5 on evenly loaded SMs, and adding up the slices 8, partly in each other's shadow.
// Eight projections of one layer, before -> now: d 4096, 2048 tokens 991 -> 829 us in a loop, 852 -> 722 ten calls from idle;
// d 2048, 203 tokens 88.8 -> 37; d 512, 21 tokens 34 -> 16; d 640, 1783 tokens 54 -> 41; d 1280, 1464 tokens 112 -> 70.
// Every wait is bounded; a wait that gives up raises the device status word and all roles leave
// through the common exit, where tensor memory is freed.
#include <cuda.h>           // tensor map types (no driver symbol is linked)
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>

#include "../../include/rwkvq.h"
#include "format.h"
#include "host_util.h"
#include "unpack.cuh"

namespace rwkvq {

int* device_status_ptr();  // api_misc.cu

namespace pf {

constexpr int kTileTokens = 208, kTileRows = 128, kKBlock = 64;     // at most; see the layout of tensor memory
// Rings: activation tiles (shared memory) and dequantised weight blocks (tensor memory).  Block kb has ONE barrier for both operands and one
// for both places, those of its activation stage: the warp that issues the tensor-core instructions waits and commits once a block.
constexpr int kXStages = 6, kWStages = 3;
static_assert(kXStages % kWStages == 0, "a weight place always belongs to the same activation stages");
constexpr uint32_t kXTileBytes = kTileTokens * kKBlock * 2;   // 26 KB: activations of one stage
constexpr int kMaxPackedSlots = 4;                            // packed chunk (+ codebook) slots: as many as fit, at least two
constexpr int kRecordWarps = 8, kDequantGroups = 2, kDequantWarps = kRecordWarps * kDequantGroups, kEpilogueWarps = 4;
constexpr uint32_t kBookBytes = 1024;                         // a warp's codebook: up to 256 pairs
constexpr uint32_t kCtrlBytes = 1024;
constexpr uint32_t kFixedSmemBytes = kCtrlBytes + kXStages * kXTileBytes + kDequantWarps * kBookBytes + 1024;  // + alignment slack
constexpr uint32_t kMaxSmemBytes = 232448;                    // per-CTA limit of the architecture
constexpr int kThreads = 32 * (3 + kDequantWarps + kEpilogueWarps);   // + activation producer, tensor-core issue, chunk producer
constexpr uint32_t kPollLimit = 1u << 22;
// Tensor memory: two accumulator stages of kTileTokens columns, then the weight ring (64 bf16 columns = 32 words per block).
constexpr uint32_t kTmemCols = 512, kACols = kKBlock / 2, kABase = 2 * kTileTokens;
static_assert(kABase + kWStages * kACols <= kTmemCols, "tensor memory");
constexpr int kMaxGroup = 16;                                 // products per launch
constexpr int kUnitQueue = 4;                                // units the producer may run ahead of the slowest role
constexpr int kMaxSlices = 8;                                 // slices of a contraction
constexpr size_t kTicketBytes = 256;                          // in a product's workspace: the ticket

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) { mbar_arrive(smem_u32(bar)); }
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) { return mbar_try_wait(smem_u32(bar), parity); }
// The same without a wait.
__device__ __forceinline__ uint32_t mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}" : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok;
}
// Bounded wait: false after kPollLimit polls (status word set) or once another role has given up.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status) {
  for (uint32_t it = 0; it < kPollLimit; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 63u) == 63u && *abort_flag) return false;
  }
  *abort_flag = 1;
  atomicExch(status, (int)RWKVQ_ETIMEOUT);
  return false;
}
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* status) {
  return mbar_wait(smem_u32(bar), parity, abort_flag, status);
}
// A tile of a row-major matrix through its tensor map: columns x .. x + 63 (x a multiple of 64) of rows y .. y + NT - 1, zeros outside.
__device__ __forceinline__ void tensor_g2s(void* dst_smem, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
               ::"r"(smem_u32(dst_smem)), "l"(map), "r"(x), "r"(y), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst_smem, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_u32(dst_smem)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

// ---- tcgen05 wrappers (one CTA per tile: cta_group::1) ------------------------------------------
__device__ __forceinline__ void tmem_alloc(uint32_t* holder_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(holder_smem)), "r"(ncols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// Shared-memory matrix descriptor of a K-major bf16 tile with 128-byte rows and the 128-byte
// swizzle: 8-row groups are 1024 bytes apart; the tile base is 1024-byte aligned and a step of
// 16 columns along K advances the start address by 32 bytes.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);          // start address, 16-byte units
  d |= (uint64_t)1 << 16;                            // leading-dimension offset (unused with this swizzle)
  d |= (uint64_t)(1024u >> 4) << 32;                 // stride between 8-row groups
  d |= (uint64_t)1 << 46;                            // descriptor version of this architecture
  d |= (uint64_t)2 << 61;                            // 128-byte swizzle
  return d;
}
// Instruction descriptor: bf16 x bf16 -> fp32, both operands K-major, M x N tile.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// One 64-column block by a converged warp: four instructions of 16 columns each and the commit that arrives on `bar` when they have completed.
// One lane is elected by predicate and the operands are uniform: the same code in a branch of one lane took 800-950 cycles a block beside
// sixteen busy warps (each instruction's operands are moved to uniform registers one lane at a time), this form takes the 4 * N / 2
// cycles of the tensor pipe with the warps busy or not.
__device__ __forceinline__ void umma_block(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t accumulate, uint32_t bar) {
  asm volatile(
      "{\n .reg .pred q, p, one;\n .reg .b32 a1, a2, a3;\n .reg .b64 b1, b2, b3;\n"
      " elect.sync _|q, 0xffffffff;\n setp.ne.b32 p, %4, 0;\n setp.eq.b32 one, 0, 0;\n"
      " add.u32 a1, %1, 8;\n add.u32 a2, %1, 16;\n add.u32 a3, %1, 24;\n add.u64 b1, %2, 2;\n add.u64 b2, %2, 4;\n add.u64 b3, %2, 6;\n"
      " @q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n"
      " @q tcgen05.mma.cta_group::1.kind::f16 [%0], [a1], b1, %3, one;\n"
      " @q tcgen05.mma.cta_group::1.kind::f16 [%0], [a2], b2, %3, one;\n"
      " @q tcgen05.mma.cta_group::1.kind::f16 [%0], [a3], b3, %3, one;\n"
      " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%5];\n}"
      ::"r"(tmem_d), "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(bar) : "memory");
}
// The elected lane's commit alone (the same lane: the choice depends on the mask only).
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n"
               " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}" ::"r"(smem_u32(bar)) : "memory");
}
// 64 columns of one record: 16 lanes of tensor memory x 32 words.  Register order of the shape: per eight words
// (row g, words 2t and 2t + 1), (row g + 8, the same); r is numbered e = 4 * step + R as the packed layout numbers it (R & 1: row
// half, R >> 1: word).
__device__ __forceinline__ void tmem_st_triple(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x256b.x4.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
      ::"r"(taddr), "r"(r[0]), "r"(r[2]), "r"(r[1]), "r"(r[3]), "r"(r[4]), "r"(r[6]), "r"(r[5]), "r"(r[7]), "r"(r[8]), "r"(r[10]),
        "r"(r[9]), "r"(r[11]), "r"(r[12]), "r"(r[14]), "r"(r[13]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// 32 lanes x 32 consecutive columns of an accumulator: register c of lane l = D[lane base + l][col + c].
// The load is asynchronous: the registers hold the data only after tmem_ld_wait on the same array.
__device__ __forceinline__ void tmem_ld32_issue(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
}
// Waits for every tcgen05.ld of this thread; the array is an in/out operand so that no use of it
// is scheduled before the wait.
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&r)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
      : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]),
        "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]),
        "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]),
        "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
      :: "memory");
}

// Byte offset of element (row r, column k) of a K-major tile with 128-byte rows (64 bf16) and the
// 128-byte swizzle: the 16-byte chunk index is XORed with the row index modulo 8.
__host__ __device__ inline uint32_t sw128_offset(uint32_t r, uint32_t k) {
  return r * 128u + ((((k >> 3) ^ r) & 7u) << 4) + (k & 7u) * 2u;
}

// ---- pre-pass: token-shift mix along the sequence, bf16, operand tile layout -----------------------
__device__ __forceinline__ uint32_t vec_index(const uint8_t* stream, int p, int bits) {
  const uint32_t bitpos = (uint32_t)p * (uint32_t)bits, byte = bitpos >> 3;
  const uint32_t v = (uint32_t)stream[byte] | ((uint32_t)stream[byte + 1] << 8);
  return (v >> (bitpos & 7u)) & ((1u << bits) - 1u);
}

// One block per operand tile (NT tokens x 64 columns).  A thread owns 8 columns (one 16-byte vector)
// and a run of kMixRun consecutive tokens: it decodes its four mu pairs once, reads each row's vector
// once (the previous token's comes from the previous iteration) and writes 16 bytes per token into the
// tile's swizzled rows; the eight threads of a row read and write 128 contiguous bytes.
constexpr int kMixRun = 8;
static_assert(kTileTokens <= 32 * kMixRun, "a block of 256 threads covers one tile");
struct MixProduct {
  const __nv_bfloat16* X;
  const __nv_bfloat16* xprev0;
  const uint8_t* mu;
  const uint8_t* mu_aux;
  uint8_t* tiles;
  int mu_bits, ic, KB;
};

struct MixArgs {
  MixProduct p[kMaxGroup];
  unsigned block_start[kMaxGroup + 1];   // first block of each product; [n] = mixing blocks
  int n, M, MT, NT;
  unsigned* ticket;                      // to clear for the main kernel
};

// One launch mixes the operands of every product that needs it: block -> (product, token tile, column block).  The first block clears the main kernel's
// ticket.
__global__ void __launch_bounds__(256) prefill_mix_kernel(const __grid_constant__ MixArgs ma) {
  asm volatile("griddepcontrol.launch_dependents;");
  if (blockIdx.x == 0 && threadIdx.x == 0) *ma.ticket = 0u;
  if (ma.n == 0) return;
  int pi = 0;
  while (pi + 1 < ma.n && blockIdx.x >= ma.block_start[pi + 1]) ++pi;
  const MixProduct& mp = ma.p[pi];
  const __nv_bfloat16* X = mp.X;
  const __nv_bfloat16* xprev0 = mp.xprev0;
  const uint8_t* mu = mp.mu;
  const uint8_t* mu_aux = mp.mu_aux;
  uint8_t* tiles = mp.tiles;
  const int mu_bits = mp.mu_bits, ic = mp.ic, KB = mp.KB, M = ma.M, MT = ma.MT;
  const unsigned blk = blockIdx.x - ma.block_start[pi];
  const int kb = (int)(blk % (unsigned)KB), mt = (int)(blk / (unsigned)KB);
  if (mt >= MT) return;
  const int cx = threadIdx.x & 7, ty = threadIdx.x >> 3, NT = ma.NT;
  const int c = kb * kKBlock + cx * 8, r0 = ty * kMixRun, t0 = mt * NT + r0;
  if (r0 >= NT) return;                      // NT is a multiple of 16
  uint8_t* tile = tiles + ((size_t)mt * KB + kb) * ((size_t)NT * 128u);
  const bool col_ok = c < ic;
  uint4 xr[kMixRun + 1];     // [0] = the token before the run
#pragma unroll
  for (int i = 0; i <= kMixRun; ++i) {
    const int t = t0 + i - 1;
    xr[i] = make_uint4(0u, 0u, 0u, 0u);
    if (col_ok && t < M && (i > 0 || mu != nullptr)) {
      if (t >= 0) xr[i] = *reinterpret_cast<const uint4*>(X + (size_t)t * ic + c);
      else if (xprev0) xr[i] = *reinterpret_cast<const uint4*>(xprev0 + c);
    }
  }
  float2 mf[4];
  if (mu && col_ok) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t mw = reinterpret_cast<const uint32_t*>(mu_aux)[vec_index(mu, (c >> 1) + k, mu_bits)];
      mf[k] = __half22float2(*reinterpret_cast<const __half2*>(&mw));
    }
  }
#pragma unroll
  for (int i = 1; i <= kMixRun; ++i) {
    const int t = t0 + i - 1;
    uint4 out = make_uint4(0u, 0u, 0u, 0u);
    if (col_ok && t < M) {
      out = xr[i];
      if (mu) {
        const uint32_t xs[4] = {xr[i].x, xr[i].y, xr[i].z, xr[i].w}, ps[4] = {xr[i - 1].x, xr[i - 1].y, xr[i - 1].z, xr[i - 1].w};
        uint32_t os[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float2 xf = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&xs[k]));
          const float2 pf = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&ps[k]));
          const __nv_bfloat162 o = __floats2bfloat162_rn(fmaf(pf.x - xf.x, mf[k].x, xf.x), fmaf(pf.y - xf.y, mf[k].y, xf.y));
          os[k] = *reinterpret_cast<const uint32_t*>(&o);
        }
        out = make_uint4(os[0], os[1], os[2], os[3]);
      }
    }
    *reinterpret_cast<uint4*>(tile + sw128_offset((uint32_t)(r0 + i - 1), (uint32_t)(cx * 8))) = out;
  }
}

struct PrefillArgs {          // one product of the group
  const uint8_t* payload;   // chunks of the packed image
  const uint8_t* aux;       // VQ codebooks
  const uint8_t* xtiles;    // x_mix in operand tile layout: [MT][KB] tiles of NT x 64; nullptr: tiles of X through the tensor map
  void* Y;
  float* pieces;            // sums of the slices, if there are several: [tile][slice][column / 4][row][column % 4]
  int oc, KT, KB, MB, fmt, S;
  uint32_t chunk_bytes, rec_bytes, cb_bytes;
};

struct GroupArgs {
  CUtensorMap xmap[kMaxGroup];
  PrefillArgs p[kMaxGroup];
  int unit_start[kMaxGroup + 1];     // slices of tiles before each product, and in all
  int n, M, MT, NT, y_dtype;
  unsigned* ticket;                  // cleared by the pre-pass; the first ticket of a CTA is its own number
  int n_slots;                       // packed chunk slots in use (2 .. kMaxPackedSlots)
  uint32_t slot_bytes;               // bytes per slot: the largest chunk + codebook of the group, 128-byte multiple
  int* status;
};
static_assert(sizeof(GroupArgs) <= 4096, "kernel parameters");

enum { PF_SQ3 = 0, PF_VQ6 = 1, PF_VQ8 = 2 };

// A slice of a tile: chunks kt0 .. kt1 - 1 of chunk row cr x token tile mt of product p; p < 0: no more.
struct Unit { int p, cr, mt, slice, kt0, kt1; };

struct Ctrl {
  uint64_t cfull[kMaxPackedSlots], cempty[kMaxPackedSlots];
  uint64_t ready[kXStages], done[kXStages];      // a block's operands are there / have been read
  uint64_t accfull[2], accempty[2];
  uint64_t uqfull[kUnitQueue], uqempty[kUnitQueue];
  Unit units[kUnitQueue];
  uint32_t tmem_base;
  int abort_flag;
};
static_assert(sizeof(Ctrl) <= kCtrlBytes, "control block");

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// 64 columns (one triple) of an SQ record.  The three-bit fields stay where they lie in the low ten bits of the halves: as fp16 subnormals
// they are q * 2^(pos - 24), pos = 0, 3 or 6, exactly, and the scales take up 2^(24 - pos), so that no bias has to be subtracted.  s * q - s * z
// with one rounding (s * z is exact in fp32: two 11-bit significands) is the fp32 rounding of the exact decode
// s * (q - z); the result is its bf16 rounding.  Two columns per multiply-add: 518 cycles for sixteen warps' blocks on an SM, 635 with
// biased fp16 integers and single multiply-adds.
__device__ __forceinline__ uint64_t pair_of(float a, float b) {
  uint64_t v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b));
  return v;
}
__device__ __forceinline__ void sq_decode_triple(uint32_t wa, uint32_t wb, uint32_t wc, uint32_t sz_lo, uint32_t sz_hi, uint32_t (&r)[16]) {
  const uint32_t ua = wa >> 9, ub = wb >> 9, uc = wc >> 9;
  const uint32_t top = and_or<0x01000100u>(wc >> 7, and_or<0x00800080u>(wb >> 8, ua & 0x00400040u));
  const uint32_t f[16] = {wa & 0x00070007u, wa & 0x00380038u, wa & 0x01C001C0u, ua & 0x00070007u, ua & 0x00380038u,
                          wb & 0x00070007u, wb & 0x00380038u, wb & 0x01C001C0u, ub & 0x00070007u, ub & 0x00380038u,
                          wc & 0x00070007u, wc & 0x00380038u, wc & 0x01C001C0u, uc & 0x00070007u, uc & 0x00380038u, top};
  const float2 s0 = __half22float2(*reinterpret_cast<const __half2*>(&sz_lo));   // (s, z) of row g
  const float2 s1 = __half22float2(*reinterpret_cast<const __half2*>(&sz_hi));   // (s, z) of row g + 8
  const float nsz0 = -__fmul_rn(s0.x, s0.y), nsz1 = -__fmul_rn(s1.x, s1.y);
  const float s[2][3] = {{s0.x * 16777216.f, s0.x * 2097152.f, s0.x * 262144.f}, {s1.x * 16777216.f, s1.x * 2097152.f, s1.x * 262144.f}};
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    const int pos = e == 15 ? 2 : e % 5 % 3;
    const float se = s[e & 1][pos], ne = (e & 1) ? nsz1 : nsz0;
    const float2 q = __half22float2(*reinterpret_cast<const __half2*>(&f[e]));
    uint64_t d;
    float x, y;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(pair_of(se, se)), "l"(pair_of(q.x, q.y)), "l"(pair_of(ne, ne)));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(d));
    r[e] = pack_bf16(x, y);
  }
}

// 64 columns of a VQ record: pairs of columns from the warp's copy of the codebook, in bf16, at a shared-memory address that is a multiple of 1024.
template <int BITS, int Q>
__device__ __forceinline__ void vq_decode_block(const uint32_t (&w)[16], uint32_t cb, uint32_t (&r)[16]) {
  constexpr uint32_t kMask = ((1u << BITS) - 1u) << 2;
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    const int bit = BITS * (16 * Q + e), wi = bit >> 5, sh = bit & 31;
    uint32_t v;
    if (sh + BITS > 32) v = __funnelshift_r(w[wi], w[wi + 1], sh - 2);
    else v = sh >= 2 ? w[wi] >> (sh - 2) : w[wi] << (2 - sh);
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(r[e]) : "r"(and_or<kMask>(v, cb)));
  }
}

// Ticket -> slice of a tile: products with the longest slices first, slice major, then token tile major, then chunk rows: CTAs that run at
// the same time read the same few activation tiles from L2.
__device__ __forceinline__ Unit unit_of(const GroupArgs& ga, int ticket) {
  Unit u;
  u.p = -1;
  if (ticket >= ga.unit_start[ga.n]) return u;
  u.p = 0;
  while (ticket >= ga.unit_start[u.p + 1]) ++u.p;
  const PrefillArgs& a = ga.p[u.p];
  const int local = ticket - ga.unit_start[u.p], rest = local / a.MB;
  u.cr = local % a.MB;
  u.mt = rest % ga.MT; u.slice = rest / ga.MT;
  u.kt0 = a.KT * u.slice / a.S; u.kt1 = a.KT * (u.slice + 1) / a.S;
  return u;
}
// The next unit of this CTA as published by the producer (false: none left, or another role gave up).
// Called by whole warps (every lane reads the entry, lane 0 frees it) or by one thread alone.
__device__ __forceinline__ bool next_unit(Ctrl* ctrl, uint32_t& uq, Unit& out, bool whole_warp, int lane, volatile int* abortp, int* status) {
  const int slot = (int)(uq % kUnitQueue);
  bool ok = mbar_wait(&ctrl->uqfull[slot], (uq / kUnitQueue) & 1u, abortp, status);
  if (whole_warp) ok = __all_sync(0xFFFFFFFFu, ok);
  if (!ok) return false;
  const volatile Unit* q = &ctrl->units[slot];
  out.p = q->p; out.cr = q->cr; out.mt = q->mt; out.slice = q->slice; out.kt0 = q->kt0; out.kt1 = q->kt1;
  if (whole_warp) __syncwarp();
  if (!whole_warp || lane == 0) mbar_arrive(&ctrl->uqempty[slot]);
  ++uq;
  return out.p >= 0;
}

// A dequantisation warp: record dw of every chunk, the 64-column blocks of parity DG.  Its counters run along instead of being divided out of a
// block number: with sixteen of these warps on an SM an instruction in a chain takes about ten cycles, and the three hundred instructions
// of bookkeeping per chunk of a version that divided cost as much as the decoding.
struct Dequant {
  uint32_t ready, done, cfull, cempty;       // shared-memory addresses of the barrier arrays
  uint32_t packed, book, tmem;               // packed slots; the warp's codebook; the record's lanes of tensor memory
  uint32_t slot_bytes, n_slots;
  uint32_t xs, xphase, cs, cphase;           // activation stage of the next block and its round's parity; packed slot, likewise
  volatile int* abort_flag;
  int* status;
};
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
  return v;
}
// The place of the next block (its stage modulo 3) was last read for the third block before: stage - 3 of this round, or stage + 3 of the round
// before.  The barrier is tested ahead of the decoding, so that the answer is there when the block is.
struct Place { uint32_t bar, parity, column, free; };
__device__ __forceinline__ Place next_place(const Dequant& d) {
  const bool late = d.xs >= (uint32_t)kWStages;
  const uint32_t place = late ? d.xs - (uint32_t)kWStages : d.xs;
  Place p;
  p.bar = d.done + 8u * (late ? place : d.xs + (uint32_t)kWStages);
  p.parity = late ? d.xphase : d.xphase ^ 1u;
  p.column = d.tmem + kABase + place * kACols;
  p.free = mbar_test(p.bar, p.parity);
  return p;
}
__device__ __forceinline__ bool put_block(Dequant& d, const Place& p, const uint32_t (&r)[16], int lane) {
  if (!__all_sync(0xFFFFFFFFu, p.free) && !__all_sync(0xFFFFFFFFu, mbar_wait(p.bar, p.parity, d.abort_flag, d.status))) return false;
  tc_fence_after();
  tmem_st_triple(p.column, r);
  const uint32_t ready = d.ready + 8u * d.xs;
  d.xs += (uint32_t)kDequantGroups;
  if (d.xs >= (uint32_t)kXStages) { d.xs -= (uint32_t)kXStages; d.xphase ^= 1u; }
  tmem_st_wait();
  tc_fence_before();
  __syncwarp();
  if (lane == 0) mbar_arrive(ready);
  return true;
}
template <int FMT, int DG>
__device__ __forceinline__ bool dequant_unit(Dequant& d, int n_chunks, uint32_t rec_bytes, uint32_t cb_bytes, int dw, int lane) {
  constexpr int kPlanes = FMT == PF_VQ8 ? 4 : 3;
  const uint32_t rec = d.packed + (uint32_t)dw * rec_bytes;
  for (int kt = 0; kt < n_chunks; ++kt) {
    if (!__all_sync(0xFFFFFFFFu, mbar_wait(d.cfull + 8u * d.cs, d.cphase, d.abort_flag, d.status))) return false;
    const uint32_t slot = d.cs * d.slot_bytes, at = rec + slot;
    uint32_t w[16], r[16];
    uint4 sz = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int p = 0; p < kPlanes; ++p) {
      const uint4 v = lds128(at + (uint32_t)(p * 512) + (uint32_t)lane * 16u);
      w[4 * p] = v.x; w[4 * p + 1] = v.y; w[4 * p + 2] = v.z; w[4 * p + 3] = v.w;
    }
    if (FMT == PF_SQ3) {
      sz = lds128(at + RWKVQ_SQ_CODE_BYTES + (uint32_t)(lane >> 2) * 16u);
    } else {
      // the codebook in bf16: an entry is converted once a warp and chunk instead of at each of its uses, half the instructions of a block
      const uint32_t src = d.packed + slot + 8u * rec_bytes;
      for (uint32_t i = (uint32_t)lane * 8u; i < cb_bytes; i += 256u) {
        uint2 v;
        asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(src + i));
        const float2 f0 = __half22float2(*reinterpret_cast<const __half2*>(&v.x)), f1 = __half22float2(*reinterpret_cast<const __half2*>(&v.y));
        asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(d.book + i), "r"(pack_bf16(f0.x, f0.y)), "r"(pack_bf16(f1.x, f1.y)) : "memory");
      }
    }
    // nothing more is needed from the packed slot
    __syncwarp();
    if (lane == 0) mbar_arrive(d.cempty + 8u * d.cs);
    if (++d.cs == d.n_slots) { d.cs = 0u; d.cphase ^= 1u; }
    Place place = next_place(d);
    if (FMT == PF_SQ3) sq_decode_triple(w[3 * DG], w[3 * DG + 1], w[3 * DG + 2], sz.x, sz.z, r);
    else vq_decode_block<FMT == PF_VQ6 ? 6 : 8, DG>(w, d.book, r);
    if (!put_block(d, place, r, lane)) return false;
    place = next_place(d);
    if (FMT == PF_SQ3) sq_decode_triple(w[6 + 3 * DG], w[7 + 3 * DG], w[8 + 3 * DG], sz.y, sz.w, r);
    else vq_decode_block<FMT == PF_VQ6 ? 6 : 8, 2 + DG>(w, d.book, r);
    if (!put_block(d, place, r, lane)) return false;
    if (FMT != PF_SQ3) __syncwarp();         // the codebook copy is written again
  }
  return true;
}
template <int DG>
__device__ __forceinline__ bool dequant_any(Dequant& d, const PrefillArgs& a, int n_chunks, int dw, int lane) {
  if (a.fmt == PF_SQ3) return dequant_unit<PF_SQ3, DG>(d, n_chunks, (uint32_t)RWKVQ_SQ_RECORD_BYTES, 0u, dw, lane);
  if (a.fmt == PF_VQ6) return dequant_unit<PF_VQ6, DG>(d, n_chunks, a.rec_bytes, a.cb_bytes, dw, lane);
  return dequant_unit<PF_VQ8, DG>(d, n_chunks, a.rec_bytes, a.cb_bytes, dw, lane);
}

__global__ void __launch_bounds__(kThreads, 1) prefill_kernel(const __grid_constant__ GroupArgs ga) {
  extern __shared__ uint8_t smem_raw[];
  // operand tiles need 1024-byte alignment (8 rows of 128 bytes per swizzle group)
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  Ctrl* ctrl = reinterpret_cast<Ctrl*>(smem);
  uint8_t* xring = smem + kCtrlBytes;                        // [kXStages] activation tiles
  uint8_t* books = xring + kXStages * kXTileBytes;           // [kDequantWarps] codebooks in bf16
  uint8_t* packed = books + kDequantWarps * kBookBytes;      // [n_slots] chunk | codebook
  const uint32_t n_slots = (uint32_t)ga.n_slots, slot_bytes = ga.slot_bytes;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* abortp = &ctrl->abort_flag;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kMaxPackedSlots; ++s) { mbar_init(&ctrl->cfull[s], 1); mbar_init(&ctrl->cempty[s], kDequantWarps); }
    for (int s = 0; s < kXStages; ++s) { mbar_init(&ctrl->ready[s], 1 + kRecordWarps); mbar_init(&ctrl->done[s], 1); }
    for (int s = 0; s < 2; ++s) { mbar_init(&ctrl->accfull[s], 1); mbar_init(&ctrl->accempty[s], kEpilogueWarps); }
    for (int s = 0; s < kUnitQueue; ++s) { mbar_init(&ctrl->uqfull[s], 1); mbar_init(&ctrl->uqempty[s], 2 + kDequantWarps + kEpilogueWarps); }
    ctrl->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(&ctrl->tmem_base, kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  asm volatile("griddepcontrol.launch_dependents;");
  const uint32_t tmem_base = ctrl->tmem_base;

  if (warp == 0) {
    // ---- activation producer -------------------------------------------------------------------------
    if (lane == 0) {
      uint32_t uq = 0, kb_iter = 0;
      bool ok = true;
      const uint32_t tile_bytes = (uint32_t)ga.NT * 128u;
      for (Unit w; ok && next_unit(ctrl, uq, w, false, 0, abortp, ga.status);) {
        if (uq == 1) {                           // the other roles are at work on the first weights while the pre-pass ends
          asm volatile("griddepcontrol.wait;" ::: "memory");
          asm volatile("fence.proxy.async;" ::: "memory");
        }
        const PrefillArgs& a = ga.p[w.p];
        const uint8_t* src = a.xtiles ? a.xtiles + (size_t)w.mt * a.KB * tile_bytes : nullptr;
        for (int kb = 4 * w.kt0; kb < 4 * w.kt1; ++kb, ++kb_iter) {
          const int st = (int)(kb_iter % kXStages);
          ok = mbar_wait(&ctrl->done[st], ((kb_iter / kXStages) & 1u) ^ 1u, abortp, ga.status);
          if (!ok) break;
          mbar_arrive_expect_tx(&ctrl->ready[st], tile_bytes);
          uint8_t* dst = xring + (size_t)st * kXTileBytes;
          if (src) bulk_g2s(dst, src + (size_t)kb * tile_bytes, tile_bytes, &ctrl->ready[st]);
          else tensor_g2s(dst, &ga.xmap[w.p], kb * kKBlock, w.mt * ga.NT, &ctrl->ready[st]);
        }
      }
      // do not leave while copies issued by this thread may still be landing
      for (uint32_t i = (kb_iter > kXStages ? kb_iter - kXStages : 0); i < kb_iter; ++i)
        for (uint32_t it = 0; it < kPollLimit; ++it) if (mbar_try_wait(&ctrl->ready[i % kXStages], (i / kXStages) & 1u)) break;
    }
  } else if (warp == 2 + kDequantWarps + kEpilogueWarps) {
    // ---- chunk producer: deals the units and streams their packed chunks (and codebooks) as far ahead as the slots allow ----
    if (lane == 0) {
      uint32_t uq = 0, ck = 0;
      bool ok = true;
      while (ok) {
        const int slot = (int)(uq % kUnitQueue);
        ok = mbar_wait(&ctrl->uqempty[slot], ((uq / kUnitQueue) & 1u) ^ 1u, abortp, ga.status);
        if (!ok) break;
        if (uq == 1) asm volatile("griddepcontrol.wait;" ::: "memory");      // the pre-pass clears the ticket
        const Unit w = unit_of(ga, uq == 0 ? (int)blockIdx.x : (int)(gridDim.x + atomicAdd(ga.ticket, 1u)));
        volatile Unit* q = &ctrl->units[slot];
        q->p = w.p; q->cr = w.cr; q->mt = w.mt; q->slice = w.slice; q->kt0 = w.kt0; q->kt1 = w.kt1;
        mbar_arrive(&ctrl->uqfull[slot]);        // release: the entry is visible to whoever sees the phase complete
        if (w.p < 0) break;
        ++uq;
        const PrefillArgs& a = ga.p[w.p];
        const int cr = w.cr;
        for (int kt = w.kt0; kt < w.kt1; ++kt, ++ck) {
          const uint32_t c = ck % n_slots;
          ok = mbar_wait(&ctrl->cempty[c], ((ck / n_slots) & 1u) ^ 1u, abortp, ga.status);
          if (!ok) break;
          uint8_t* slot_base = packed + (size_t)c * slot_bytes;
          mbar_arrive_expect_tx(&ctrl->cfull[c], a.chunk_bytes + a.cb_bytes);
          bulk_g2s(slot_base, a.payload + (size_t)(cr * a.KT + kt) * a.chunk_bytes, a.chunk_bytes, &ctrl->cfull[c]);
          if (a.cb_bytes) bulk_g2s(slot_base + a.chunk_bytes, a.aux + (size_t)((cr >> 1) * a.KT + kt) * a.cb_bytes, a.cb_bytes, &ctrl->cfull[c]);
        }
      }
      for (uint32_t i = (ck > n_slots ? ck - n_slots : 0); i < ck; ++i)
        for (uint32_t it = 0; it < kPollLimit; ++it) if (mbar_try_wait(&ctrl->cfull[i % n_slots], (i / n_slots) & 1u)) break;
    }
  } else if (warp == 1) {
    // ---- tensor-core issue (the whole warp waits, one lane issues) ----------------------------------
    const uint32_t idesc = idesc_bf16(kTileRows, ga.NT);
    uint32_t uq = 0, st = 0, phase = 0, tile_iter = 0, wplace = tmem_base + kABase;
    const uint32_t ready = smem_u32(ctrl->ready), done = smem_u32(ctrl->done), wend = wplace + kWStages * kACols;
    const uint64_t xdesc = smem_desc_sw128(smem_u32(xring));
    uint64_t xd = xdesc;
    bool ok = true;
    for (Unit w; ok && next_unit(ctrl, uq, w, true, lane, abortp, ga.status);) {
      const int KB = 4 * (w.kt1 - w.kt0);
      const uint32_t as = tile_iter & 1u;
      ok = __all_sync(0xFFFFFFFFu, mbar_wait(&ctrl->accempty[as], ((tile_iter >> 1) & 1u) ^ 1u, abortp, ga.status));
      if (!ok) break;
      tc_fence_after();
      const uint32_t acc = tmem_base + as * (uint32_t)kTileTokens;
      uint32_t accumulate = 0u;
      for (int kb = KB; kb > 0; --kb) {
        ok = __all_sync(0xFFFFFFFFu, mbar_wait(ready + 8u * st, phase, abortp, ga.status));
        if (!ok) break;
        tc_fence_after();
        umma_block(acc, wplace, xd, idesc, accumulate, done + 8u * st);
        accumulate = 1u;
        xd += (uint64_t)(kXTileBytes >> 4); wplace += kACols;
        if (++st == (uint32_t)kXStages) { st = 0; phase ^= 1u; xd = xdesc; }
        if (wplace == wend) wplace = wend - kWStages * kACols;
      }
      if (ok) umma_commit(&ctrl->accfull[as]);
      ++tile_iter;
    }
  } else if (warp < 2 + kDequantWarps) {
    // ---- dequantisation: warp dw takes record dw (16 rows) of the chunk, group dg the blocks of parity dg ----
    // a warp reaches the 32 lanes of tensor memory of its number modulo 4
    const int dw = 2 * (warp & 3) + (((warp - 2) >> 2) & 1), dg = (warp - 2) / kRecordWarps;
    Dequant d;
    d.ready = smem_u32(ctrl->ready); d.done = smem_u32(ctrl->done); d.cfull = smem_u32(ctrl->cfull); d.cempty = smem_u32(ctrl->cempty);
    d.packed = smem_u32(packed); d.book = smem_u32(books) + (uint32_t)(warp - 2) * kBookBytes;
    d.tmem = tmem_base + ((uint32_t)(16 * dw) << 16);
    d.slot_bytes = slot_bytes; d.n_slots = n_slots;
    d.xs = (uint32_t)dg; d.xphase = d.cs = d.cphase = 0u;
    d.abort_flag = abortp; d.status = ga.status;
    uint32_t uq = 0;
    bool ok = true;
    for (Unit w; ok && next_unit(ctrl, uq, w, true, lane, abortp, ga.status);)
      ok = dg == 0 ? dequant_any<0>(d, ga.p[w.p], w.kt1 - w.kt0, dw, lane) : dequant_any<1>(d, ga.p[w.p], w.kt1 - w.kt0, dw, lane);
  } else if (warp < 2 + kDequantWarps + kEpilogueWarps) {
    // ---- epilogue: warp quarter qd reads lanes 32 qd .. 32 qd + 31 (weight rows) of an accumulator stage ----
    const int qd = warp & 3;
    asm volatile("griddepcontrol.wait;" ::: "memory");      // outputs are written only once all that came before the pre-pass is done
    uint32_t uq = 0, tile_iter = 0;
    bool ok = true;
    const int NT = ga.NT;
    for (Unit w; ok && next_unit(ctrl, uq, w, true, lane, abortp, ga.status);) {
      const PrefillArgs& a = ga.p[w.p];
      const uint32_t as = tile_iter & 1u;
      ok = __all_sync(0xFFFFFFFFu, mbar_wait(&ctrl->accfull[as], (tile_iter >> 1) & 1u, abortp, ga.status));
      if (!ok) break;
      tc_fence_after();
      const int t0 = w.mt * NT, nt = min(NT, ga.M - t0), row = w.cr * kTileRows + qd * 32 + lane, oc = a.oc;
      const uint32_t acc = tmem_base + as * (uint32_t)kTileTokens + ((uint32_t)(qd * 32) << 16);
      if (a.S > 1) {
        // the sums of a slice go to the workspace
        float4* dst = reinterpret_cast<float4*>(a.pieces) + ((size_t)(w.mt * a.MB + w.cr) * a.S + w.slice) * ((size_t)NT * (kTileRows / 4)) + qd * 32 + lane;
        uint32_t r[32];
#pragma unroll 1
        for (int cc = 0; cc < nt; cc += 32) {
          tmem_ld32_issue(acc + (uint32_t)cc, r);
          tmem_ld_wait(r);
#pragma unroll
          for (int k = 0; k < 8; ++k, dst += kTileRows)
            if (cc + 4 * k < nt)
              __stcg(dst, make_float4(__uint_as_float(r[4 * k]), __uint_as_float(r[4 * k + 1]), __uint_as_float(r[4 * k + 2]), __uint_as_float(r[4 * k + 3])));
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&ctrl->accempty[as]);
        ++tile_iter;
        continue;
      }
      const bool f32 = ga.y_dtype == RWKVQ_F32, row_ok = row < oc;
      const uint32_t stride = (uint32_t)oc;
      uint8_t* dst = static_cast<uint8_t*>(a.Y) + ((size_t)t0 * oc + row) * (f32 ? 4u : 2u);
      auto put = [&](const uint32_t (&r)[32], int c0) {
        if (!row_ok) return;
        const int n = nt - c0;
        if (f32) {
          float* p = reinterpret_cast<float*>(dst) + (size_t)c0 * stride;
          if (n >= 32) {
#pragma unroll
            for (int c = 0; c < 32; ++c, p += stride) *p = __uint_as_float(r[c]);
          } else {
#pragma unroll
            for (int c = 0; c < 32; ++c, p += stride)
              if (c < n) *p = __uint_as_float(r[c]);
          }
        } else {
          __nv_bfloat16* p = reinterpret_cast<__nv_bfloat16*>(dst) + (size_t)c0 * stride;
          if (n >= 32) {
#pragma unroll
            for (int c = 0; c < 32; ++c, p += stride) *p = __float2bfloat16_rn(__uint_as_float(r[c]));
          } else {
#pragma unroll
            for (int c = 0; c < 32; ++c, p += stride)
              if (c < n) *p = __float2bfloat16_rn(__uint_as_float(r[c]));
          }
        }
      };
        // two register buffers: the load of the next 32 columns is in flight while these are stored
        uint32_t ra[32], rb[32];
        tmem_ld32_issue(acc, ra);
#pragma unroll 1
        for (int cc = 0; cc < nt; cc += 64) {
          tmem_ld_wait(ra);
          if (cc + 32 < nt) tmem_ld32_issue(acc + (uint32_t)(cc + 32), rb);
          put(ra, cc);
          if (cc + 32 >= nt) break;
          tmem_ld_wait(rb);
          if (cc + 64 < nt) tmem_ld32_issue(acc + (uint32_t)(cc + 64), ra);
          put(rb, cc + 32);
        }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&ctrl->accempty[as]);
      ++tile_iter;
    }
  }
  // common exit: every role's loops are bounded, so all threads arrive here
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_base, kTmemCols);
}

// Adds up the slices of the tiles that are cut, in order.  Block (tile, kSumCols of its columns); one thread a row, so that what a warp
// reads and writes is contiguous.
constexpr int kSumCols = 16;
struct SumArgs {
  const float* pieces[kMaxGroup];
  void* Y[kMaxGroup];
  int tile_start[kMaxGroup + 1], oc[kMaxGroup], MB[kMaxGroup], S[kMaxGroup];
  int n, M, NT, y_dtype;
};
__global__ void __launch_bounds__(kTileRows) prefill_sum_kernel(const __grid_constant__ SumArgs sa) {
  int p = 0;
  while ((int)blockIdx.x >= sa.tile_start[p + 1]) ++p;
  const int row = threadIdx.x, tile = (int)blockIdx.x - sa.tile_start[p], t0 = tile / sa.MB[p] * sa.NT, c0 = (int)blockIdx.y * kSumCols;
  const int orow = tile % sa.MB[p] * kTileRows + row, nt = min(sa.NT, sa.M - t0), S = sa.S[p], oc = sa.oc[p];
  if (c0 >= nt) return;
  const size_t step = (size_t)sa.NT * (kTileRows / 4);
  const float4* src = reinterpret_cast<const float4*>(sa.pieces[p]) + (size_t)tile * S * step + (size_t)(c0 / 4) * kTileRows + row;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  float4 v[kSumCols / 4];
#pragma unroll
  for (int j = 0; j < kSumCols / 4; ++j) v[j] = __ldcg(src + j * kTileRows);
#pragma unroll 4
  for (int i = 1; i < S; ++i) {
    src += step;
#pragma unroll
    for (int j = 0; j < kSumCols / 4; ++j) {
      const float4 q = __ldcg(src + j * kTileRows);
      v[j].x += q.x; v[j].y += q.y; v[j].z += q.z; v[j].w += q.w;
    }
  }
  if (orow >= oc) return;
#pragma unroll
  for (int j = 0; j < kSumCols; ++j) {
    const float f = (j & 3) == 0 ? v[j / 4].x : ((j & 3) == 1 ? v[j / 4].y : ((j & 3) == 2 ? v[j / 4].z : v[j / 4].w));
    if (c0 + j < nt) {
      const size_t y = (size_t)(t0 + c0 + j) * oc + orow;
      if (sa.y_dtype == RWKVQ_F32) static_cast<float*>(sa.Y[p])[y] = f;
      else static_cast<__nv_bfloat16*>(sa.Y[p])[y] = __float2bfloat16_rn(f);
    }
  }
}

}  // namespace pf
}  // namespace rwkvq

using namespace rwkvq;

namespace {

struct HostProduct {
  pf::PrefillArgs a;
  const void* X; const void* xprev0;
  const uint8_t* mup; const uint8_t* mua; int mu_bits, ic;
  uint8_t* ws;
};

// Slices of a product's contraction: where it has so few tiles that its long contraction would be what the others wait for, about four
// chunks each (a slice costs its sums in the workspace, about a chunk's time), not more in all than leave room for other products.  Of limits from
// 48 to 296 and lengths from 3 to 7, 64 to 74 and 4 were the best over 22 layers (d 2048, 203 tokens: 53.6 us with whole tiles, 37 with
// slices; d 768, 48 tokens: 22.6, 14.4; d 640, 1368 tokens, limit 64: no slices, 32.8 where two each took 36.9).  Short contractions, whose slices
// are a chunk or two shorter than the whole, not where their sums (tiles x tokens of a tile) are many: d 512, 1000 tokens (4160): two slices 26.8 us,
// one 22.8; d 768, 400 tokens (2496): three 24.5, two 20.7; d 2048, 400 tokens (6656): two 62.8, one 56.2; 203 tokens (3328): two 34.9, one 37.2.
// Of 63 layers of d 512 to 2816 that this rule cuts otherwise (17 to 1368 tokens), 46 gain by it, up to 1.19 times, and 12 lose, up to 1.11 times: what it comes to
// is how evenly the layer's units fill the SMs (d 2176, 203 tokens, 3536: two 36.9, one 40.8, but d 2304, 3744: 41.4, 41.2; d 2816, 150 tokens, 3520: 47.1,
// 49.8, but d 2048, 224 tokens, 3584: 46.2, 44.9), and the mean is 1.04.  Of twelve chunks whole ones lose more than they gain: d 2944, 17 to 203 tokens, two
// 42.5 to 55.9, one 49.1 to 62.3; d 896, 400 tokens, three 26.9, two 28.9, one 26.8, and only from 500 tokens on one is better (28.9, 26.8).  A function of
// the product and M alone, so that a product gives the same bits in every group.
constexpr int kMaxSlicedTiles = 64;
int slices_of(int KT, long long tiles, int NT) {
  constexpr int kMinChunks = 6, kSliceChunks = 4, kShortChunks = 11, kMaxShortSums = 7000;
  if (KT < kMinChunks) return 1;
  long long most = kMaxSlicedTiles / tiles;
  if (KT <= kShortChunks) most = std::min(most, kMaxShortSums / (tiles * NT));
  return (int)std::min<long long>({(long long)pf::kMaxSlices, (long long)((KT + kSliceChunks / 2) / kSliceChunks), std::max<long long>(1, most)});
}

// A product's workspace: operand tiles, the ticket, sums of the slices.
struct Layout { int NT, MT, S; size_t off_ticket, off_pieces, bytes; };
Layout layout_of(const rwkvq_desc* d, int M) {
  Layout l;
  l.MT = (M + pf::kTileTokens - 1) / pf::kTileTokens;
  l.NT = ((M + l.MT - 1) / l.MT + 15) / 16 * 16;
  const size_t KB = (size_t)d->ic_pad / pf::kKBlock, tiles = (size_t)(d->oc_pad / 128) * l.MT;
  l.S = slices_of((int)(KB / 4), (long long)tiles, l.NT);
  l.off_ticket = round_up_sz((size_t)l.MT * KB * l.NT * 128, 256);
  l.off_pieces = l.off_ticket + pf::kTicketBytes;
  l.bytes = l.off_pieces + (l.S > 1 ? tiles * l.S * l.NT * 512 : 0);
  return l;
}

rwkvq_status check_product(const rwkvq_prefill_op& o, int M, HostProduct* out) {
  const rwkvq_desc* d = o.W_desc;
  if (!d || !o.W_image_dev || !o.X_bf16_dev || !o.Y_dev) return RWKVQ_EINVAL;
  if (o.mu_image_dev && !o.mu_desc) return RWKVQ_EINVAL;
  if (!o.mu_image_dev && o.xprev0_bf16_dev) return RWKVQ_EINVAL;
  if (d->oc == 1) return RWKVQ_ESHAPE;
  rwkvq_status st = check_matrix_desc(d);
  if (st != RWKVQ_OK) return st;
  if (o.mu_image_dev) {
    st = check_vector_desc(o.mu_desc, d->ic);
    if (st != RWKVQ_OK) return st;
  }
  if (d->ic % 8) return RWKVQ_ESHAPE;
  if (!aligned16(o.W_image_dev) || !aligned16(o.X_bf16_dev) || !aligned16(o.Y_dev) || (o.mu_image_dev && !aligned16(o.mu_image_dev)) ||
      (o.xprev0_bf16_dev && !aligned16(o.xprev0_bf16_dev)))
    return RWKVQ_EALIGN;
  const size_t need = layout_of(d, M).bytes;
  if (!o.workspace_dev || o.workspace_bytes < need) return RWKVQ_ENOMEM;
  if ((reinterpret_cast<uintptr_t>(o.workspace_dev) & 127u) != 0) return RWKVQ_EALIGN;
  const uint8_t* img = static_cast<const uint8_t*>(o.W_image_dev);
  pf::PrefillArgs& a = out->a;
  a.payload = img + RWKVQ_HEADER_BYTES;
  a.aux = img + matrix_aux_offset(d);
  a.xtiles = static_cast<const uint8_t*>(o.workspace_dev);
  a.Y = o.Y_dev;
  a.oc = d->oc; out->ic = d->ic;
  a.KT = d->ic_pad / 256; a.KB = a.KT * 4; a.MB = d->oc_pad / 128; a.S = 1;
  a.fmt = d->method == RWKVQ_SQ ? pf::PF_SQ3 : (d->bits == 6 ? pf::PF_VQ6 : pf::PF_VQ8);
  a.rec_bytes = d->method == RWKVQ_SQ ? (uint32_t)RWKVQ_SQ_RECORD_BYTES : rwkvq_vq_record_bytes(d->bits);
  a.chunk_bytes = 8u * a.rec_bytes;
  a.cb_bytes = d->method == RWKVQ_SQ ? 0u : (uint32_t)d->entries * 4u;
  out->X = o.X_bf16_dev; out->xprev0 = o.xprev0_bf16_dev;
  out->mup = nullptr; out->mua = nullptr; out->mu_bits = 0;
  if (o.mu_image_dev) {
    const uint8_t* m = static_cast<const uint8_t*>(o.mu_image_dev);
    out->mup = m + RWKVQ_HEADER_BYTES; out->mua = m + vector_aux_offset(o.mu_desc); out->mu_bits = o.mu_desc->bits;
  }
  out->ws = static_cast<uint8_t*>(o.workspace_dev);
  return RWKVQ_OK;
}


typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
// The driver's tensor map encoder, through the runtime's entry-point query; nullptr if it cannot be had.
EncodeTiledFn encode_tiled() {
  static const EncodeTiledFn fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) f = nullptr;
    return reinterpret_cast<EncodeTiledFn>(f);
  }();
  return fn;
}
// X[M][ic] bf16 as tiles of 64 columns x NT rows in the 128-byte swizzle.
bool encode_x(CUtensorMap* map, const void* X, int M, int ic, int NT) {
  EncodeTiledFn fn = encode_tiled();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)ic, (cuuint64_t)M}, strides[1] = {(cuuint64_t)ic * 2u};
  const cuuint32_t box[2] = {(cuuint32_t)pf::kKBlock, (cuuint32_t)NT}, step[2] = {1u, 1u};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(X), dims, strides, box, step, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

extern "C" {

size_t rwkvq_prefill_workspace_bytes(const rwkvq_desc* d, int M, int has_mu) {
  (void)has_mu;   // the room for operand tiles is there whether or not a token shift is applied
  if (!d || M <= 0 || check_matrix_desc(d) != RWKVQ_OK) return 0;
  // fewer tokens may be cut into more slices: a workspace for M tokens serves every shorter prompt
  size_t most = layout_of(d, M).bytes;
  const int sliced = pf::kTileTokens * (kMaxSlicedTiles / (d->oc_pad / 128));
  for (int m = 16; m < M && m <= sliced; m += 16) most = std::max(most, layout_of(d, m).bytes);      // tokens a tile are a multiple of 16
  return most;
}

rwkvq_status rwkvq_gemm_prefill_grouped(const rwkvq_prefill_op* ops, int n_ops, int M, int y_dtype, void* stream) {
  if (!ops || n_ops <= 0 || M <= 0) return RWKVQ_EINVAL;
  if (n_ops > pf::kMaxGroup) return RWKVQ_EUNSUPPORTED;
  if (y_dtype != RWKVQ_F32 && y_dtype != RWKVQ_BF16) return RWKVQ_EINVAL;
  HostProduct hp[pf::kMaxGroup];
  Layout lay[pf::kMaxGroup];
  for (int i = 0; i < n_ops; ++i) {
    const rwkvq_status st = check_product(ops[i], M, &hp[i]);
    if (st != RWKVQ_OK) return st;
    for (int j = 0; j < i; ++j)
      if (ops[j].Y_dev == ops[i].Y_dev || ops[j].workspace_dev == ops[i].workspace_dev) return RWKVQ_EINVAL;
    lay[i] = layout_of(ops[i].W_desc, M);
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int MT = lay[0].MT, NT = lay[0].NT, sms = sm_count();
  pf::GroupArgs ga;
  memset(&ga, 0, sizeof(ga));
  ga.n = n_ops; ga.M = M; ga.MT = MT; ga.NT = NT; ga.y_dtype = y_dtype;
  ga.status = device_status_ptr();
  if (!ga.status) return RWKVQ_ECUDA;
  pf::MixArgs ma;
  memset(&ma, 0, sizeof(ma));
  ma.M = M; ma.MT = MT; ma.NT = NT;
  // longest slice first: the long ones are dealt before the short ones fill the gaps
  int order[pf::kMaxGroup];
  for (int i = 0; i < n_ops; ++i) order[i] = i;
  std::stable_sort(order, order + n_ops, [&](int x, int y) { return hp[x].a.KT * lay[y].S > hp[y].a.KT * lay[x].S; });
  pf::SumArgs sa;
  sa.n = 0; sa.M = M; sa.NT = NT; sa.y_dtype = y_dtype; sa.tile_start[0] = 0;
  long long units = 0;
  unsigned long long mix_blocks = 0;
  uint32_t slot = 0;
  for (int i = 0; i < n_ops; ++i) {
    const HostProduct& h = hp[order[i]];
    const Layout& l = lay[order[i]];
    pf::PrefillArgs& a = ga.p[i];
    a = h.a;
    a.S = l.S;
    a.pieces = reinterpret_cast<float*>(h.ws + l.off_pieces);
    if (i == 0) ma.ticket = ga.ticket = reinterpret_cast<unsigned*>(h.ws + l.off_ticket);
    ga.unit_start[i] = (int)units;
    units += (long long)a.MB * MT * a.S;
    if (units > 0x3FFFFFFF) return RWKVQ_EUNSUPPORTED;
    if (a.S > 1) {
      sa.pieces[sa.n] = a.pieces; sa.Y[sa.n] = a.Y; sa.oc[sa.n] = a.oc; sa.MB[sa.n] = a.MB; sa.S[sa.n] = a.S;
      sa.tile_start[sa.n + 1] = sa.tile_start[sa.n] + a.MB * MT;
      ++sa.n;
    }
    slot = std::max(slot, (a.chunk_bytes + a.cb_bytes + 127u) & ~127u);
    // operands: straight from X, or through the pre-pass
    if (!h.mup && encode_x(&ga.xmap[i], h.X, M, h.ic, NT)) {
      a.xtiles = nullptr;
    } else {
      pf::MixProduct& mp = ma.p[ma.n];
      mp.X = static_cast<const __nv_bfloat16*>(h.X); mp.xprev0 = static_cast<const __nv_bfloat16*>(h.xprev0);
      mp.mu = h.mup; mp.mu_aux = h.mua; mp.tiles = h.ws; mp.mu_bits = h.mu_bits; mp.ic = h.ic; mp.KB = a.KB;
      ma.block_start[ma.n++] = (unsigned)mix_blocks;
      mix_blocks += (unsigned long long)MT * (unsigned long long)a.KB;
      if (mix_blocks > 0x7FFFFFF0ull) return RWKVQ_EUNSUPPORTED;
    }
  }
  ga.unit_start[n_ops] = (int)units;
  ma.block_start[ma.n] = (unsigned)mix_blocks;
  ga.slot_bytes = slot;
  ga.n_slots = (int)std::min<uint32_t>(pf::kMaxPackedSlots, (pf::kMaxSmemBytes - pf::kFixedSmemBytes) / slot);
  if (ga.n_slots < 2) return RWKVQ_EUNSUPPORTED;
  pf::prefill_mix_kernel<<<(unsigned)std::max<unsigned long long>(mix_blocks, 1), 256, 0, s>>>(ma);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_status(e);
  static SmemOptIn opt_in;
  e = opt_in((const void*)pf::prefill_kernel, (int)pf::kMaxSmemBytes);
  if (e != cudaSuccess) return cuda_status(e);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)std::min<long long>(units, sms)); cfg.blockDim = dim3(pf::kThreads);
  cfg.dynamicSmemBytes = pf::kFixedSmemBytes + (uint32_t)ga.n_slots * slot; cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, pf::prefill_kernel, ga);
  if (e != cudaSuccess || sa.n == 0) return cuda_status(e);
  cfg.gridDim = dim3((unsigned)sa.tile_start[sa.n], (unsigned)(NT + pf::kSumCols - 1) / pf::kSumCols); cfg.blockDim = dim3(pf::kTileRows); cfg.dynamicSmemBytes = 0;
  return cuda_status(cudaLaunchKernelEx(&cfg, pf::prefill_sum_kernel, sa));
}

rwkvq_status rwkvq_gemm_prefill(const rwkvq_desc* d, const void* W, const rwkvq_desc* mud, const void* mu, const void* X,
                                const void* xprev0, int M, void* Y, int y_dtype, void* ws, size_t ws_bytes, void* stream) {
  if (!d || !W || !X || !Y || M <= 0) return RWKVQ_EINVAL;
  if (mu && !mud) return RWKVQ_EINVAL;
  rwkvq_prefill_op op;
  op.W_desc = d; op.W_image_dev = W; op.mu_desc = mud; op.mu_image_dev = mu; op.X_bf16_dev = X; op.xprev0_bf16_dev = xprev0;
  op.Y_dev = Y; op.workspace_dev = ws; op.workspace_bytes = ws_bytes;
  return rwkvq_gemm_prefill_grouped(&op, 1, M, y_dtype, stream);
}

}  // extern "C"
