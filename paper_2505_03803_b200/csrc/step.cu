// A whole decode step as one persistent launch.
//
// Decode at batch 1..16 reads every packed weight once and does almost no arithmetic per byte
// (the paper's compute-to-memory argument, Section 1 and Appendix A.3), and one projection of a
// 7B-class layer is only a few microseconds of HBM time.  Launching one kernel per projection
// leaves the memory system idle between launches, so the step is ONE kernel with one CTA per SM:
//
//   * a producer warp streams packed weights from HBM into a ring of shared-memory slots with
//     bulk asynchronous copies (cp.async.bulk + mbarrier transaction counts).  Weights never depend
//     on activations, so the stream runs ahead across products and across stage boundaries;
//   * the stager warps (three, or seven for batches above 8: Shape) build the fp16 input x_mix = x + (x_prev - x) (.) mu_hat (Appendix A.1
//     Eq. 20) of the next run of units in one of two shared-memory buffers.  What does not depend
//     on the previous stage (mu_hat, x_prev) is prepared before the grid-wide stage barrier; the
//     stagers also clear the next stage's outputs and post this CTA's arrival at the barrier;
//   * consumer warps in groups of eight (two groups; one for batches above 8, whose record routine
//     needs the registers of two).  A unit is a 256-row x 256-column tile (two 128-row chunks of the
//     packed image); the groups take the CTA's units alternately, so one group computes while the
//     other waits, flushes or synchronises.  Warp w of a group owns rows
//     16w..16w+15 of both chunks and runs the m16n8k16 tensor-core steps of gemv_core.cuh with
//     every input fragment shared by the two records.  Partial sums go to y with fp32 reductions
//     (16 bytes per lane after a transpose among lanes) at the end of a run along K.  In plans of small
//     stages a group's first unit is unpacked into tensor memory while the inputs are on their way.
//
// For larger inputs per CTA, and whenever a product's input is an element-wise operator on
// earlier outputs (rwkvq_input_xform: the WKV recurrence and sigmoid gate of Appendix A.1 Eqs. 23-24,
// the squared ReLU and output gate of Eq. 27, optionally a root-mean-square normalisation), the
// inputs of a stage are not built per CTA: after the stage barrier all CTAs together compute the
// stage's x_mix once (mix_slice: a quarter-warp per 128-column group of a plain input, a warp where an operator is in front)
// into a scratch region of the plan, publish it through a second barrier, and every CTA fetches its segments with bulk copies.  (Squared inputs
// alone, few to a CTA, are staged by the CTAs that read them: stage_squares.)
//
// The host plans the step once: every stage's units are dealt WHOLE to the CTAs, in runs of neighbouring units by the
// smallest estimated time of the slowest CTA, along rows of tiles where that is no worse; the plan is a per-CTA
// list of 128-byte unit descriptors plus a list of 64-byte input events (segments and barrier
// arrivals).
#include <cuda.h>           // types of the stream memory operations (no driver symbol is linked)
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <unordered_map>
#include <vector>

#include "../../include/rwkvq.h"
#include "gemv_core.cuh"
#include "host_util.h"

namespace rwkvq {

int* device_status_ptr();  // api_misc.cu
unsigned abort_epoch();     // api_misc.cu: bumped whenever rwkvq_device_status reports a failed wait

// UF_HEAD: reads the head of its segment, announced by itself (UF_PHASE: in the barrier's second phase); UF_REST: its group's first unit behind the head.
enum { UF_FLUSH = 1, UF_VQ = 2, UF_BITS8 = 4, UF_HEAD = 8, UF_REST = 16, UF_PHASE = 32 };

struct StepUnit {            // 128 bytes, copied into the slot header by the producer
  uint64_t src0, src1;       // global addresses of chunk A / chunk B (0 = absent)
  uint64_t cb_src;           // VQ: codebook of the tile
  uint32_t bytes0, bytes1;   // bytes of each chunk
  uint32_t cb_bytes;
  uint32_t off0;             // unused
  uint32_t flags;            // UF_*
  uint32_t seg;              // number, within this CTA, of the input segment the unit reads
  uint32_t stage;            // stage number (0-based)
  uint32_t xcol0;            // column of the unit's tile inside the segment
  uint32_t row0, oc;         // first output row of chunk A; rows of the product
  uint64_t y;                // float y[B][oc]
  uint32_t xstride, gs_off;  // geometry of the segment: bytes between batch rows, offset of the sums
  uint32_t nbp, reserved;
  uint32_t chunk_bytes;      // distance between chunk A and chunk B inside the slot
  uint32_t rec_bytes;
  uint32_t ev_index;         // position of the unit's segment in this CTA's event list
  uint32_t between_mask;     // events between the group's previous segment and this one, oldest in bit 0:
                             // 1 = barrier arrival, 0 = segment of the other group (valid for up to 32 events)
  uint32_t after_count;      // set on a group's last unit of a stage: events after its segment up to and
  uint32_t after_mask;       // including the stage's barrier arrival, to be passed right after the unit
  uint32_t pad[4];
};
static_assert(sizeof(StepUnit) == 128, "unit descriptor size");

enum { EV_SEGMENT = 0, EV_ARRIVE = 1 };

struct StepEvent {           // 64 bytes
  union {
    // segment.  Mixed in the CTA: x, xprev, mu, mu_aux as given by the caller.  Copied from the
    // stage's pre-pass (StepArgs::mix): x = first byte of the segment in the pre-pass rows,
    // xprev = first byte of its sums, mu = 0.
    struct { uint64_t x, xprev, mu, mu_aux; } seg;
    // arrival: float ranges to clear before arriving; then this CTA's share of the stage's
    // pre-pass: groups [grp_lo, grp_hi) of the (product, batch row, 128-column group) list that begins with product op_first
    struct { uint64_t zptr[3]; uint32_t grp_lo, grp_hi; } arr;
  };
  union {
    struct { uint32_t ic, col0, ncols; uint16_t mu_bits, mu_entries; } segd;   // copied segments: ic = bytes between rows
    struct { uint32_t zcount[3]; uint16_t op_first, op_count; } arrd;          // products this CTA's share falls in
  };
  uint32_t kind;             // EV_SEGMENT / EV_ARRIVE
  uint32_t barrier;          // segment: index + 1 of the stage barrier to pass first; arrival: index of the barrier
  uint32_t xstride_sums;     // segment: xstride | sums << 31
  uint16_t mu_off16;         // segment: offset / 16 of the decoded mu row inside the buffer
  uint16_t flags;            // EF_*
};
// EF_SQUARES: of a stage whose inputs every CTA squares for itself (see kSquaresShare); arrival: the stage that begins.  EF_READ_FIRST: arrival; the
// outputs to clear are inputs of the stage that ends, which every CTA has read when that stage's second barrier opens.
// EF_HEAD: segment; its first kHeadTiles tiles are announced ahead of the rest.  EF_BEHIND_SQUARES: copied segment; its buffer was last filled by
// stage_squares.
enum { EF_SQUARES = 1, EF_READ_FIRST = 2, EF_HEAD = 4, EF_BEHIND_SQUARES = 8 };
static_assert(sizeof(StepEvent) == 64, "event descriptor size");

// One product's share of a stage's pre-pass: where its inputs are and where x_mix (fp16 rows of
// ic_pad columns, zero beyond ic) and the per-group sums ([group][3][nbp] floats) go.
struct StepMixOp {           // 64 bytes
  uint64_t x, xprev, mu, mu_aux, dst_x, dst_sums;
  uint32_t ic, ic_pad;
  // kind: rwkvq_input_kind | 0x100 when the row is RMS-normalised | 0x200 when this token's input is stored
  // (xprev_out) | on every product of the stage: 0x400 where some input is normalised, 0x800 where all are
  // plain buffers; a kind with any of the low ten bits set has a StepMixX beside it
  uint16_t mu_bits, mu_entries, sums, kind;
};
static_assert(sizeof(StepMixOp) == 64, "pre-pass descriptor size");
// Element-wise operator in front of the product (rwkvq_input_xform): fp32 sources [B][ic], state,
// parameters.  Kept apart so that the pre-pass of plain products reads 64 bytes per item as before.
struct StepMixX {            // 80 bytes
  uint64_t src, k, v, state_a, state_b, state_p, u, w;   // `k` holds the gate for RWKVQ_IN_F32
  uint64_t xprev_out, scale;         // scale: device address of one float that multiplies the operator's result (0 = none)
};
static_assert(sizeof(StepMixX) == 80, "pre-pass operator descriptor size");

constexpr int kGroupWarps = 8, kGroupThreads = kGroupWarps * 32;
// Thread layout of a CTA, by the number of batch blocks NB a record is multiplied with.
//   NB = 1 (B <= 8): two consumer groups of eight warps, three stager warps, one producer warp: 640 threads,
//     96 registers each at launch.  They stay so for all roles (with 104 for the consumers and 64 for the others, which the compiler takes as the limit of these
//     roles' code, the pre-pass of a stage spilled, and behind a barrier's acquire a spilled word is a trip to L2: blocks 136 us where
//     they took 127), except with units unpacked ahead and no pre-pass (consumer_regs, stager_regs).
//   NB = 2 (B > 8): the record routine wants about 150 registers, which sixteen consumer warps cannot have,
//     and eight warps that keep everything in registers outrun sixteen that spill: ONE consumer group,
//     seven stager warps (the stage pre-pass is theirs), one producer: 512 threads, 128 registers at
//     launch, re-divided to 152 for the two consumer warpgroups (what their routine needs to keep
//     everything in registers) and 104 for the other two (measured: 168 / 88 and 144 / 112 are slower).
template <int NB> struct Shape {
  static constexpr int kGroups = NB == 2 ? 1 : 2;
  static constexpr int kStagerWarps = NB == 2 ? 7 : 3;
  static constexpr int kConsumerWarps = kGroupWarps * kGroups;
  static constexpr int kConsumerThreads = kConsumerWarps * 32, kStagerThreads = kStagerWarps * 32;
  static constexpr int kThreads = kConsumerThreads + kStagerThreads + 32;
  static constexpr int kLaunchRegs = NB == 2 ? 128 : 96;
  static_assert(kConsumerWarps % 4 == 0 && (kStagerWarps + 1) % 4 == 0, "register re-division works on warpgroups of four warps");
  static_assert(kLaunchRegs * kThreads <= 65536, "register file");
};
// With units unpacked ahead and inputs that the CTAs mix themselves the consumers' code wants eight more, and the stagers', without a pre-pass, make do with
// 64 (1.6B-class, twelve layers, batch 1: 180.6 us at 96 each, 179.4).  The kernels that unpack ahead still spill a few words of the consumers' (<1, 0, true, true> 12 bytes of
// stores and 44 of loads, <1, 1, true> and <1, 2, true> 12 and 36; the others up to eight rows none).  They cost nothing that can be measured: with values read again where they are
// rarely wanted (no spills in the first, 4 and 8 bytes in the other two) the steps are no faster (1.6B-class 347.9 us, without 348.5 to 353.7; blocks, batch 2, 108.6, 108.7).
__host__ __device__ constexpr int consumer_regs(int NB, int MIX, bool PARK) { return NB == 2 ? 152 : PARK && MIX == 0 ? 104 : 96; }
__host__ __device__ constexpr int stager_regs(int NB, int MIX, bool PARK) { return NB == 2 ? 104 : PARK && MIX == 0 ? 64 : 96; }
constexpr int groups_of(int NB) { return NB == 2 ? 1 : 2; }
constexpr int threads_of(int NB) { return NB == 2 ? Shape<2>::kThreads : Shape<1>::kThreads; }
// Slots of the weight ring: a unit for each consumer group and one on its way.  More are filled while a stage's first inputs are read, and hold those
// up (7B-class stack, batch 1: two 1257 us, three 1134, four 1144, five 1153; batch 8: 1478, 1355, 1359); above eight rows, with one group, two do
// as well as four (14B-class stack: 3420 us each).
constexpr int kMaxSlots = 3;
constexpr uint32_t kCtrlBytes = 1024, kMuScratch = 1024;
// Input-segment buffers, one in use and one being filled, as large as the ring leaves: every hand-over of a segment costs all roles a pass through the
// barriers.  Above eight rows 62 KB hold the 1792 columns of sixteen rows that a CTA's seven units of a 4096-column product read (14B-class stack,
// batch 16: 32 KB 3420 us, 48 KB 3348, 62 KB 3327).  Up to eight rows 31 KB hold the 1792 columns of eight and leave the ring three slots beside the
// copies of two codebooks of 256 entries (7B-class stack with them: batch 1 1276 -> 1154 us, batch 8 1471 -> 1362; without them, batch 8: 40 KB 1345,
// 30 KB 1350; a size that the plan chooses costs more, 1.6B-class batch 1 414.7 -> 417.3, 14B-class batch 16 3332 -> 3352).
constexpr uint32_t xbuf_bytes_of(int NB) { return NB == 2 ? 63488u : 31488u; }
template <int MIX, int NB> struct XBufs { static constexpr uint32_t kCount = 2u, kBytes = xbuf_bytes_of(NB); };
// Tiles at the head of a stage's first segment: one for each of two consumer groups' first units.
constexpr int kHeadTiles = 2;
constexpr uint32_t kSmemLimit = 232448;  // 227 KB
// Of a CTA that allocates tensor memory.  tcgen05.alloc waits, without a limit, for columns that another CTA on the SM holds, and beside this kernel's registers
// (61 440 of 65 536) a small one would fit.  An SM has 228 KB, of which every CTA takes 1 KB for the system: beside this none does (128: the kernels' static
// shared memory), so the columns are always there.  1.6B-class, batch 1: 347.9 us without and with; 1.6B-class blocks, batch 2: 108.6, 108.7.
constexpr uint32_t kSmemAlone = kSmemLimit - 128;
static_assert(233472 - (kSmemAlone + 1024) < 1024, "room for another CTA");
constexpr uint32_t kDefaultPollLimit = 1u << 22;

struct StepArgs {
  const StepUnit* units;
  const StepEvent* events;
  const uint32_t* unit_off;   // [P+1]
  const uint32_t* event_off;  // [P+1]
  unsigned* counter;          // stage barriers: arrivals at barrier k, summed over all runs, in counter[k]
  unsigned target;            // arrivals that open a barrier in this run: run number * CTAs (mod 2^32)
  unsigned wait_skew;         // added to the target the WAITS compare with (0; a test sets it to make them run out)
  uint32_t poll_limit;        // polls after which a wait gives up
  int* status;
  int B, n_slots, n_stages;
  uint32_t slot_bytes, replica_bytes;
  // Larger batches: x_mix and the sums of a stage are computed ONCE by all CTAs together after the
  // stage barrier (instead of by every CTA that reads a column), published through a second
  // barrier per stage (counter[n_stages + 1 + s]), and fetched into the segment buffers with bulk copies.
  int mix;
  const StepMixOp* mixops;    // dst_x / dst_sums are offsets into `scratch`
  const StepMixX* mixx;       // parallel to mixops
  uint8_t* scratch;
  // Host-buffer runs (rwkvq_step_run_host): the activations arrive in chunks of 2^in_shift bytes while
  // the step is already running, several to a copy; after a copy that ends with chunk i the copy stream stores in_base + i + 1 in *in_flag.
  // Whoever reads inputs inside [in_lo, in_hi) first waits for the chunk that holds their last byte.
  // in_flag == nullptr: the inputs are resident.
  const unsigned* in_flag;
  unsigned in_base, in_shift;
  uint64_t in_lo, in_hi;
};

// ---- mbarrier / bulk-copy wrappers ------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// The hardware parks the warp for a while (it is woken when the phase completes), so that waiting warps do not compete for
// issue slots with computing ones.  Whole warps wait: from an arrival to the waiting warp's next instruction it takes about
// 115 cycles then, 145 with a time limit as a third operand, and 750 when one lane waits while the others sit at the
// warp's next meeting point.
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}
// The launch's poll limit sits directly behind the CTA's abort flag in the control block (Ctrl).
__device__ __forceinline__ uint32_t poll_limit_of(volatile int* abort_flag) { return (uint32_t)abort_flag[1]; }
// Bounded wait by one thread: gives up (and raises the CTA-wide abort flag) after that many polls
// or when another role of this CTA has already given up.
__device__ __forceinline__ bool mbar_wait_one(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* status) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint32_t limit = poll_limit_of(abort_flag);
  for (uint32_t it = 0; it < limit; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 63u) == 63u && *abort_flag) return false;
  }
  *abort_flag = 1;
  atomicExch(status, (int)RWKVQ_ETIMEOUT);
  return false;
}
// Warp-collective bounded wait: every lane polls (so that each lane itself observes the completed
// phase and with it the data the barrier guards); the verdict is made warp-uniform.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* status) {
  const bool ok = mbar_wait_one(bar, parity, abort_flag, status);
  return __all_sync(0xFFFFFFFFu, ok);
}
// Named barrier over `nthreads` threads that also ANDs a predicate: a uniform verdict for a role.
__device__ __forceinline__ bool named_bar_and(int id, int nthreads, bool pred) {
  uint32_t r;
  asm volatile("{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.and.pred q, %2, %3, p;\n selp.u32 %0, 1, 0, q;\n}"
               : "=r"(r) : "r"((uint32_t)pred), "r"(id), "r"(nthreads) : "memory");
  return r != 0;
}
// Packed weights are read exactly once per step: they are marked evict-first so that streaming
// them does not push the activations, the plan and the outputs out of L2.
__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ void bulk_g2s(void* dst_smem, const void* src, uint32_t bytes, uint64_t* bar, uint64_t policy) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
               ::"r"(smem_u32(dst_smem)), "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy) : "memory");
}
__device__ __forceinline__ void bulk_g2s_plain(void* dst_smem, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_u32(dst_smem)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void named_bar_sync(int id, int nthreads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}
__device__ __forceinline__ unsigned ld_acquire_sys(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.sys.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release_gpu(unsigned* p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t smem_add_acq_rel(uint32_t* p, uint32_t v) {
  uint32_t old;
  asm volatile("atom.acq_rel.cta.shared::cta.add.u32 %0, [%1], %2;" : "=r"(old) : "r"(smem_u32(p)), "r"(v) : "memory");
  return old;
}

// A slot's data is announced to the consumer group that takes the unit, on a barrier of that group's: with one barrier for both and an odd number of
// slots a group would meet every second of its phases only, and while the other group's unit is still arriving in the slot, the phase before it
// looks like the one the group waits for (waits see the parity of a phase, not its number).
struct Ctrl {
  uint64_t full[2][kMaxSlots], empty[kMaxSlots];
  uint64_t xfull[4], xempty[4], xhead[2];
  uint32_t stage_cnt[64];    // one 8-bit count per grid barrier (four per word): how many of the parties
                             // of this CTA (every consumer warp, and the stagers as one) have reported the
                             // stage that the barrier closes.  Per barrier, not one running total: consumer
                             // warps of a CTA without work in the coming stages may run any number of
                             // stages ahead of the stagers.
  uint32_t mix_at[8];        // batch row | group << 16 of the item in each stager warp's MixSlot
  int abort_flag;
  int poll_limit;            // must follow abort_flag (poll_limit_of)
  uint32_t tmem_base;
};
static_assert(sizeof(Ctrl) <= kCtrlBytes, "control block");
constexpr uint32_t kMaxBarriers = 256;   // barriers that close a stage (8-bit counts in Ctrl::stage_cnt)

// One of the parties of grid barrier `b` (each consumer warp, the stagers as one) reports that its part of the stage the barrier
// closes is done; whoever reports last posts the CTA's arrival.  The count is an acquire-release
// read-modify-write at CTA scope and the arrival a GPU-scope release, so the arrival is ordered
// after everything every party did before reporting (the consumers' reductions into y, the
// stagers' clearing of the next outputs): block-level synchronisation followed by one thread's
// release, the pattern of a cooperative grid barrier.
template <int NB>
__device__ __forceinline__ void stage_report(Ctrl* ctrl, const StepArgs& a, uint32_t b) {
  const uint32_t sh = 8u * (b & 3u);
  const uint32_t old = smem_add_acq_rel(&ctrl->stage_cnt[b >> 2], 1u << sh);
  if (((old >> sh) & 0xFFu) == (uint32_t)Shape<NB>::kConsumerWarps) red_release_gpu(a.counter + b, 1u);
}
// Where the consumer warps are the busy role (two batch blocks per record) they only count
// themselves in, and a stager thread, which has nothing else to do at that point, waits (bounded)
// for the consumer warps' reports of THIS barrier and arrives: the release, which waits for the CTA's
// outstanding reductions, stays off the consumer warps.  The count is per barrier (the 8-bit
// fields of stage_cnt): a warp without work in the next stages runs ahead through their events,
// so a running total over all stages would reach its value for this stage while warps of
// this stage are still adding to the outputs.
__device__ __forceinline__ void stage_report_total(Ctrl* ctrl, uint32_t b) {
  asm volatile("red.release.cta.shared::cta.add.u32 [%0], %1;" ::"r"(smem_u32(&ctrl->stage_cnt[b >> 2])), "r"(1u << (8u * (b & 3u))) : "memory");
}
template <int NB>
__device__ __forceinline__ bool stage_wait_total_and_arrive(Ctrl* ctrl, const StepArgs& a, uint32_t b, volatile int* abort_flag) {
  const uint32_t limit = poll_limit_of(abort_flag) << 4;
  const uint32_t sh = 8u * (b & 3u);
  for (uint32_t it = 0; it < limit; ++it) {
    uint32_t v;
    asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(&ctrl->stage_cnt[b >> 2])) : "memory");
    if (((v >> sh) & 0xFFu) >= (uint32_t)Shape<NB>::kConsumerWarps) { red_release_gpu(a.counter + b, 1u); return true; }
    if ((it & 255u) == 255u && *abort_flag) return false;
  }
  *abort_flag = 1;
  atomicExch(a.status, (int)RWKVQ_ETIMEOUT);
  return false;
}

// One thread: wait (bounded) until the chunk that holds byte `last` (the address of the last input byte
// about to be read) has arrived.  Addresses outside the arriving range are resident already.
__device__ __forceinline__ bool wait_inputs(const StepArgs& a, uint64_t last, volatile int* abort_flag) {
  if (!a.in_flag || last < a.in_lo || last >= a.in_hi) return true;
  const unsigned need = a.in_base + (unsigned)((last - a.in_lo) >> a.in_shift) + 1u;
  const uint32_t limit = a.poll_limit << 2;
  for (uint32_t it = 0; it < limit; ++it) {
    if ((int)(ld_acquire_sys(a.in_flag) - need) >= 0) return true;
    if ((it & 255u) == 255u && *abort_flag) return false;
  }
  *abort_flag = 1;
  atomicExch(a.status, (int)RWKVQ_ETIMEOUT);
  return false;
}

// How often a group has had the slot of its unit before: once a round of the ring, or every second round where the ring's odd number of slots makes
// the two groups take turns.
template <int NB>
__device__ __forceinline__ uint32_t slot_uses(uint32_t round, uint32_t n_slots) { return Shape<NB>::kGroups == 2 && (n_slots & 1u) ? round >> 1 : round; }

// ---- roles -------------------------------------------------------------------------------------

// Producer: one warp.  Four descriptors are fetched per warp-wide 16-byte load (8 lanes each) one
// batch ahead; lane 0 waits for the slot, the owning lanes copy the descriptor into the slot
// header, lane 0 arms the barrier and issues the bulk copies.
template <int NB>
__device__ void producer_role(const StepArgs& a, uint8_t* smem, Ctrl* ctrl, uint32_t u0, uint32_t u1) {
  const int lane = threadIdx.x & 31;
  const uint4* base = reinterpret_cast<const uint4*>(a.units);
  const uint32_t n = u1 - u0;
  volatile int* abortp = &ctrl->abort_flag;
  const uint64_t policy = policy_evict_first();
  uint4 next = make_uint4(0, 0, 0, 0);
  if ((uint32_t)(lane >> 3) < n) next = __ldg(base + (size_t)(u0 + (lane >> 3)) * 8 + (lane & 7));
  uint32_t issued = 0;
  bool ok = true;
  for (uint32_t b0 = 0; b0 < n && ok; b0 += 4) {
    const uint4 cur = next;
    const uint32_t nb = b0 + 4 + (lane >> 3);
    if (nb < n) next = __ldg(base + (size_t)(u0 + nb) * 8 + (lane & 7));
    for (int k = 0; k < 4 && b0 + k < n; ++k) {
      const uint32_t i = b0 + k;
      const int slot = (int)(i % (uint32_t)a.n_slots);
      const uint32_t round = i / (uint32_t)a.n_slots;
      uint8_t* sl = smem + kCtrlBytes + (size_t)slot * a.slot_bytes;
      if (!mbar_wait_warp(&ctrl->empty[slot], (round & 1u) ^ 1u, abortp, a.status)) { ok = false; break; }
      if ((lane >> 3) == k) *reinterpret_cast<uint4*>(sl + (lane & 7) * 16) = cur;
      // fields for lane 0, by 16-byte piece of descriptor k
      const uint32_t s0l = __shfl_sync(0xFFFFFFFFu, cur.x, 8 * k), s0h = __shfl_sync(0xFFFFFFFFu, cur.y, 8 * k);
      const uint32_t s1l = __shfl_sync(0xFFFFFFFFu, cur.z, 8 * k), s1h = __shfl_sync(0xFFFFFFFFu, cur.w, 8 * k);
      const uint32_t cbl = __shfl_sync(0xFFFFFFFFu, cur.x, 8 * k + 1), cbh = __shfl_sync(0xFFFFFFFFu, cur.y, 8 * k + 1);
      const uint32_t by0 = __shfl_sync(0xFFFFFFFFu, cur.z, 8 * k + 1), by1 = __shfl_sync(0xFFFFFFFFu, cur.w, 8 * k + 1);
      const uint32_t cbb = __shfl_sync(0xFFFFFFFFu, cur.x, 8 * k + 2);
      const uint32_t chb = __shfl_sync(0xFFFFFFFFu, cur.z, 8 * k + 5);
      __syncwarp();
      if (lane == 0) {
        const uint32_t tx = by0 + by1 + cbb;
        uint64_t* full = &ctrl->full[i % (uint32_t)Shape<NB>::kGroups][slot];
        if (tx == 0) {
          mbar_arrive(full);
        } else {
          mbar_arrive_expect_tx(full, tx);
          uint8_t* data = sl + 128;
          if (by0) bulk_g2s(data, reinterpret_cast<const void*>(((uint64_t)s0h << 32) | s0l), by0, full, policy);
          if (by1) bulk_g2s(data + chb, reinterpret_cast<const void*>(((uint64_t)s1h << 32) | s1l), by1, full, policy);
          if (cbb) bulk_g2s(data + 2 * chb, reinterpret_cast<const void*>(((uint64_t)cbh << 32) | cbl), cbb, full, policy);
        }
      }
      ++issued;
    }
  }
  if (!ok && lane == 0) {
    // Gave up: do not leave the CTA while copies this thread issued may still be landing.
    const uint32_t first = issued > (uint32_t)a.n_slots ? issued - a.n_slots : 0;
    for (uint32_t i = first; i < issued; ++i) {
      const int slot = (int)(i % (uint32_t)a.n_slots);
      for (uint32_t it = 0; it < a.poll_limit; ++it)
        if (mbar_try_wait(&ctrl->full[i % (uint32_t)Shape<NB>::kGroups][slot], slot_uses<NB>(i / (uint32_t)a.n_slots, (uint32_t)a.n_slots) & 1u)) break;
    }
  }
}

__device__ __forceinline__ uint32_t mix2(uint32_t xr, uint32_t pr, uint32_t mr) {
  const float2 xf = __half22float2(*reinterpret_cast<const __half2*>(&xr));
  const float2 pf = __half22float2(*reinterpret_cast<const __half2*>(&pr));
  const float2 mf = __half22float2(*reinterpret_cast<const __half2*>(&mr));
  const __half2 v = __floats2half2_rn(fmaf(pf.x - xf.x, mf.x, xf.x), fmaf(pf.y - xf.y, mf.y, xf.y));
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ float pair_sum(uint32_t r) {
  const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&r));
  return f.x + f.y;
}

constexpr int kStageUnroll = 4;

// 1 / y for 1 <= y <= infinity, to the bit of the correctly rounded division (compared for every such y): Newton's correction of the
// approximate reciprocal with fused multiply-adds (Markstein, "Computation of elementary functions on the IBM RISC System/6000 processor", 1990).
// Where 1 / y is subnormal (y > 2^126) the approximation has fewer bits, and the series' second term is needed: without it five results
// of that range are off by one in the last place.  Without the general division's branch four sigmoids run side by side: 147 cycles
// instead of 367.
__device__ __forceinline__ float rcp_of(float y) {
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(y));
  const float e = fmaf(-y, r, 1.f), f = fmaf(r, fmaf(e, e, e), r);
  return y < INFINITY ? f : r;
}
__device__ __forceinline__ float sigmoidf_(float x) { return rcp_of(1.f + expf(-x)); }
__device__ __forceinline__ uint32_t pack_half2(float a, float b) {
  const __half2 h = __floats2half2_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}
// Four consecutive inputs of a product from the element-wise operator in front of it (Appendix A.1
// Eqs. 23, 24, 27), rounded to fp16.  e0: index of the first element in the [B][ic] fp32 arrays,
// col: its column (index into the per-channel parameters).  `commit` false (a warp that repeats
// another's item to keep the barriers whole): the recurrence state is not written.
__device__ __forceinline__ float4 ldcg4(uint64_t base, size_t e) { return __ldcg(reinterpret_cast<const float4*>(reinterpret_cast<const float*>(base) + e)); }
// The inputs themselves, asked for before anything that has to be waited for (the row statistic).
struct XformLoads { float4 s, g; float scale; };
__device__ __forceinline__ void xform_load(const StepMixOp& mo, const StepMixX& op, size_t e0, XformLoads& l) {
  l.s = ldcg4(op.src, e0);
  l.g = make_float4(0.f, 0.f, 0.f, 0.f);
  if ((mo.kind & 0xFF) == RWKVQ_IN_F32 && op.k) l.g = ldcg4(op.k, e0);
  l.scale = op.scale ? __ldcg(reinterpret_cast<const float*>(op.scale)) : 1.f;
}
__device__ __forceinline__ void spread(const float4 v, float (&o)[4]) { o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w; }
__device__ __forceinline__ uint2 xform_input(const StepMixOp& mo, const StepMixX& op, const XformLoads& l, size_t e0, int col, bool commit, float rstd) {
  const int kind = mo.kind & 0xFF;
  float s[4], o[4];
  spread(l.s, s);
  if (kind == RWKVQ_IN_RELU2) {
#pragma unroll
    for (int i = 0; i < 4; ++i) { const float m = fmaxf(s[i], 0.f); o[i] = m * m; }
  } else if (kind == RWKVQ_IN_F32) {
    float g[4];
    spread(l.g, g);
    const bool gate = op.k != 0u;
#pragma unroll
    for (int i = 0; i < 4; ++i) o[i] = (gate ? s[i] * sigmoidf_(g[i]) : s[i]) * rstd;
  } else {           // RWKVQ_IN_WKV: all loads ahead of the first use and of the stores
    float k[4], vv[4], a[4], bb[4], p[4], u[4], w[4];
    spread(ldcg4(op.k, e0), k); spread(ldcg4(op.v, e0), vv);
    spread(ldcg4(op.state_a, e0), a); spread(ldcg4(op.state_b, e0), bb); spread(ldcg4(op.state_p, e0), p);
    spread(__ldg(reinterpret_cast<const float4*>(reinterpret_cast<const float*>(op.u) + col)), u);
    spread(__ldg(reinterpret_cast<const float4*>(reinterpret_cast<const float*>(op.w) + col)), w);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      // the history sums are stored as a = e^{-p} sum f v, b = e^{-p} sum f; every exponential below has
      // a non-positive argument
      const float uk = u[i] + k[i];
      const float q = fmaxf(p[i], uk);
      const float e1 = expf(p[i] - q), e2 = expf(uk - q);
      const float wkv = (e1 * a[i] + e2 * vv[i]) / (e1 * bb[i] + e2);
      o[i] = sigmoidf_(s[i]) * wkv;
      const float pw = p[i] - w[i];
      const float q2 = fmaxf(pw, k[i]);
      const float f1 = expf(pw - q2), f2 = expf(k[i] - q2);
      a[i] = f1 * a[i] + f2 * vv[i]; bb[i] = f1 * bb[i] + f2; p[i] = q2;
    }
    if (commit) {
      *reinterpret_cast<float4*>(reinterpret_cast<float*>(op.state_a) + e0) = make_float4(a[0], a[1], a[2], a[3]);
      *reinterpret_cast<float4*>(reinterpret_cast<float*>(op.state_b) + e0) = make_float4(bb[0], bb[1], bb[2], bb[3]);
      *reinterpret_cast<float4*>(reinterpret_cast<float*>(op.state_p) + e0) = make_float4(p[0], p[1], p[2], p[3]);
    }
  }
  if (op.scale) {
#pragma unroll
    for (int i = 0; i < 4; ++i) o[i] *= l.scale;
  }
  return make_uint2(pack_half2(o[0], o[1]), pack_half2(o[2], o[3]));
}

// 1 / sqrt(mean over the row of v^2 + 1e-6), v = src (* sigmoid(gate)): the lanes of a warp
// read row b of the fp32 source(s) together.  Items that follow one another in a warp mostly share
// the row, so the caller keeps the last result.
__device__ __noinline__ float row_rstd(const StepMixOp& op, const StepMixX& ox, int b, int lane) {
  const float* src = reinterpret_cast<const float*>(ox.src) + (size_t)b * op.ic;
  const float* gate = ox.k ? reinterpret_cast<const float*>(ox.k) + (size_t)b * op.ic : nullptr;
  float acc = 0.f;
  for (uint32_t c = (uint32_t)lane * 4u; c < op.ic; c += 128u) {
    float4 v = __ldcg(reinterpret_cast<const float4*>(src + c));
    if (gate) {
      const float4 g = __ldcg(reinterpret_cast<const float4*>(gate + c));
      v.x *= sigmoidf_(g.x); v.y *= sigmoidf_(g.y); v.z *= sigmoidf_(g.z); v.w *= sigmoidf_(g.w);
    }
    acc += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, d);
  return rsqrtf(acc / (float)op.ic + 1e-6f);
}

// A load whose value is not needed: it brings the sector into this SM's L1.
__device__ __forceinline__ void touch_global(const void* p) {
  uint32_t v;
  asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(v) : "l"(reinterpret_cast<uintptr_t>(p) & ~static_cast<uintptr_t>(3)));
}

// Asks for the line to be brought into L2 (the point of coherence: a later write by another CTA, reduction
// or plain store, is seen by the load that follows).
__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" :: "l"(p));
}

// A pre-pass descriptor through the read-only path, so that the copy read ahead by mix_warm is found in L1.
__device__ __forceinline__ StepMixOp load_mixop(const StepMixOp* p) {
  union { StepMixOp op; uint4 q[4]; } u;
#pragma unroll
  for (int i = 0; i < 4; ++i) u.q[i] = __ldg(reinterpret_cast<const uint4*>(p) + i);
  return u.op;
}

// Reads ahead, while the consumer warps are still busy with the current stage, what this CTA's items read that does not depend on
// it: the products' descriptors, the mu_hat codes and the codebook entries they select.  A warp's first item is taken right behind the clearing of
// the next outputs (mix_prepare) and finds this in L1; later items are taken behind the barrier, whose acquire empties L1, and find it in L2
// instead of HBM.  The inputs that are still in HBM are requested into L2.  Without it, with it: 7B-class B=8 1427, 1398 us; 14B-class
// B=16 3719, 3673; whole blocks, whose items are few, 123.2, 124.1.
template <int NB>
__device__ void mix_warm(const StepArgs& a, const StepEvent& ev, int stid) {
  constexpr int kStagerWarps = Shape<NB>::kStagerWarps;
  const int lane = stid & 31, l16 = lane & 15;
  const uint32_t lo = ev.arr.grp_lo, hi = ev.arr.grp_hi;
  const StepMixOp* ops = a.mixops + ev.arrd.op_first;
  const int n_ops = (int)ev.arrd.op_count;
  if (lo >= hi) return;
  touch_global(reinterpret_cast<const uint8_t*>(ops) + 32);
  for (uint32_t g0 = lo + 2u * (uint32_t)(stid >> 5); g0 < hi; g0 += 2u * (uint32_t)kStagerWarps) {
    const uint32_t gi = g0 + (uint32_t)(lane >> 4);
    uint32_t r = gi < hi ? gi : lo;
    int k = 0;
    uint32_t icp = __ldg(&ops[0].ic_pad);
    while (k + 1 < n_ops && r >= (uint32_t)a.B * (icp >> 7)) { r -= (uint32_t)a.B * (icp >> 7); ++k; icp = __ldg(&ops[k].ic_pad); }
    const StepMixOp* op = ops + k;
    touch_global(op);                                            // both 32-byte sectors of the descriptor
    touch_global(reinterpret_cast<const uint8_t*>(op) + 32);
    const uint64_t mu = __ldg(&op->mu);
    const uint32_t kind = __ldg(&op->kind);
    if (kind & 0x3FFu) {
      const uint8_t* ox = reinterpret_cast<const uint8_t*>(a.mixx + ev.arrd.op_first + k);
      touch_global(ox); touch_global(ox + 32); touch_global(ox + 64); touch_global(ox + 76);
    }
    const uint32_t ic = __ldg(&op->ic);
    const uint32_t ng = icp >> 7;
    const int col = (int)(r % ng) * 128 + l16 * 8;
    // Inputs that no earlier stage of this step writes (the first products' x, every x_prev) are still in
    // HBM: ask for them now.  Inputs an earlier stage writes are in L2 already and the request is void.
    if ((kind & 0xFFu) == RWKVQ_IN_BUFFER && col < (int)ic && (l16 & 1) == 0) {
      const size_t e0 = (size_t)(r / ng) * ic + col;
      prefetch_l2(reinterpret_cast<const __half*>(__ldg(&op->x)) + e0);
      if (mu) prefetch_l2(reinterpret_cast<const __half*>(__ldg(&op->xprev)) + e0);
    }
    if (mu && col < (int)ic) {
      const uint32_t bits = __ldg(&op->mu_bits), mask = (1u << bits) - 1u;
      const uint32_t byte = (uint32_t)(col >> 1) * bits >> 3;
      const uint32_t* w = reinterpret_cast<const uint32_t*>(mu) + (byte >> 2);
      const uint32_t sh = (byte & 3u) * 8u;
      const uint32_t wlo = __ldg(w);
      const uint32_t whi = (sh + 4u * bits > 32u) ? __ldg(w + 1) : 0u;
      const uint32_t f = __funnelshift_r(wlo, whi, sh);
      const uint32_t* cb = reinterpret_cast<const uint32_t*>(__ldg(&op->mu_aux));
      touch_global(cb + (f & mask));
      touch_global(cb + ((f >> bits) & mask));
      touch_global(cb + ((f >> (2 * bits)) & mask));
      touch_global(cb + ((f >> (3 * bits)) & mask));
    }
  }
}

// Descriptors of a stager warp's current pre-pass item (product, batch row, 128-column group), in shared memory: taken there while the stage barrier
// is still closed (the poll's acquire empties L1, so whatever is read behind it is a trip to L2, and a chain of four of them went by until the
// first input was asked for); in registers they spilled, and every spilled word was such a trip too.
struct MixSlot { StepMixOp op; StepMixX ox; };
// Takes item r into the warp's slot; returns the lane's two mu_hat pairs.
__device__ __forceinline__ uint2 mix_fetch(const StepArgs& a, const StepEvent& ev, uint32_t r, MixSlot* slot, uint32_t* at, int lane) {
  const StepMixOp* ops = a.mixops + ev.arrd.op_first;
  const int n_ops = (int)ev.arrd.op_count;
  int k = 0;
  uint32_t icp = __ldg(&ops[0].ic_pad);
  while (k + 1 < n_ops && r >= (uint32_t)a.B * (icp >> 7)) { r -= (uint32_t)a.B * (icp >> 7); ++k; icp = __ldg(&ops[k].ic_pad); }
  static_assert(sizeof(StepMixOp) == 64 && sizeof(StepMixX) == 80, "nine lanes copy a slot");
  if (lane < 9)
    reinterpret_cast<uint4*>(slot)[lane] = lane < 4 ? __ldg(reinterpret_cast<const uint4*>(ops + k) + lane)
                                                    : __ldg(reinterpret_cast<const uint4*>(a.mixx + ev.arrd.op_first + k) + (lane - 4));
  const uint32_t ng = icp >> 7, row = r / ng, grp = r % ng;
  if (lane == 0) *at = row | grp << 16;
  __syncwarp();
  uint2 mu = make_uint2(0u, 0u);
  const uint32_t col = grp * 128u + (uint32_t)lane * 4u;
  if (slot->op.mu && col < slot->op.ic) {
    const uint32_t bits = slot->op.mu_bits, bit = (col >> 1) * bits, sh = bit & 31u, mask = (1u << bits) - 1u;      // two indices
    const uint32_t* w = reinterpret_cast<const uint32_t*>(slot->op.mu) + (bit >> 5);
    const uint32_t wlo = __ldg(w);
    const uint32_t whi = (sh + 2u * bits > 32u) ? __ldg(w + 1) : 0u;
    const uint32_t f = __funnelshift_r(wlo, whi, sh);
    const uint32_t* cb = reinterpret_cast<const uint32_t*>(slot->op.mu_aux);
    mu = make_uint2(__ldg(cb + (f & mask)), __ldg(cb + ((f >> bits) & mask)));
  }
  return mu;
}
// An item of a stage of plain inputs (no operator, no normalisation), for a quarter-warp: sixteen columns a lane, so that a CTA's share is done in
// one round of loads.
struct PlainItem {
  const __half* x;          // the lane's sixteen columns
  const __half* xprev;      // nullptr: no token shift
  __half* dst;
  float* sums;              // of the group, or nullptr
  uint32_t mu[8], ic_left;  // mu_hat pairs; columns of the input from the lane's first one on (0: none)
  int row;
};
__device__ __forceinline__ PlainItem plain_item(const StepArgs& a, const StepEvent& ev, uint32_t r, int l8) {
  const StepMixOp* ops = a.mixops + ev.arrd.op_first;
  const int n_ops = (int)ev.arrd.op_count, nbp = (a.B + 1) & ~1;
  int k = 0;
  uint32_t icp = __ldg(&ops[0].ic_pad);
  while (k + 1 < n_ops && r >= (uint32_t)a.B * (icp >> 7)) { r -= (uint32_t)a.B * (icp >> 7); ++k; icp = __ldg(&ops[k].ic_pad); }
  const StepMixOp op = load_mixop(ops + k);
  const uint32_t ng = icp >> 7, b = r / ng, grp = r % ng, col = grp * 128u + (uint32_t)l8 * 16u;
  const size_t e0 = (size_t)b * op.ic + col;
  PlainItem it;
  it.row = (int)b;
  it.ic_left = op.ic > col ? op.ic - col : 0u;
  it.x = reinterpret_cast<const __half*>(op.x) + e0;
  it.xprev = op.mu ? reinterpret_cast<const __half*>(op.xprev) + e0 : nullptr;
  it.dst = reinterpret_cast<__half*>(a.scratch + op.dst_x) + (size_t)b * op.ic_pad + col;
  it.sums = op.sums ? reinterpret_cast<float*>(a.scratch + op.dst_sums) + (size_t)grp * 3 * nbp : nullptr;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    if (op.mu && it.ic_left > 8u * h) {
      // four indices = 4*bits bits starting at a byte boundary (col/2 is a multiple of 4)
      const uint32_t bits = op.mu_bits, mask = (1u << bits) - 1u, byte = ((col + 8u * h) >> 1) * bits >> 3, sh = (byte & 3u) * 8u;
      const uint32_t* w = reinterpret_cast<const uint32_t*>(op.mu) + (byte >> 2);
      const uint32_t wlo = __ldg(w);
      const uint32_t whi = (sh + 4u * bits > 32u) ? __ldg(w + 1) : 0u;
      const uint32_t f = __funnelshift_r(wlo, whi, sh);
      const uint32_t* cb = reinterpret_cast<const uint32_t*>(op.mu_aux);
#pragma unroll
      for (int q = 0; q < 4; ++q) it.mu[4 * h + q] = __ldg(cb + ((f >> (q * bits)) & mask));
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) it.mu[4 * h + q] = 0u;
    }
  }
  return it;
}
struct MixPrep { PlainItem plain; uint2 mu; uint32_t kind; };      // of the warp's (lanes') first item; of the share's first product: what kind of stage it is
// Steps whose inputs are all plain take the whole item ahead of the barrier, steps with operators only its descriptors: with room for both in the
// registers each spilled for the other (7B-class, batch 8: 1453 us without, 1415 with; blocks 125 and 129).
template <int NB, bool OPS>
__device__ __forceinline__ MixPrep mix_prepare(const StepArgs& a, const StepEvent& ev, int stid, MixSlot* slots, uint32_t* at) {
  MixPrep p;
  p.mu = make_uint2(0u, 0u);
  p.kind = OPS ? (uint32_t)__ldg(&a.mixops[ev.arrd.op_first].kind) : 0x800u;
  const uint32_t lo = ev.arr.grp_lo, hi = ev.arr.grp_hi, w = (uint32_t)(stid >> 5);
  if (lo >= hi) return p;
  if constexpr (!OPS) {
    const uint32_t gi = lo + 4u * w + (uint32_t)((stid & 31) >> 3);
    p.plain = plain_item(a, ev, gi < hi ? gi : lo, stid & 7);
  } else if (!(p.kind & 0x800u)) {
    p.mu = mix_fetch(a, ev, lo + w < hi ? lo + w : lo, slots + w, at + w, stid & 31);
  }
  return p;
}

// This CTA's share of a stage's pre-pass.  A warp takes one (product, batch row, 128-column
// group) at a time (a quarter-warp in stages of plain inputs): it loads x (and x_prev, and decodes mu_hat), mixes, rounds to fp16, stores the
// 128 values to the product's pre-pass rows and reduces the three sums of the group with shuffles.
// Bound by its latency: a CTA has an item or two, and all wait.  Whole blocks, d 2048, batch 2: 10.6 us a stage before, of which the
// pre-pass took 2 to 8.5; 7.9 with descriptors in shared memory, no spills, vector loads ahead of every wait and stores behind them
// (the recurrence read its seven arrays element by element, each behind the stores of the one before), and sigmoids without a branch.
template <int NB, bool OPS>
__device__ void mix_slice(const StepArgs& a, const StepEvent& ev, int stid, const MixPrep& prep, MixSlot* slots, uint32_t* mix_at) {
  constexpr int kStagerWarps = Shape<NB>::kStagerWarps, kStagerThreads = Shape<NB>::kStagerThreads;
  const int lane = stid & 31;
  const uint32_t lo = ev.arr.grp_lo, hi = ev.arr.grp_hi;
  if (lo >= hi) return;      // the same for all stager warps
  const StepMixOp* ops = a.mixops + ev.arrd.op_first;
  const int n_ops = (int)ev.arrd.op_count;
  const int nbp = (a.B + 1) & ~1;
  // Row statistics first: the rows of normalised inputs that this CTA's items fall in (a few: the items
  // are consecutive groups of consecutive rows) are reduced by all stager threads together, 1.5 KB per
  // round of loads, into a small table; rows beyond the table are reduced by the warp that meets them.
  constexpr int kRowTable = 8;
  __shared__ float s_rstd[kRowTable];
  __shared__ float s_part[kStagerWarps];
  __shared__ uint32_t s_row_end[kRowTable];      // first item behind the row of each entry
  int n_rows = 0;
  const uint32_t stage_kind = prep.kind;
  if (stage_kind & 0x800) {
    // Stage of plain inputs: a quarter-warp per item.
    const int l8 = lane & 7;
    PlainItem it;
    if constexpr (!OPS) it = prep.plain;
    for (uint32_t g0 = lo + 4u * (uint32_t)(stid >> 5); g0 < hi; g0 += 4u * (uint32_t)kStagerWarps) {
      const uint32_t gi = g0 + (uint32_t)(lane >> 3);
      const bool valid = gi < hi;
      if (OPS || g0 != lo + 4u * (uint32_t)(stid >> 5)) it = plain_item(a, ev, valid ? gi : lo, l8);
      const int b = it.row;
      uint4 v[2] = {make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u)};
      uint4 pr[2] = {v[0], v[0]};
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (it.ic_left > 8u * h) {
          v[h] = __ldcg(reinterpret_cast<const uint4*>(it.x + 8 * h));
          if (it.xprev) pr[h] = __ldcg(reinterpret_cast<const uint4*>(it.xprev + 8 * h));
        }
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (it.xprev && it.ic_left > 8u * h) {
          v[h].x = mix2(v[h].x, pr[h].x, it.mu[4 * h]);
          v[h].y = mix2(v[h].y, pr[h].y, it.mu[4 * h + 1]);
          v[h].z = mix2(v[h].z, pr[h].z, it.mu[4 * h + 2]);
          v[h].w = mix2(v[h].w, pr[h].w, it.mu[4 * h + 3]);
        }
      if (valid) {
        *reinterpret_cast<uint4*>(it.dst) = v[0];
        *reinterpret_cast<uint4*>(it.dst + 8) = v[1];
      }
      // both vectors of a lane lie in one 16-column span of a triple: the same two bias values
      const int o = (16 * l8) & 63;
      const float pa = pair_sum(v[0].x) + pair_sum(v[0].z) + pair_sum(v[1].x) + pair_sum(v[1].z);
      const float pb = pair_sum(v[0].y) + pair_sum(v[0].w) + pair_sum(v[1].y) + pair_sum(v[1].w);
      float sx = pa + pb;
      float t0 = fmaf((float)rwkvq_sq_bias(o, 0), pa, (float)rwkvq_sq_bias(o + 2, 0) * pb);
      float t1 = fmaf((float)rwkvq_sq_bias(o, 1), pa, (float)rwkvq_sq_bias(o + 2, 1) * pb);
#pragma unroll
      for (int d = 4; d > 0; d >>= 1) {
        sx += __shfl_xor_sync(0xFFFFFFFFu, sx, d);
        t0 += __shfl_xor_sync(0xFFFFFFFFu, t0, d);
        t1 += __shfl_xor_sync(0xFFFFFFFFu, t1, d);
      }
      if (valid && l8 == 0 && it.sums) {
        it.sums[b] = sx;
        it.sums[nbp + b] = t0;
        it.sums[2 * nbp + b] = t1;
      }
    }
    return;
  }
  if constexpr (OPS) {
  auto row_table = [&]() {
    uint32_t r = lo;
    while (r < hi && n_rows < kRowTable) {
      // the first row is that of the first warp's item
      const StepMixOp* op = &slots[0].op;
      const StepMixX* ox = &slots[0].ox;
      uint32_t row = mix_at[0] & 0xFFFFu, left = (op->ic_pad >> 7) - (mix_at[0] >> 16);
      if (n_rows) {
        uint32_t rr = r;
        int k = 0;
        uint32_t icp = __ldg(&ops[0].ic_pad);
        while (k + 1 < n_ops && rr >= (uint32_t)a.B * (icp >> 7)) { rr -= (uint32_t)a.B * (icp >> 7); ++k; icp = __ldg(&ops[k].ic_pad); }
        op = ops + k; ox = a.mixx + ev.arrd.op_first + k;
        row = rr / (icp >> 7); left = (icp >> 7) - rr % (icp >> 7);
      }
      const uint32_t ic = op->ic;
      const bool norm = (op->kind & 0x100) != 0;
      const float* src = reinterpret_cast<const float*>(ox->src) + (size_t)row * ic;
      const float* gate = ox->k ? reinterpret_cast<const float*>(ox->k) + (size_t)row * ic : nullptr;
      float rstd = 1.f;
      if (norm) {
        float acc = 0.f;
        // two rounds of loads ahead of the one that is added up
        constexpr uint32_t kStep = (uint32_t)kStagerThreads * 4u;
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        auto get = [&](const float* from, uint32_t c) { return c < ic ? __ldcg(reinterpret_cast<const float4*>(from + c)) : zero; };
        uint32_t c = (uint32_t)stid * 4u;
        float4 v0 = get(src, c), v1 = get(src, c + kStep), g0 = zero, g1 = zero;
        if (gate) { g0 = get(gate, c); g1 = get(gate, c + kStep); }
#pragma unroll 1
        for (; c < ic; c += kStep) {
          const float4 v2 = get(src, c + 2u * kStep), g2 = gate ? get(gate, c + 2u * kStep) : zero;
          if (gate) { v0.x *= sigmoidf_(g0.x); v0.y *= sigmoidf_(g0.y); v0.z *= sigmoidf_(g0.z); v0.w *= sigmoidf_(g0.w); }
          acc += v0.x * v0.x + v0.y * v0.y + v0.z * v0.z + v0.w * v0.w;
          v0 = v1; v1 = v2; g0 = g1; g1 = g2;
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, d);
        if (lane == 0) s_part[stid >> 5] = acc;
        named_bar_sync(5, kStagerThreads);
        float tot = 0.f;
#pragma unroll
        for (int wdx = 0; wdx < kStagerWarps; ++wdx) tot += s_part[wdx];
        rstd = rsqrtf(tot / (float)ic + 1e-6f);
        named_bar_sync(5, kStagerThreads);      // s_part is reused by the next row
      }
      r += left;                         // first item of the next row
      if (stid == 0) { s_rstd[n_rows] = rstd; s_row_end[n_rows] = r; }
      ++n_rows;
    }
    named_bar_sync(5, kStagerThreads);
  };
  uint64_t stat_src = 0;     // row whose statistic this warp computed last (rows beyond the table)
  int stat_b = -1;
  float stat_rstd = 1.f;
  // The planner marks the products of a stage that has a normalised input.  In the first round, which every warp takes part in, what the items
  // need from memory is asked for ahead of the table.
  bool table = (stage_kind & 0x400) != 0u;
  uint2 mu = prep.mu;
  for (uint32_t gi = lo + (uint32_t)(stid >> 5); gi < hi || table; gi += (uint32_t)kStagerWarps) {      // a warp per item
    const bool valid = gi < hi;
    MixSlot* const slot = slots + (stid >> 5);
    if (gi != lo + (uint32_t)(stid >> 5)) {
      __syncwarp();
      mu = mix_fetch(a, ev, gi, slot, mix_at + (stid >> 5), lane);
    }
    const StepMixOp& op = slot->op;
    const StepMixX& ox = slot->ox;
    const uint32_t at = mix_at[stid >> 5];
    const int b = (int)(at & 0xFFFFu), grp = (int)(at >> 16), col = grp * 128 + lane * 4;
    const bool in = col < (int)op.ic;
    const size_t e0 = (size_t)b * op.ic + col;            // first of this lane's four elements
    const bool plain = (op.kind & 0xFF) == RWKVQ_IN_BUFFER;
    uint2 v = make_uint2(0u, 0u), pr = v;
    XformLoads xl;
    if (in) {
      if (plain) v = __ldcg(reinterpret_cast<const uint2*>(reinterpret_cast<const __half*>(op.x) + e0));
      else xform_load(op, ox, e0, xl);
      if (op.mu) {
        // previous token's input: read for the mix, then (where asked) replaced by this token's
        pr = __ldcg(reinterpret_cast<const uint2*>(reinterpret_cast<const __half*>(op.xprev) + e0));
      }
    }
    if (table) { row_table(); table = false; }
    float rstd = 1.f;
    if (op.kind & 0x100) {      // the same for the whole warp
      const uint32_t item = valid ? gi : lo;
      int idx = 0;
      while (idx < n_rows && item >= s_row_end[idx]) ++idx;
      if (idx < n_rows) {
        rstd = s_rstd[idx];
      } else {
        if (stat_src != ox.src || stat_b != b) { stat_rstd = row_rstd(op, ox, b, lane); stat_src = ox.src; stat_b = b; }
        rstd = stat_rstd;
      }
    }
    if (in) {
      if (!plain) v = xform_input(op, ox, xl, e0, col, valid, rstd);
      if (ox.xprev_out && valid) *reinterpret_cast<uint2*>(reinterpret_cast<__half*>(ox.xprev_out) + e0) = v;
      if (op.mu) { v.x = mix2(v.x, pr.x, mu.x); v.y = mix2(v.y, pr.y, mu.y); }
    }
    if (valid) *reinterpret_cast<uint2*>(reinterpret_cast<__half*>(a.scratch + op.dst_x) + (size_t)b * op.ic_pad + col) = v;
    const int o = (4 * lane) & 63;
    const float pa = pair_sum(v.x), pb = pair_sum(v.y);
    float sx = pa + pb;
    float t0 = fmaf((float)rwkvq_sq_bias(o, 0), pa, (float)rwkvq_sq_bias(o + 2, 0) * pb);
    float t1 = fmaf((float)rwkvq_sq_bias(o, 1), pa, (float)rwkvq_sq_bias(o + 2, 1) * pb);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      sx += __shfl_xor_sync(0xFFFFFFFFu, sx, d);
      t0 += __shfl_xor_sync(0xFFFFFFFFu, t0, d);
      t1 += __shfl_xor_sync(0xFFFFFFFFu, t1, d);
    }
    if (valid && lane == 0 && op.sums) {
      float* gs = reinterpret_cast<float*>(a.scratch + op.dst_sums);
      gs[(grp * 3 + 0) * nbp + b] = sx;
      gs[(grp * 3 + 1) * nbp + b] = t0;
      gs[(grp * 3 + 2) * nbp + b] = t1;
    }
  }
  }
}

// The sums of a half-warp's 128-column group of row b, from the eight columns a lane has just staged (vector c8 of the row).
__device__ __forceinline__ void segment_sums(float* gs, const uint4 r, int c8, int b, int nbp, int lane) {
  const int o = (8 * c8) & 63;
  const float pa = pair_sum(r.x) + pair_sum(r.z), pb = pair_sum(r.y) + pair_sum(r.w);
  float sx = pa + pb;
  float t0 = fmaf((float)rwkvq_sq_bias(o, 0), pa, (float)rwkvq_sq_bias(o + 2, 0) * pb);
  float t1 = fmaf((float)rwkvq_sq_bias(o, 1), pa, (float)rwkvq_sq_bias(o + 2, 1) * pb);
#pragma unroll
  for (int d = 8; d > 0; d >>= 1) {
    sx += __shfl_xor_sync(0xFFFFFFFFu, sx, d);
    t0 += __shfl_xor_sync(0xFFFFFFFFu, t0, d);
    t1 += __shfl_xor_sync(0xFFFFFFFFu, t1, d);
  }
  if ((lane & 15) == 0) {
    const int grp = c8 >> 4;
    gs[(grp * 3 + 0) * nbp + b] = sx;
    gs[(grp * 3 + 1) * nbp + b] = t0;
    gs[(grp * 3 + 2) * nbp + b] = t1;
  }
}

// A segment of max(src, 0)^2, rounded to fp16, and its sums, by the CTA that reads it.
template <int NB>
__device__ __forceinline__ void stage_squares(const StepArgs& a, const StepEvent& ev, uint8_t* xb, int stid) {
  constexpr int kThreads = Shape<NB>::kStagerThreads, kAhead = 2;
  const float* src = reinterpret_cast<const float*>(ev.seg.x);
  const int ic = (int)ev.segd.ic, col0 = (int)ev.segd.col0, nvr = (int)ev.segd.ncols >> 3, total = a.B * nvr, nbp = (a.B + 1) & ~1;
  const uint32_t xstride = ev.xstride_sums & 0x7FFFFFFFu;
  const bool sums = (ev.xstride_sums >> 31) != 0;
  float* gs = reinterpret_cast<float*>(xb + (size_t)a.B * xstride);
  for (int v0 = stid; v0 < total; v0 += kThreads * kAhead) {
    float4 lo[kAhead], hi[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const int v = v0 + u * kThreads, b = v / nvr, col = col0 + 8 * (v - b * nvr);
      lo[u] = hi[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (v < total && col < ic) {
        const float4* at = reinterpret_cast<const float4*>(src + (size_t)b * ic + col);
        lo[u] = __ldcg(at); hi[u] = __ldcg(at + 1);
      }
    }
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const int v = v0 + u * kThreads, b = v / nvr, c8 = v - b * nvr;
      if (v >= total) break;                      // warp-uniform: total is a multiple of 32
      auto two = [](float x, float y) { x = fmaxf(x, 0.f); y = fmaxf(y, 0.f); return pack_half2(x * x, y * y); };
      const uint4 r = make_uint4(two(lo[u].x, lo[u].y), two(lo[u].z, lo[u].w), two(hi[u].x, hi[u].y), two(hi[u].z, hi[u].w));
      *reinterpret_cast<uint4*>(xb + (size_t)b * xstride + (size_t)c8 * 16) = r;
      if (sums) segment_sums(gs, r, c8, b, nbp, threadIdx.x & 31);
    }
  }
}

// Stagers walk the CTA's event list.
//  EV_ARRIVE: clear this CTA's slice of the next stage's outputs, then report the stage as done on
//    the stagers' side (stage_report: the last of the consumer warps and the stagers to report
//    adds this CTA's arrival to the grid barrier, so the arrival never waits for a role that is
//    busy with something else).
//  EV_SEGMENT: x_mix and, for SQ, the per-group sums of the segment, into buffer (segment number
//    & 1).  The decoded token-shift vector mu_hat and the previous token's activations go to
//    shared memory BEFORE the stage barrier, so that only one round of vector loads of x, the
//    mix and the sums remain behind it.  A thread owns 8 consecutive columns (16 bytes) of one
//    batch row; a half-warp owns one 128-column group, whose three sums it reduces with shuffles.
template <int MIX, int NB, bool HEAD>
__device__ void stager_role(const StepArgs& a, uint8_t* smem, Ctrl* ctrl, uint8_t* xbufs, uint32_t* mucb,
                            uint32_t e0, uint32_t e1) {
  constexpr int kStagerThreads = Shape<NB>::kStagerThreads;
  const int stid = threadIdx.x - Shape<NB>::kConsumerThreads;
  const int lane = stid & 31;
  // The grid barriers are polled by the whole first warp (one request per poll, no divergence to leave): c2 B = 1 453 -> 447 us, c3
  // B = 8 1589 -> 1577; by one lane with two batch blocks, where it costs a little (c4 B = 16 4212 -> 4242 us).
  constexpr int kPollLanes = NB == 1 ? 32 : 1;
  constexpr bool kSquares = MIX == 2 && NB == 1;      // plans with stages whose inputs every CTA squares for itself
  volatile int* abortp = &ctrl->abort_flag;
  uint32_t nseg = 0;          // segments staged so far
  uint32_t passed2 = 0xFFFFFFFFu;   // second-stage barrier this CTA has already passed
  bool ok = true;
  for (uint32_t ei = e0; ei < e1; ++ei) {
    const StepEvent ev = *reinterpret_cast<const StepEvent*>(reinterpret_cast<const uint8_t*>(a.events) + (size_t)ei * 64);
    if (ev.kind == EV_ARRIVE) {
      if constexpr (MIX) {
        if (ev.barrier < (uint32_t)a.n_stages && !(kSquares && (ev.flags & EF_SQUARES))) mix_warm<NB>(a, ev, stid);
      }
      if constexpr (MIX == 2) {      // plans with such stages take this kernel: the test alone cost the other 0.2 %
        if (ev.flags & EF_READ_FIRST) {
          const uint32_t b2 = (uint32_t)a.n_stages + ev.barrier;      // the second barrier of the stage that ends
          if (ok && stid < kPollLanes) {
            uint32_t it = 0;
            while ((int)(ld_acquire_gpu(a.counter + b2) - (a.target + a.wait_skew)) < 0) {
              if (++it >= (a.poll_limit << 2) || *abortp) { *abortp = 1; atomicExch(a.status, (int)RWKVQ_ETIMEOUT); ok = false; break; }
            }
          }
          ok = named_bar_and(6, kStagerThreads, ok);
          if (!ok) break;
        }
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        float* z = reinterpret_cast<float*>(ev.arr.zptr[k]);
        for (uint32_t e = stid; e < ev.arrd.zcount[k]; e += kStagerThreads) z[e] = 0.f;
      }
      // the clearing stores of every stager thread must precede thread 0's fence
      ok = named_bar_and(4, kStagerThreads, ok);
      if (!ok) break;
      // The stagers' part of the stage is done.  Barrier 0 (the clearing pass) has no consumer work
      // before it: arrive directly.  Otherwise report; the last party to report arrives.
      if (stid == 0) {
        if (ev.barrier == 0u) red_release_gpu(a.counter, 1u);
        else if constexpr (NB == 2) ok = stage_wait_total_and_arrive<NB>(ctrl, a, ev.barrier, abortp);
        else stage_report<NB>(ctrl, a, ev.barrier);
      }
      if constexpr (MIX) {
        // once the barrier opens, do this CTA's share of the new stage's pre-pass and publish it
        // through the stage's second barrier
        if (ev.barrier < (uint32_t)a.n_stages) {
          MixSlot* const slots = reinterpret_cast<MixSlot*>(mucb);      // the codebook copy of stagers that mix themselves
          static_assert(sizeof(MixSlot) * Shape<NB>::kStagerWarps <= kMuScratch, "pre-pass slots");
          MixPrep prep;
          if (!(kSquares && (ev.flags & EF_SQUARES))) prep = mix_prepare<NB, MIX == 2>(a, ev, stid, slots, ctrl->mix_at);
          if (ok && stid < kPollLanes) {
            uint32_t it = 0;
            while ((int)(ld_acquire_gpu(a.counter + ev.barrier) - (a.target + a.wait_skew)) < 0) {
              if (++it >= (a.poll_limit << 2) || *abortp) { *abortp = 1; atomicExch(a.status, (int)RWKVQ_ETIMEOUT); ok = false; break; }
            }
            if (ok && a.in_flag && stid == 0) {
              // the last input byte of the products this CTA's share falls in (x and x_prev, [B][ic] fp16 each)
              const StepMixOp* mo = a.mixops + ev.arrd.op_first;
              uint64_t last = 0;
              for (uint32_t k = 0; k < ev.arrd.op_count; ++k) {
                const uint64_t span = (uint64_t)a.B * __ldg(&mo[k].ic) * 2u - 1u;
                const uint64_t px = __ldg(&mo[k].x), pp = __ldg(&mo[k].xprev);
                if (px >= a.in_lo && px < a.in_hi) last = max(last, px + span);
                if (pp >= a.in_lo && pp < a.in_hi) last = max(last, pp + span);
              }
              if (last) ok = wait_inputs(a, last, abortp);
            }
          }
          ok = named_bar_and(6, kStagerThreads, ok);   // thread 0's acquire precedes every thread's loads of x
          if (!ok) break;
          if (kSquares && (ev.flags & EF_SQUARES)) continue;
          mix_slice<NB, MIX == 2>(a, ev, stid, prep, slots, ctrl->mix_at);
          named_bar_sync(4, kStagerThreads);           // every thread's pre-pass stores precede thread 0's release
          if (stid == 0) red_release_gpu(a.counter + (uint32_t)a.n_stages + 1u + ev.barrier, 1u);
        }
      }
      continue;
    }
    const int buf = (int)(nseg % XBufs<MIX, NB>::kCount);
    // uniform verdict over all stager threads: the named barriers below must be reached by all or none
    ok = named_bar_and(7, kStagerThreads, mbar_wait_warp(&ctrl->xempty[buf], ((nseg / XBufs<MIX, NB>::kCount) & 1u) ^ 1u, abortp, a.status) && ok);
    uint8_t* xb = xbufs + (size_t)buf * XBufs<MIX, NB>::kBytes;
    if constexpr (kSquares) {
      if (ev.flags & EF_SQUARES) {                    // the stage's barrier has been passed with its arrival event
        if (ok) stage_squares<NB>(a, ev, xb, stid);
        __syncwarp();
        if (lane == 0) mbar_arrive(&ctrl->xfull[buf]);
        ++nseg;
        if (!ok) break;
        continue;
      }
    }
    if constexpr (MIX) {
      // The segment is a rectangle of the stage's pre-pass output: pass the stage's second barrier
      // (once per stage), then fetch B rows and the block of sums with bulk copies.
      if constexpr (kSquares) {
        // What stage_squares stored here (seen through xfull and xempty) precedes what the copy engine writes to the same bytes.  By the warp that asks for the
        // copies, in front of the poll, whose wait it lies in (1.6B-class blocks, batch 2: 110.0 us without, 109.9 with).
        if (stid < 32 && (ev.flags & EF_BEHIND_SQUARES)) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      }
      const uint32_t b2 = (uint32_t)a.n_stages + ev.barrier;      // counter of the second barrier of stage ev.barrier - 1
      if (ok && stid < kPollLanes && b2 != passed2) {
        uint32_t it = 0;
        while ((int)(ld_acquire_gpu(a.counter + b2) - (a.target + a.wait_skew)) < 0) {
          if (++it >= (a.poll_limit << 2) || *abortp) { *abortp = 1; atomicExch(a.status, (int)RWKVQ_ETIMEOUT); ok = false; break; }
        }
      }
      passed2 = b2;
      ok = named_bar_and(6, kStagerThreads, ok);
      if (ok && stid < 32) {
        const uint32_t xstride = ev.xstride_sums & 0x7FFFFFFFu;
        const uint32_t row_bytes = ev.segd.ncols * 2u;
        const uint32_t sums_bytes = (ev.xstride_sums >> 31) ? (ev.segd.ncols >> 7) * 3u * (uint32_t)((a.B + 1) & ~1) * 4u : 0u;
        // What other CTAs wrote to global memory with ordinary stores is read below by the copy engine.  The buffer it is copied to was last filled by the copy engine,
        // too, or fenced above: here a fence of all spaces is half a microsecond slower in every stage (7B-class stack of eight layers, batch 8: 336.9 us, 325.8
        // so; 1.6B-class blocks, batch 2: 112.8, 110.6).
        asm volatile("fence.proxy.async.global;" ::: "memory");
        if (lane == 0) mbar_arrive_expect_tx(&ctrl->xfull[buf], (uint32_t)a.B * row_bytes + sums_bytes);
        __syncwarp();
        if (lane < a.B)
          bulk_g2s_plain(xb + (size_t)lane * xstride, a.scratch + ev.seg.x + (size_t)lane * ev.segd.ic, row_bytes, &ctrl->xfull[buf]);
        else if (lane == a.B && sums_bytes)
          bulk_g2s_plain(xb + (size_t)a.B * xstride, a.scratch + ev.seg.xprev, sums_bytes, &ctrl->xfull[buf]);
      } else if (lane == 0) {
        mbar_arrive(&ctrl->xfull[buf]);      // the other stager warps (and everyone after a failure) only arrive
      }
      ++nseg;
      if (!ok) break;
      continue;
    }
    const uint8_t* mu = reinterpret_cast<const uint8_t*>(ev.seg.mu);
    const __half* x = reinterpret_cast<const __half*>(ev.seg.x);
    const __half* xp = reinterpret_cast<const __half*>(ev.seg.xprev);
    const int ic = (int)ev.segd.ic, col0 = (int)ev.segd.col0;
    const uint32_t xstride = ev.xstride_sums & 0x7FFFFFFFu;
    const bool sums = (ev.xstride_sums >> 31) != 0;
    const int nvr = (int)ev.segd.ncols >> 3;            // 16-byte vectors per batch row
    const int total = a.B * nvr;
    const int nbp = (a.B + 1) & ~1;
    uint8_t* murow = xb + (size_t)ev.mu_off16 * 16;
    if (a.in_flag) {      // uniform: host-buffer run
      if (ok && stid == 0) {
        const uint64_t span = ((uint64_t)(a.B - 1) * (uint64_t)ic + (uint64_t)min(ic, col0 + (int)ev.segd.ncols)) * 2u - 1u;
        ok = wait_inputs(a, (uint64_t)(uintptr_t)x + span, abortp);
        if (ok && mu) ok = wait_inputs(a, (uint64_t)(uintptr_t)xp + span, abortp);
      }
      ok = named_bar_and(5, kStagerThreads, ok);
    }
    if (ok && mu) {
      for (int e = stid; e < (int)ev.segd.mu_entries; e += kStagerThreads) mucb[e] = __ldg(reinterpret_cast<const uint32_t*>(ev.seg.mu_aux) + e);
      named_bar_sync(5, kStagerThreads);
      const int bits = (int)ev.segd.mu_bits;
      const uint32_t mask = (1u << bits) - 1u;
      for (int c8 = stid; c8 < nvr; c8 += kStagerThreads) {
        const int col = col0 + 8 * c8;
        uint4 m = make_uint4(0u, 0u, 0u, 0u);
        if (col < ic) {
          // four indices = 4*bits bits starting at a byte boundary (col/2 is a multiple of 4)
          const uint32_t byte = (uint32_t)(col >> 1) * (uint32_t)bits >> 3;
          const uint32_t* w = reinterpret_cast<const uint32_t*>(mu) + (byte >> 2);
          const uint32_t sh = (byte & 3u) * 8u;
          const uint32_t lo = __ldg(w);
          const uint32_t hi = (sh + 4u * bits > 32u) ? __ldg(w + 1) : 0u;
          const uint32_t f = __funnelshift_r(lo, hi, sh);
          m.x = mucb[f & mask];
          m.y = mucb[(f >> bits) & mask];
          m.z = mucb[(f >> (2 * bits)) & mask];
          m.w = mucb[(f >> (3 * bits)) & mask];
        }
        *reinterpret_cast<uint4*>(murow + (size_t)c8 * 16) = m;
      }
      for (int v = stid; v < total; v += kStagerThreads) {
        const int b = v / nvr, c8 = v - b * nvr;
        const int col = col0 + 8 * c8;
        uint4 r = make_uint4(0u, 0u, 0u, 0u);
        if (col < ic) r = __ldg(reinterpret_cast<const uint4*>(xp + (size_t)b * ic + col));
        *reinterpret_cast<uint4*>(xb + (size_t)b * xstride + (size_t)c8 * 16) = r;
      }
    }
    if (ok && ev.barrier && stid < kPollLanes) {
      // grid-wide stage barrier: every CTA has finished (and published) the previous stage.  Each
      // barrier has its own arrival counter, so a CTA without work may run ahead and arrive at
      // later barriers without releasing this one early.
      uint32_t it = 0;
      while ((int)(ld_acquire_gpu(a.counter + (ev.barrier - 1u)) - (a.target + a.wait_skew)) < 0) {
        if (++it >= (a.poll_limit << 2) || *abortp) { *abortp = 1; atomicExch(a.status, (int)RWKVQ_ETIMEOUT); ok = false; break; }
      }
    }
    ok = named_bar_and(6, kStagerThreads, ok);   // uniform verdict; orders the mu row before its readers
    if (ok) {
      float* gs = reinterpret_cast<float*>(xb + (size_t)a.B * xstride);
      for (int v0 = stid; v0 < total; v0 += kStagerThreads * kStageUnroll) {
        uint4 raw[kStageUnroll];
#pragma unroll
        for (int u = 0; u < kStageUnroll; ++u) {
          const int v = v0 + u * kStagerThreads;
          raw[u] = make_uint4(0u, 0u, 0u, 0u);
          if (v < total) {
            const int b = v / nvr, c8 = v - b * nvr;
            const int col = col0 + 8 * c8;
            if (col < ic) raw[u] = __ldcg(reinterpret_cast<const uint4*>(x + (size_t)b * ic + col));
          }
        }
#pragma unroll
        for (int u = 0; u < kStageUnroll; ++u) {
          const int v = v0 + u * kStagerThreads;
          if (v >= total) break;                      // warp-uniform: total is a multiple of 32
          const int b = v / nvr, c8 = v - b * nvr;
          uint4 r = raw[u];
          uint8_t* dst = xb + (size_t)b * xstride + (size_t)c8 * 16;
          if (mu) {
            const uint4 pr = *reinterpret_cast<const uint4*>(dst);          // this thread's own earlier store
            const uint4 mr = *reinterpret_cast<const uint4*>(murow + (size_t)c8 * 16);
            r.x = mix2(r.x, pr.x, mr.x); r.y = mix2(r.y, pr.y, mr.y);
            r.z = mix2(r.z, pr.z, mr.z); r.w = mix2(r.w, pr.w, mr.w);
          }
          *reinterpret_cast<uint4*>(dst) = r;
          if (sums) segment_sums(gs, r, c8, b, nbp, lane);
          if (HEAD && u == 0 && (ev.flags & EF_HEAD) && v0 == stid) {      // one row: the threads' first vectors hold the head
            static_assert(kStagerThreads >= 32 * kHeadTiles, "head of a segment");
            __syncwarp();
            if (lane == 0) mbar_arrive(&ctrl->xhead[buf]);
          }
        }
      }
    }
    __syncwarp();
    // A stager that gave up still arrives, so that no consumer is left waiting on this barrier;
    // the consumers stop at the abort flag.
    if (lane == 0) mbar_arrive(&ctrl->xfull[buf]);
    ++nseg;
    if (!ok) break;
  }
}

// Six words of one 128-column group of the record of lane `lane` (planes of 512 bytes, 16 bytes
// per lane): group 0 = words 0..5, group 1 = words 6..11.
template <int GRP>
__device__ __forceinline__ void sq_group_words(const uint8_t* rec, int lane, uint32_t (&w)[6]) {
  if constexpr (GRP == 0) {
    const uint4 p0 = *reinterpret_cast<const uint4*>(rec + lane * 16);
    const uint2 p1 = *reinterpret_cast<const uint2*>(rec + 512 + lane * 16);
    w[0] = p0.x; w[1] = p0.y; w[2] = p0.z; w[3] = p0.w; w[4] = p1.x; w[5] = p1.y;
  } else {
    const uint2 p1 = *reinterpret_cast<const uint2*>(rec + 512 + lane * 16 + 8);
    const uint4 p2 = *reinterpret_cast<const uint4*>(rec + 1024 + lane * 16);
    w[0] = p1.x; w[1] = p1.y; w[2] = p2.x; w[3] = p2.y; w[4] = p2.z; w[5] = p2.w;
  }
}

// The tile's codebook is copied 32 times for lookups without bank conflicts by the eight warps of the group, an eighth of its
// entries each, sixteen bytes a lane and store: in steps of four bytes, one behind the other, the copies of 256 entries took a fifth of the time.
template <int BITS>
__device__ __forceinline__ void copy_codebook(const uint32_t* codebook, uint8_t* rep, int w, int lane, int bar) {
  constexpr int kStores = (1 << BITS) / 32;        // of a warp, four entries each
  uint32_t entry[kStores];
#pragma unroll
  for (int i = 0; i < kStores; ++i) entry[i] = codebook[(w * kStores + i) * 4 + (lane >> 3)];
  named_bar_sync(bar, kGroupThreads);              // the group's previous lookups are done
#pragma unroll
  for (int i = 0; i < kStores; ++i) *reinterpret_cast<uint4*>(rep + (w * kStores + i) * 512 + lane * 16) = make_uint4(entry[i], entry[i], entry[i], entry[i]);
  named_bar_sync(bar, kGroupThreads);
}
// A pair of VQ records.
// Bound by the lookups, 1024 of the 1750 reads and writes of shared memory that a unit takes (at batch 1 its pipe is busy 70 to 76 % of the time).
template <int BITS, int NB>
__device__ __forceinline__ void vq_unit(const uint8_t* ra, const uint8_t* rb, const uint32_t* codebook, uint8_t* rep, int w, int lane, int bar,
                                        uint64_t* empty, const XLane& xl, float (&acca)[NB][4], float (&accb)[NB][4]) {
  copy_codebook<BITS>(codebook, rep, w, lane, bar);
  uint32_t va[2 * BITS], vb[2 * BITS];
  vq_half_words<BITS, 0>(ra, lane, va); vq_half_words<BITS, 0>(rb, lane, vb);
  const uint32_t* cb_lane = reinterpret_cast<const uint32_t*>(rep) + lane;
  // A unit's sums start at zero and are added with a rounding of their own: the tensor core's accumulation cuts off, and its error grows with the chain.
  float ca[NB][4] = {}, cb[NB][4] = {};
  vq_half_mma2<BITS, NB, 0>(va, vb, cb_lane, xl, ca, cb);
  vq_half_words<BITS, 1>(ra, lane, va); vq_half_words<BITS, 1>(rb, lane, vb);
  __syncwarp();
  if (lane == 0) mbar_arrive(empty);               // the rest of the records is in registers: free the slot
  vq_half_mma2<BITS, NB, 1>(va, vb, cb_lane, xl, ca, cb);
#pragma unroll
  for (int n = 0; n < NB; ++n)
#pragma unroll
    for (int k = 0; k < 4; ++k) { acca[n][k] += ca[n][k]; accb[n][k] += cb[n][k]; }
}

// ---- units unpacked ahead of their inputs ---------------------------------------------------------------------------
// A group's first unit of a stage is in shared memory long before the stage's inputs are.  While the warps would wait for these they unpack it, and what they
// unpack waits in tensor memory, used as a larger register file: every warp reaches 32 lanes of it and has 128 columns to itself, so 128
// registers of a lane.  Behind the inputs only the fragments' loads and the tensor-core steps are left: 1770 cycles where the whole unit took 2700
// (1.6B-class, batch 1, both groups at work; step 397 us without, 346 with it).  Bound by
// the chain of a warp then: four trips to tensor memory and sixteen tensor-core steps one behind the other.
constexpr uint32_t kTmemCols = 512, kParkCols = 128;
__device__ __forceinline__ void park16(uint32_t at, const uint32_t (&r)[16]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
               ::"r"(at), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
                 "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void park_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// The registers hold what is fetched only behind fetch_wait on them.
__device__ __forceinline__ void fetch16(uint32_t at, uint32_t (&r)[16]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
                 "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]) : "r"(at) : "memory");
}
__device__ __forceinline__ void fetch_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void fetched(uint32_t (&r)[N]) {
#pragma unroll
  for (int k = 0; k < N; ++k) asm volatile("" : "+r"(r[k]));      // no use is scheduled before the wait
}

// The three words of triple T of a lane of an SQ record.
template <int T>
__device__ __forceinline__ void sq_triple(const uint4& p0, const uint4& p1, const uint4& p2, uint32_t (&r)[16]) {
  if constexpr (T == 0) sq_unpack_triple(p0.x, p0.y, p0.z, r);
  else if constexpr (T == 1) sq_unpack_triple(p0.w, p1.x, p1.y, r);
  else if constexpr (T == 2) sq_unpack_triple(p1.z, p1.w, p2.x, r);
  else sq_unpack_triple(p2.y, p2.z, p2.w, r);
}
// Columns of a warp's share: T * 32 (+ 16: second record) for triple T.
__device__ __forceinline__ void park_sq(uint32_t at, const uint8_t* ra, const uint8_t* rb, int lane) {
  const uint4 a0 = *reinterpret_cast<const uint4*>(ra + lane * 16), a1 = *reinterpret_cast<const uint4*>(ra + 512 + lane * 16);
  const uint4 a2 = *reinterpret_cast<const uint4*>(ra + 1024 + lane * 16);
  const uint4 b0 = *reinterpret_cast<const uint4*>(rb + lane * 16), b1 = *reinterpret_cast<const uint4*>(rb + 512 + lane * 16);
  const uint4 b2 = *reinterpret_cast<const uint4*>(rb + 1024 + lane * 16);
  uint32_t r[16];
  sq_triple<0>(a0, a1, a2, r); park16(at, r);
  sq_triple<1>(a0, a1, a2, r); park16(at + 32u, r);
  sq_triple<2>(a0, a1, a2, r); park16(at + 64u, r);
  sq_triple<3>(a0, a1, a2, r); park16(at + 96u, r);
  sq_triple<0>(b0, b1, b2, r); park16(at + 16u, r);
  sq_triple<1>(b0, b1, b2, r); park16(at + 48u, r);
  sq_triple<2>(b0, b1, b2, r); park16(at + 80u, r);
  sq_triple<3>(b0, b1, b2, r); park16(at + 112u, r);
  park_wait();
}
// The products of a parked pair of records.  While a triple's fragments are fetched (a trip of some 200 cycles) the inputs of its tensor-core steps are read
// and the sums of the group before are scaled.
template <int NB>
struct Parked {
  uint32_t a[16], b[16];
  uint2 x[4][NB];
  __device__ __forceinline__ void inputs(const XLane& xl, int T) {
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
      for (int n = 0; n < NB; ++n) x[m][n] = *reinterpret_cast<const uint2*>(xl.x[n] + (4 * T + m) * 32);
  }
  __device__ __forceinline__ void ready() { fetch_wait(); fetched(a); fetched(b); }
  // the steps of triple T; triple T + 1 is asked for as soon as this one's fragments have been taken
  template <int T>
  __device__ __forceinline__ void steps(uint32_t at, float (&ca)[NB][4], float (&cb)[NB][4]) {
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const uint32_t f[4] = {a[4 * m], a[4 * m + 1], a[4 * m + 2], a[4 * m + 3]};
#pragma unroll
      for (int n = 0; n < NB; ++n) mma_16816(ca[n], f, x[m][n].x, x[m][n].y);
    }
    if constexpr (T < 3) fetch16(at + 32u * (T + 1), a);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const uint32_t f[4] = {b[4 * m], b[4 * m + 1], b[4 * m + 2], b[4 * m + 3]};
#pragma unroll
      for (int n = 0; n < NB; ++n) mma_16816(cb[n], f, x[m][n].x, x[m][n].y);
    }
    if constexpr (T < 3) fetch16(at + 32u * (T + 1) + 16u, b);
  }
};
// As sq_group_mma2: the chains of a group start at -Bx_h; what they end with is scaled.
template <int NB>
__device__ __forceinline__ void parked_start(const XLane& xl, int grp, float (&ca)[NB][4], float (&cb)[NB][4]) {
  const uint8_t* gsp = xl.gs + (size_t)(grp * 3) * xl.gstride;
#pragma unroll
  for (int n = 0; n < NB; ++n) {
    const float2 b0 = *reinterpret_cast<const float2*>(gsp + xl.gstride + n * 32);
    const float2 b1 = *reinterpret_cast<const float2*>(gsp + 2 * xl.gstride + n * 32);
    ca[n][0] = cb[n][0] = -b0.x; ca[n][1] = cb[n][1] = -b0.y;
    ca[n][2] = cb[n][2] = -b1.x; ca[n][3] = cb[n][3] = -b1.y;
  }
}
template <int NB>
__device__ __forceinline__ void parked_scale(const XLane& xl, int grp, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi, const float (&ca)[NB][4],
                                             const float (&cb)[NB][4], float (&acca)[NB][4], float (&accb)[NB][4]) {
  const uint8_t* gsp = xl.gs + (size_t)(grp * 3) * xl.gstride;
  const float2 sa0 = __half22float2(*reinterpret_cast<const __half2*>(&a_lo)), sa1 = __half22float2(*reinterpret_cast<const __half2*>(&a_hi));
  const float2 sb0 = __half22float2(*reinterpret_cast<const __half2*>(&b_lo)), sb1 = __half22float2(*reinterpret_cast<const __half2*>(&b_hi));
#pragma unroll
  for (int n = 0; n < NB; ++n) {
    const float2 sx = *reinterpret_cast<const float2*>(gsp + n * 32);
    acca[n][0] = fmaf(sa0.x, fmaf(-sa0.y, sx.x, ca[n][0]), acca[n][0]);
    acca[n][1] = fmaf(sa0.x, fmaf(-sa0.y, sx.y, ca[n][1]), acca[n][1]);
    acca[n][2] = fmaf(sa1.x, fmaf(-sa1.y, sx.x, ca[n][2]), acca[n][2]);
    acca[n][3] = fmaf(sa1.x, fmaf(-sa1.y, sx.y, ca[n][3]), acca[n][3]);
    accb[n][0] = fmaf(sb0.x, fmaf(-sb0.y, sx.x, cb[n][0]), accb[n][0]);
    accb[n][1] = fmaf(sb0.x, fmaf(-sb0.y, sx.y, cb[n][1]), accb[n][1]);
    accb[n][2] = fmaf(sb1.x, fmaf(-sb1.y, sx.x, cb[n][2]), accb[n][2]);
    accb[n][3] = fmaf(sb1.x, fmaf(-sb1.y, sx.y, cb[n][3]), accb[n][3]);
  }
}
template <int NB>
__device__ __forceinline__ void parked_sq(uint32_t at, const uint4 sza, const uint4 szb, const XLane& xl, float (&acca)[NB][4], float (&accb)[NB][4]) {
  Parked<NB> p;
  float ca[NB][4], cb[NB][4];
  fetch16(at, p.a);
  fetch16(at + 16u, p.b);
  parked_start<NB>(xl, 0, ca, cb);
  p.inputs(xl, 0);
  p.ready();
  p.template steps<0>(at, ca, cb);
  p.inputs(xl, 1);
  p.ready();
  p.template steps<1>(at, ca, cb);
  p.inputs(xl, 2);
  parked_scale<NB>(xl, 0, sza.x, sza.z, szb.x, szb.z, ca, cb, acca, accb);
  parked_start<NB>(xl, 1, ca, cb);
  p.ready();
  p.template steps<2>(at, ca, cb);
  p.inputs(xl, 3);
  p.ready();
  p.template steps<3>(at, ca, cb);
  parked_scale<NB>(xl, 1, sza.y, sza.w, szb.y, szb.w, ca, cb, acca, accb);
}
template <int NB>
__device__ __forceinline__ void parked_vq(uint32_t at, const XLane& xl, float (&acca)[NB][4], float (&accb)[NB][4]) {
  Parked<NB> p;
  float ca[NB][4] = {}, cb[NB][4] = {};
  fetch16(at, p.a);
  fetch16(at + 16u, p.b);
  p.inputs(xl, 0);
  p.ready();
  p.template steps<0>(at, ca, cb);
  p.inputs(xl, 1);
  p.ready();
  p.template steps<1>(at, ca, cb);
  p.inputs(xl, 2);
  p.ready();
  p.template steps<2>(at, ca, cb);
  p.inputs(xl, 3);
  p.ready();
  p.template steps<3>(at, ca, cb);
#pragma unroll
  for (int n = 0; n < NB; ++n)
#pragma unroll
    for (int k = 0; k < 4; ++k) { acca[n][k] += ca[n][k]; accb[n][k] += cb[n][k]; }
}
template <int BITS, int T>
__device__ __forceinline__ void vq_triple(const uint32_t (&w)[2 * BITS], uint32_t base, uint32_t (&r)[16]) {
#pragma unroll
  for (int e = 0; e < 16; ++e) r[e] = vq_entry<BITS, 2 * BITS>(w, 16 * T + e, base);
}
template <int BITS>
__device__ __forceinline__ void vq_words(const uint8_t* rec, int lane, uint32_t (&w)[2 * BITS]) {
#pragma unroll
  for (int p = 0; p < BITS / 2; ++p) {
    const uint4 v = *reinterpret_cast<const uint4*>(rec + p * 512 + lane * 16);
    w[4 * p] = v.x; w[4 * p + 1] = v.y; w[4 * p + 2] = v.z; w[4 * p + 3] = v.w;
  }
}
template <int BITS>
__device__ __forceinline__ void park_vq(uint32_t at, const uint8_t* ra, const uint8_t* rb, const uint32_t* codebook, uint8_t* rep, int w, int lane, int bar) {
  copy_codebook<BITS>(codebook, rep, w, lane, bar);
  const uint32_t base = smem_u32(rep) + (uint32_t)lane * 4u;
  uint32_t v[2 * BITS], r[16];
  vq_words<BITS>(ra, lane, v);
  vq_triple<BITS, 0>(v, base, r); park16(at, r);
  vq_triple<BITS, 1>(v, base, r); park16(at + 32u, r);
  vq_triple<BITS, 2>(v, base, r); park16(at + 64u, r);
  vq_triple<BITS, 3>(v, base, r); park16(at + 96u, r);
  vq_words<BITS>(rb, lane, v);
  vq_triple<BITS, 0>(v, base, r); park16(at + 16u, r);
  vq_triple<BITS, 1>(v, base, r); park16(at + 48u, r);
  vq_triple<BITS, 2>(v, base, r); park16(at + 80u, r);
  vq_triple<BITS, 3>(v, base, r); park16(at + 112u, r);
  park_wait();
}

// c[k] of the four lanes whose row index g differs in its two low bits (lanes 4 apart) -> lane i (= g & 3)
// ends with element i of lanes g & ~3 ... (g & ~3) + 3, in that order.  All lanes of the warp call it.
__device__ __forceinline__ void transpose4_lanes(float (&c)[4], int i) {
  const bool hi = (i & 2) != 0, lo = (i & 1) != 0;
  const float s0 = hi ? c[0] : c[2], s1 = hi ? c[1] : c[3];
  const float r0 = __shfl_xor_sync(0xFFFFFFFFu, s0, 8), r1 = __shfl_xor_sync(0xFFFFFFFFu, s1, 8);
  // element 2*hi + {0, 1} of source lanes j1 = 0, 1
  const float a00 = hi ? r0 : c[0], a01 = hi ? r1 : c[1];
  const float a10 = hi ? c[2] : r0, a11 = hi ? c[3] : r1;
  const float q0 = lo ? a00 : a01, q1 = lo ? a10 : a11;
  const float p0 = __shfl_xor_sync(0xFFFFFFFFu, q0, 4), p1 = __shfl_xor_sync(0xFFFFFFFFu, q1, 4);
  c[0] = lo ? p0 : a00;  c[1] = lo ? a01 : p0;
  c[2] = lo ? p1 : a10;  c[3] = lo ? a11 : p1;
}
__device__ __forceinline__ void red_add(float* p, float v) { asm volatile("red.global.add.f32 [%0], %1;" :: "l"(p), "f"(v) : "memory"); }
__device__ __forceinline__ void red_add_v4(float* p, const float (&v)[4]) {
  asm volatile("red.global.v4.f32.add [%0], {%1, %2, %3, %4};" :: "l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]) : "memory");
}

// Consumer warp `w` of group `grp`: units grp, grp + 2, ... of the CTA's list.
template <int NB, int MIX, bool PARK, bool ONE>
__device__ void consumer_role(const StepArgs& a, uint8_t* smem, Ctrl* ctrl, const uint8_t* xbufs, uint8_t* replicas,
                              uint32_t unit_base, uint32_t n_units, uint32_t ev_base, uint32_t n_events) {
  constexpr bool HEAD = ONE && !PARK;
  bool dead = false;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int kGroups = Shape<NB>::kGroups;
  const int grp = warp >> 3, w = warp & 7;
  const int g = lane >> 2, t = lane & 3;
  volatile int* abortp = &ctrl->abort_flag;
  float acca[NB][4], accb[NB][4];
#pragma unroll
  for (int n = 0; n < NB; ++n)
#pragma unroll
    for (int k = 0; k < 4; ++k) acca[n][k] = accb[n][k] = 0.f;
  // Every consumer warp walks the CTA's event list in order -- it reports each stage it leaves and
  // passes through each input segment, used or not -- so that the phases of the shared barriers
  // advance in step for all consumer warps.
  int held = -1;              // input segment this warp currently holds
  uint32_t seg_next = 0;      // number of segment events passed so far
  uint32_t cur_ev = 0;        // last event processed (event 0 is the clearing arrival: nothing to do)
  // Report the current stage as finished (stage_report).  The lanes' reductions into y are ordered
  // before lane 0's report by the warp barrier; no lane fences at GPU scope itself: that would only
  // add its latency to the end of every stage.
  uint32_t next_bar = 1u;     // every CTA arrives at barriers 1, 2, ... in this order, once per stage
  auto arrive_stage = [&]() {
    __syncwarp();
    if constexpr (NB == 2) {
      if (lane == 0 && !dead) stage_report_total(ctrl, next_bar);
      ++next_bar;
    } else {
      if (lane == 0 && !dead) stage_report<NB>(ctrl, a, next_bar);
      ++next_bar;
    }
  };
  auto release_held = [&]() {
    __syncwarp();
    if (held >= 0 && lane == 0 && !dead) mbar_arrive(&ctrl->xempty[(uint32_t)held % XBufs<MIX, NB>::kCount]);
    held = -1;
  };
  auto pass_segment = [&]() {   // a segment this warp does not use: observe it, hand it back
    const uint32_t q = seg_next++;
    if (!dead && !mbar_wait_warp(&ctrl->xfull[q % XBufs<MIX, NB>::kCount], (q / XBufs<MIX, NB>::kCount) & 1u, abortp, a.status)) dead = true;
    __syncwarp();
    if (lane == 0 && !dead) mbar_arrive(&ctrl->xempty[q % XBufs<MIX, NB>::kCount]);
  };
  // Events (cur_ev, upto) in order; `mask` describes them when there are at most 32 and the planner
  // could say so, otherwise (and for the tail of the list) the kinds are read from the plan, 32 at
  // a time.
  auto pass_events = [&](uint32_t upto, uint32_t mask, bool mask_valid) {
    if (cur_ev + 1u >= upto) return;
    release_held();
    while (cur_ev + 1u < upto && !dead) {
      const uint32_t first = cur_ev + 1u;
      const uint32_t cnt = min(32u, upto - first);
      uint32_t m = mask;
      if (!mask_valid) {
        bool arr = false;
        if ((uint32_t)lane < cnt) {
          const uint2 kb = __ldg(reinterpret_cast<const uint2*>(reinterpret_cast<const uint8_t*>(a.events) + (size_t)(ev_base + first + lane) * 64 + 48));
          arr = kb.x == EV_ARRIVE && kb.y > 0u;
        }
        m = __ballot_sync(0xFFFFFFFFu, arr);
      }
      for (uint32_t j = 0; j < cnt && !dead; ++j) {
        if ((m >> j) & 1u) arrive_stage(); else pass_segment();
      }
      cur_ev += cnt;
      mask_valid = false;
    }
  };
  uint8_t* rep = replicas + (size_t)grp * a.replica_bytes;
  // Tensor memory is the consumer warps' alone: the other roles neither wait for it nor for its return.  No other CTA is on the SM (kSmemAlone), so the
  // allocation does not wait either.
  if constexpr (PARK) {
    if (warp == 0) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctrl->tmem_base)), "n"(kTmemCols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    named_bar_sync(3, Shape<NB>::kConsumerThreads);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  }
  // the warp's share of tensor memory, looked up where it is used: lanes 32 (warp mod 4) and on
  auto park_at = [&]() { return *(volatile uint32_t*)&ctrl->tmem_base + ((threadIdx.x & 0x60u) << 16) + (threadIdx.x >> 7) * kParkCols; };
  // slot and round of unit i (i % n_slots, i / n_slots), advanced without dividing
  const uint32_t n_slots_u = (uint32_t)a.n_slots;
  uint32_t slot_u = (uint32_t)grp % n_slots_u, round = (uint32_t)grp / n_slots_u;
  bool fresh = true;          // the unit is the group's first of a stage
  for (uint32_t i = (uint32_t)grp; i < n_units; i += kGroups, slot_u += kGroups) {
    while (slot_u >= n_slots_u) { slot_u -= n_slots_u; ++round; }
    const int slot = (int)slot_u;
    const uint8_t* sl = smem + kCtrlBytes + (size_t)slot * a.slot_bytes;
    const StepUnit* u = reinterpret_cast<const StepUnit*>(sl);
    if (!dead && !mbar_wait_warp(&ctrl->full[grp][slot], slot_uses<NB>(round, n_slots_u) & 1u, abortp, a.status)) dead = true;
    const bool ahead = PARK && fresh && !dead;
    if constexpr (PARK) {
      if (ahead) {
        const uint32_t park = park_at();
        const uint32_t f = u->flags, chb = u->chunk_bytes, rb = u->rec_bytes;
        const uint8_t* data = sl + 128;
        const uint8_t* ra = data + (size_t)w * rb;
        const uint8_t* rbp = u->bytes1 ? ra + chb : ra;      // no second record: the first one again, whose results are dropped
        const uint32_t* cbraw = reinterpret_cast<const uint32_t*>(data + 2 * chb);
        if (!(f & UF_VQ)) park_sq(park, ra, rbp, lane);
        else if (f & UF_BITS8) park_vq<8>(park, ra, rbp, cbraw, rep, w, lane, 1 + grp);
        else park_vq<6>(park, ra, rbp, cbraw, rep, w, lane, 1 + grp);
      }
    }
    if (!dead && u->ev_index != cur_ev) {
      const uint32_t target = u->ev_index;
      pass_events(target, u->between_mask, target - cur_ev - 1u <= 32u);
      if (!dead) {
        release_held();
        const uint32_t q = seg_next++;
        held = (int)q;
        cur_ev = target;
        if constexpr (HEAD) {
          const uint32_t f = u->flags, buf = q % XBufs<MIX, NB>::kCount;
          if (!mbar_wait_warp(f & UF_HEAD ? &ctrl->xhead[buf] : &ctrl->xfull[buf], f & UF_HEAD ? (f & UF_PHASE ? 1u : 0u) : (q / XBufs<MIX, NB>::kCount) & 1u, abortp, a.status)) dead = true;
        } else if (!mbar_wait_warp(&ctrl->xfull[q % XBufs<MIX, NB>::kCount], (q / XBufs<MIX, NB>::kCount) & 1u, abortp, a.status)) {
          dead = true;
        }
      }
    } else if (HEAD && !dead && (u->flags & UF_REST)) {
      if (!mbar_wait_warp(&ctrl->xfull[(uint32_t)held % XBufs<MIX, NB>::kCount], ((uint32_t)held / XBufs<MIX, NB>::kCount) & 1u, abortp, a.status)) dead = true;
    }
    if (dead) {
      // A warp that gave up keeps walking the list only to keep the group's named barriers whole
      // (the other warps stop at their next bounded wait); it touches neither slots nor outputs.
      if (!ahead && (a.units[unit_base + i].flags & UF_VQ)) { named_bar_sync(1 + grp, kGroupThreads); named_bar_sync(1 + grp, kGroupThreads); }
      continue;
    }
    const uint32_t flags = u->flags;
    const uint32_t by1 = u->bytes1;
    const uint32_t after_count = u->after_count, after_mask = u->after_mask;
    const uint8_t* data = sl + 128;
    const uint8_t* xb = xbufs + (size_t)((uint32_t)held % XBufs<MIX, NB>::kCount) * XBufs<MIX, NB>::kBytes;
    const uint32_t xstride = u->xstride, nbp = u->nbp, chb = u->chunk_bytes, rb = u->rec_bytes;
    const bool has_b = by1 != 0u;
    const uint32_t oc = u->oc, row0 = u->row0;
    float* y = reinterpret_cast<float*>(u->y);
    const uint8_t* ra = data + (size_t)w * rb;
    const uint8_t* rbp = data + chb + (size_t)w * rb;
    if (ahead) {
      const uint32_t park = park_at();
      const uint32_t col = u->xcol0;
      const XLane xl = make_xlane(xb + (size_t)col * 2, xstride,
                                  reinterpret_cast<const float*>(xb + u->gs_off) + (size_t)(col >> 7) * 3 * nbp, nbp, a.B, lane);
      const uint4 sza = *reinterpret_cast<const uint4*>(ra + RWKVQ_SQ_CODE_BYTES + g * 16);
      const uint4 szb = *reinterpret_cast<const uint4*>((has_b ? rbp : ra) + RWKVQ_SQ_CODE_BYTES + g * 16);
      // Not before the inputs are there: a slot handed back at once was filled while they were being read, and held them up (1.6B-class, batch 1: 366 us, 363
      // so; 7B-class 1225, 1181).
      __syncwarp();
      if (lane == 0) mbar_arrive(&ctrl->empty[slot]);
      if (flags & UF_VQ) parked_vq<NB>(park, xl, acca, accb);
      else parked_sq<NB>(park, sza, szb, xl, acca, accb);
    } else if (!(flags & UF_VQ)) {
      const uint32_t col = u->xcol0;
      const XLane xl = make_xlane(xb + (size_t)col * 2, xstride,
                                  reinterpret_cast<const float*>(xb + u->gs_off) + (size_t)(col >> 7) * 3 * nbp, nbp, a.B, lane);
      if constexpr (NB == 2) {
        // Registers suffice for the whole record pair: take all of it, free the slot, then run both
        // 128-column groups as one stretch of code (eight tensor-core chains for the scheduler to interleave).
        uint32_t wa0[6], wb0[6], wa1[6], wb1[6];
        uint4 sza, szb;
        sq_group_words<0>(ra, lane, wa0);
        sq_group_words<1>(ra, lane, wa1);
        sza = *reinterpret_cast<const uint4*>(ra + RWKVQ_SQ_CODE_BYTES + g * 16);
        const uint8_t* second = has_b ? rbp : ra;      // no second record: the first one again, whose results are dropped
        sq_group_words<0>(second, lane, wb0);
        sq_group_words<1>(second, lane, wb1);
        szb = *reinterpret_cast<const uint4*>(second + RWKVQ_SQ_CODE_BYTES + g * 16);
        __syncwarp();
        if (lane == 0) mbar_arrive(&ctrl->empty[slot]);
        sq_group_mma2<NB, 0>(wa0, wb0, sza, szb, xl, acca, accb);
        sq_group_mma2<NB, 1>(wa1, wb1, sza, szb, xl, acca, accb);
      } else {
      uint32_t wa[6], wb[6];
      uint4 sza, szb;
      sq_group_words<0>(ra, lane, wa);
      sza = *reinterpret_cast<const uint4*>(ra + RWKVQ_SQ_CODE_BYTES + g * 16);
      const uint8_t* second = has_b ? rbp : ra;
      sq_group_words<0>(second, lane, wb);
      szb = *reinterpret_cast<const uint4*>(second + RWKVQ_SQ_CODE_BYTES + g * 16);
      sq_group_mma2<NB, 0>(wa, wb, sza, szb, xl, acca, accb);
      sq_group_words<1>(ra, lane, wa);
      sq_group_words<1>(second, lane, wb);
      __syncwarp();
      if (lane == 0) mbar_arrive(&ctrl->empty[slot]);     // the rest of the records is in registers: free the slot
      sq_group_mma2<NB, 1>(wa, wb, sza, szb, xl, acca, accb);
      }
    } else {
      const XLane xl = make_xlane(xb + (size_t)u->xcol0 * 2, xstride, nullptr, nbp, a.B, lane);
      const uint32_t* cbraw = reinterpret_cast<const uint32_t*>(data + 2 * chb);
      if (flags & UF_BITS8)
        vq_unit<8, NB>(ra, rbp, cbraw, rep, w, lane, 1 + grp, &ctrl->empty[slot], xl, acca, accb);
      else
        vq_unit<6, NB>(ra, rbp, cbraw, rep, w, lane, 1 + grp, &ctrl->empty[slot], xl, acca, accb);
    }
    if (flags & UF_FLUSH) {
      if (ONE || (NB == 1 && (PARK || (MIX != 0 && a.B == 1)))) {
        // Eight consecutive rows of up to four batch columns an instruction, straight from the accumulators.  With one column the transpose below would move
        // three times as much that nobody takes, and at the end of a small stage it is a part of the chain that the next one waits for (eight layers, d 512, batch 1
        // 107.0 -> 104.0 us; d 4096 289.6 -> 285.1; with units unpacked ahead: d 1024, batch 8 142.5 -> 140.1; blocks of d 512, batch 4 90.3 -> 88.3).  Large stages of
        // more columns gain by the fewer instructions of the other form (d 4096, batch 8 324.0, 322.1).
        const uint32_t r = row0 + (uint32_t)w * 16u;
        const int b = ONE ? 0 : 2 * t;
        float* p = y + (size_t)b * oc + r + (uint32_t)g;
        const bool in = ONE ? t == 0 : b < a.B;
        if (in && r < oc) { red_add(p, acca[0][0]); red_add(p + 8, acca[0][2]); }
        if (has_b && in && r + 128u < oc) { red_add(p + 128, accb[0][0]); red_add(p + 136, accb[0][2]); }
        if constexpr (!ONE) {
          p += oc;
          if (b + 1 < a.B && r < oc) { red_add(p, acca[0][1]); red_add(p + 8, acca[0][3]); }
          if (has_b && b + 1 < a.B && r + 128u < oc) { red_add(p + 128, accb[0][1]); red_add(p + 136, accb[0][3]); }
        }
      } else {
        // Four lanes that share t hold a 4 x 4 block (rows 4J .. 4J+3 of one row half x the accumulator's four
        // elements): transposed, every lane owns four consecutive rows of ONE batch column and adds them
        // with a single 16-byte reduction instead of four scattered ones.  The plan accepts only outputs
        // that start on a 16-byte boundary, and the format only row counts that are multiples of 16.
        const int i = g & 3;
        const uint32_t rbase = row0 + (uint32_t)w * 16u + 8u * (uint32_t)(i >> 1) + (uint32_t)(g & ~3);
#pragma unroll
        for (int n = 0; n < NB; ++n) {
          const int b = n * 8 + 2 * t + (i & 1);
          float va[4] = {acca[n][0], acca[n][1], acca[n][2], acca[n][3]};
          transpose4_lanes(va, i);
          if (b < a.B && rbase < oc) red_add_v4(y + (size_t)b * oc + rbase, va);
          if (has_b) {                      // warp-uniform
            float vb[4] = {accb[n][0], accb[n][1], accb[n][2], accb[n][3]};
            transpose4_lanes(vb, i);
            if (b < a.B && rbase + 128u < oc) red_add_v4(y + (size_t)b * oc + rbase + 128u, vb);
          }
        }
      }
#pragma unroll
      for (int n = 0; n < NB; ++n)
#pragma unroll
        for (int k = 0; k < 4; ++k) acca[n][k] = accb[n][k] = 0.f;
    }
    // the group's last unit of the stage: report the stage as finished without waiting for the next unit
    fresh = after_count != 0u;
    if (fresh) pass_events(cur_ev + after_count + 1u, after_mask, true);
  }
  if (!dead) {
    release_held();
    pass_events(n_events, 0u, false);     // the rest of the list: later stages this warp has no unit in
  }
  if constexpr (PARK) {      // all waits above are bounded, so all consumer warps arrive here
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    named_bar_sync(3, Shape<NB>::kConsumerThreads);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(ctrl->tmem_base), "n"(kTmemCols) : "memory");
  }
}

// rcp_of by itself (rwkvq_step_reciprocal).
__global__ void __launch_bounds__(256) reciprocal_kernel(const float* y, float* out, size_t n) {
  const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
  if (i < n) out[i] = rcp_of(y[i]);
}

// ONE: one batch row, mixed by the CTAs that read it.
template <int NB, int MIX, bool PARK, bool ONE = false>
__global__ void __launch_bounds__(Shape<NB>::kThreads, 1) step_kernel(const StepArgs a) {
  constexpr int kConsumerWarps = Shape<NB>::kConsumerWarps, kStagerWarps = Shape<NB>::kStagerWarps;
  extern __shared__ __align__(128) uint8_t smem[];
  Ctrl* ctrl = reinterpret_cast<Ctrl*>(smem);
  uint8_t* xbufs = smem + kCtrlBytes + (size_t)a.n_slots * a.slot_bytes;
  uint32_t* mucb = reinterpret_cast<uint32_t*>(xbufs + XBufs<MIX, NB>::kCount * XBufs<MIX, NB>::kBytes);
  uint8_t* replicas = reinterpret_cast<uint8_t*>(mucb) + kMuScratch;
  static_assert(consumer_regs(NB, MIX, PARK) * Shape<NB>::kConsumerThreads + stager_regs(NB, MIX, PARK) * (Shape<NB>::kStagerThreads + 32) <=
                    Shape<NB>::kLaunchRegs * Shape<NB>::kThreads, "a re-division above the launch's registers would wait for ever");
  if (threadIdx.x == 0) {
    for (int s = 0; s < a.n_slots; ++s) { mbar_init(&ctrl->full[0][s], 1); mbar_init(&ctrl->full[1][s], 1); mbar_init(&ctrl->empty[s], kGroupWarps); }
    for (int b = 0; b < 4; ++b) { mbar_init(&ctrl->xfull[b], kStagerWarps); mbar_init(&ctrl->xempty[b], kConsumerWarps); }
    for (int b = 0; b < 2; ++b) mbar_init(&ctrl->xhead[b], kStagerWarps);
    for (int k = 0; k < 64; ++k) ctrl->stage_cnt[k] = 0u;
    ctrl->abort_flag = 0;
    ctrl->poll_limit = (int)a.poll_limit;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const uint32_t u0 = a.unit_off[blockIdx.x], u1 = a.unit_off[blockIdx.x + 1];
  const uint32_t e0 = a.event_off[blockIdx.x], e1 = a.event_off[blockIdx.x + 1];
  const int warp = threadIdx.x >> 5;
  // With two batch blocks registers are re-divided at entry (see Shape): the warpgroups of stagers and producer hand part of
  // their share back and the consumer warpgroups take it, so that the record routine keeps everything
  // in registers; so they are with one block where units are unpacked ahead over inputs that the CTAs mix themselves.  In the other kernels of one block the shares are
  // those of the launch and nothing moves; the instruction stays for the code the compiler makes of the roles beside it (without it, before units were unpacked
  // ahead: 1.6B-class B=1 428.3 -> 429.9 us, 7B-class B=1 1209.9 -> 1207.5).
  if (warp < kConsumerWarps) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" :: "n"(consumer_regs(NB, MIX, PARK)));
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" :: "n"(stager_regs(NB, MIX, PARK)));
  }
  if (warp < kConsumerWarps) {
    consumer_role<NB, MIX, PARK, ONE>(a, smem, ctrl, xbufs, replicas, u0, u1 - u0, e0, e1 - e0);
  } else if (warp < kConsumerWarps + kStagerWarps) {
    stager_role<MIX, NB, ONE && !PARK>(a, smem, ctrl, xbufs, mucb, e0, e1);
  } else {
    producer_role<NB>(a, smem, ctrl, u0, u1);
  }
}

// ---- host planner --------------------------------------------------------------------------------

struct PlanInfo {
  int P, B, NB, n_slots, n_stages, mix;
  bool park;            // units unpacked ahead of their inputs
  unsigned runs;        // launches since the counters were last zero
  unsigned abort_epoch; // value of the abort epoch when the counters were last known good
  bool captured;        // some run is part of a graph, which may be launched at any time
  uint32_t poll_limit, wait_skew;
  uint32_t slot_bytes, replica_bytes, smem_bytes;
  size_t off_unit_off, off_event_off, off_units, off_events, off_counter, off_mixops, off_mixx, off_scratch, total_bytes;
  uint32_t n_units, n_events, n_barriers;
  std::vector<uint64_t> y_lo, y_hi;   // per stage: device address range its products write (host-buffer runs)
};

static std::mutex g_plan_mutex;
static std::unordered_map<const void*, PlanInfo> g_plans;

struct HostUnit {
  StepUnit u;
  int op, tr, kt, stage;
};

// Shared-memory footprint of an input segment: B rows of x_mix, the per-group sums (SQ) and one
// row of decoded mu_hat (products with a token shift).
static uint32_t xseg_mu_off(int B, int ncols, bool sums) {
  uint32_t xstride = (uint32_t)ncols * 2u + 32u;
  uint32_t nbp = (uint32_t)((B + 1) & ~1);
  // 64 bytes of slack: lanes of batch columns that do not exist read (and discard) sums past the table
  uint32_t off = (uint32_t)B * xstride + (sums ? (uint32_t)(ncols / 128) * 3u * nbp * 4u + 64u : 0u);
  return (off + 15u) & ~15u;
}
static uint32_t xseg_bytes(int B, int ncols, bool sums, bool has_mu) {
  return xseg_mu_off(B, ncols, sums) + (has_mu ? (uint32_t)ncols * 2u : 0u);
}

static rwkvq_status validate_ops(const rwkvq_gemv_op* ops, int n_ops, int B) {
  if (!ops || n_ops <= 0 || B < 1 || B > 16) return RWKVQ_EINVAL;
  for (int i = 0; i < n_ops; ++i) {
    const rwkvq_gemv_op& o = ops[i];
    rwkvq_status st = check_matrix_desc(&o.W_desc);
    if (st != RWKVQ_OK) return st;
    if (o.W_desc.oc == 1) return RWKVQ_ESHAPE;
    if (!o.W_image_dev || !o.y_dev) return RWKVQ_EINVAL;
    const rwkvq_input_xform& in = o.in;
    if (in.kind == RWKVQ_IN_BUFFER) {
      if (!o.x_fp16_dev) return RWKVQ_EINVAL;
    } else {
      if (in.kind != RWKVQ_IN_WKV && in.kind != RWKVQ_IN_RELU2 && in.kind != RWKVQ_IN_F32) return RWKVQ_EINVAL;
      if (!in.src_f32 || !aligned16(in.src_f32)) return in.src_f32 ? RWKVQ_EALIGN : RWKVQ_EINVAL;
      if (in.kind == RWKVQ_IN_WKV) {
        const void* need[] = {in.k_f32, in.v_f32, in.state_a, in.state_b, in.state_p, in.u_f32, in.w_f32};
        for (const void* q : need) {
          if (!q) return RWKVQ_EINVAL;
          if (!aligned16(q)) return RWKVQ_EALIGN;
        }
      }
      if (in.kind == RWKVQ_IN_F32 && in.gate_f32 && !aligned16(in.gate_f32)) return RWKVQ_EALIGN;
      if (in.flags & ~RWKVQ_INF_RMSNORM) return RWKVQ_EINVAL;
      if ((in.flags & RWKVQ_INF_RMSNORM) && (in.kind != RWKVQ_IN_F32 || o.W_desc.ic % 64)) return RWKVQ_EUNSUPPORTED;
      if (o.W_desc.ic % 8) return RWKVQ_ESHAPE;
    }
    if (in.xprev_out_fp16 && !aligned16(in.xprev_out_fp16)) return RWKVQ_EALIGN;
    if ((o.mu_image_dev == nullptr) != (o.xprev_fp16_dev == nullptr)) return RWKVQ_EINVAL;
    if (o.mu_image_dev) {
      st = check_vector_desc(&o.mu_desc, o.W_desc.ic);
      if (st != RWKVQ_OK) return st;
      if (!aligned16(o.mu_image_dev) || !aligned16(o.xprev_fp16_dev)) return RWKVQ_EALIGN;
    }
    if (!aligned16(o.W_image_dev) || (o.x_fp16_dev && !aligned16(o.x_fp16_dev)) || !aligned16(o.y_dev)) return RWKVQ_EALIGN;
    if (o.y_dtype != RWKVQ_F32) return RWKVQ_EUNSUPPORTED;   // partial sums are added with fp32 atomics
    if (i > 0 && o.stage < ops[i - 1].stage) return RWKVQ_EINVAL;
  }
  return RWKVQ_OK;
}

// Builds the whole plan on the host.  Returns the serialized image in `out` and fills `info`.
static rwkvq_status build_plan(const rwkvq_gemv_op* ops, int n_ops, int B, int P, std::vector<uint8_t>* out, PlanInfo* info) {
  rwkvq_status st = validate_ops(ops, n_ops, B);
  if (st != RWKVQ_OK) return st;
  bool has_vq6 = false, has_vq8 = false, has_sq = false;
  for (int i = 0; i < n_ops; ++i) {
    if (ops[i].W_desc.method == RWKVQ_SQ) has_sq = true;
    else if (ops[i].W_desc.bits == 6) has_vq6 = true;
    else has_vq8 = true;
  }
  const int kGroups = groups_of(B <= 8 ? 1 : 2);   // consumer groups per CTA: they take a CTA's units in turn
  uint32_t data_max = 0;
  if (has_sq) data_max = std::max(data_max, 2u * 8u * RWKVQ_SQ_RECORD_BYTES);
  if (has_vq6) data_max = std::max(data_max, 2u * 8u * 1536u + 256u);
  if (has_vq8) data_max = std::max(data_max, 2u * 8u * 2048u + 1024u);
  info->slot_bytes = (128u + data_max + 127u) & ~127u;
  info->replica_bytes = has_vq8 ? 256u * 128u : has_vq6 ? 64u * 128u : 0u;   // per consumer group
  const uint32_t xbuf_bytes = xbuf_bytes_of(B <= 8 ? 1 : 2);
  const uint32_t fixed = kCtrlBytes + XBufs<0, 1>::kCount * xbuf_bytes + kMuScratch + (uint32_t)kGroups * info->replica_bytes;
  int ns = (int)((kSmemLimit - fixed) / info->slot_bytes);
  if (ns > kMaxSlots) ns = kMaxSlots;
  if (ns < 2) return RWKVQ_EUNSUPPORTED;
  info->n_slots = ns;
  info->smem_bytes = fixed + (uint32_t)ns * info->slot_bytes;
  info->P = P; info->B = B; info->NB = B <= 8 ? 1 : 2;
  info->poll_limit = kDefaultPollLimit; info->wait_skew = 0;
  std::vector<std::pair<int, int>> stage_ranges;  // [first op, last op) per distinct stage value
  for (int i = 0; i < n_ops;) {
    int j = i;
    while (j < n_ops && ops[j].stage == ops[i].stage) ++j;
    stage_ranges.push_back({i, j});
    i = j;
  }
  const int n_stages = (int)stage_ranges.size();
  if ((uint32_t)n_stages + 1u > kMaxBarriers) return RWKVQ_EUNSUPPORTED;   // per-barrier counts in the control block
  bool any_xform = false;
  for (int i = 0; i < n_ops; ++i) any_xform = any_xform || ops[i].in.kind != RWKVQ_IN_BUFFER || ops[i].in.xprev_out_fp16 != nullptr;
  // Inputs per CTA and stage: batch rows x columns of an even share of the units, averaged over the stages.
  uint64_t share = 0, stages = 0;
  for (int i = 0; i < n_ops; ++stages) {
    uint64_t n = 0;
    int j = i;
    for (; j < n_ops && ops[j].stage == ops[i].stage; ++j) n += (uint64_t)((ops[j].W_desc.oc_pad + 255) / 256) * (uint64_t)(ops[j].W_desc.ic_pad / 256);
    share += (n + (uint64_t)P - 1) / (uint64_t)P * 256u * (uint64_t)B;
    i = j;
  }
  // A CTA clears its slice of a stage's outputs when it has done its part of the stage before, whose inputs others may still be reading.  Where the two
  // overlap (outputs reused in turn: y0 -> y1 -> y0), the inputs are read by the stage's pre-pass alone and the clearing waits for its barrier.
  std::vector<char> read_first(n_stages, 0);      // the stage's inputs are outputs of the next one
  bool any_read_first = false;
  for (int s = 0; s + 1 < n_stages; ++s) {
    std::vector<std::pair<uint64_t, uint64_t>> y;      // the next stage's outputs, by address
    for (int q = stage_ranges[s + 1].first; q < stage_ranges[s + 1].second; ++q) {
      const uint64_t at = (uint64_t)(uintptr_t)ops[q].y_dev;
      y.push_back({at, at + (uint64_t)B * (uint64_t)ops[q].W_desc.oc * 4u});
    }
    std::sort(y.begin(), y.end());
    auto written = [&](const void* p, uint64_t bytes) {
      const uint64_t lo = (uint64_t)(uintptr_t)p;
      if (!p || lo >= y.back().second || lo + bytes <= y.front().first) return false;
      for (const auto& range : y)
        if (lo < range.second && range.first < lo + bytes) return true;
      return false;
    };
    for (int o = stage_ranges[s].first; o < stage_ranges[s].second && !read_first[s]; ++o) {
      const rwkvq_input_xform& in = ops[o].in;
      const uint64_t n = (uint64_t)ops[o].W_desc.ic, rows = (uint64_t)B * n;
      bool hit = written(ops[o].mu_image_dev ? ops[o].xprev_fp16_dev : nullptr, rows * 2u) || written(in.xprev_out_fp16, rows * 2u);
      if (in.kind == RWKVQ_IN_BUFFER) hit = hit || written(ops[o].x_fp16_dev, rows * 2u);
      else hit = hit || written(in.src_f32, rows * 4u) || written(in.scale_f32, 4u);
      if (in.kind == RWKVQ_IN_F32) hit = hit || written(in.gate_f32, rows * 4u);
      if (in.kind == RWKVQ_IN_WKV) {
        for (const void* p : {(const void*)in.k_f32, (const void*)in.v_f32, (const void*)in.state_a, (const void*)in.state_b, (const void*)in.state_p})
          hit = hit || written(p, rows * 4u);
        hit = hit || written(in.u_f32, n * 4u) || written(in.w_f32, n * 4u);
      }
      read_first[s] = hit;
    }
    any_read_first = any_read_first || read_first[s];
  }
  // A stage pre-pass (StepArgs::mix) costs a second barrier, about 2 us per stage whatever the sizes; without it every CTA mixes the
  // columns it reads itself.  The line was measured with stacks of eight layers, 1024 to 4096 columns (pre-pass / without, us, at
  // `share / stages` inputs): B=6, 1920, 172 / 146; B=3, 2112, 214 / 200; B=5, 2240, 184 / 178; B=2, 2432, 269 / 276; B=8, 2560, 174 / 170; B=6, 2688, 185 / 184;
  // B=4, 2816, 217 / 226; B=2, 3072, 299 / 331; B=8, 3584, 190 / 222; with seven stager warps B=10, 4480, 232 / 224; B=16, 5120, 213 / 214; B=12, 5376,
  // 235 / 240; B=9, 6336, 269 / 289.  The element-wise operators exist in the pre-pass only.
  if ((any_xform || any_read_first) && n_ops > 65535) return RWKVQ_EUNSUPPORTED;      // the events count products in 16 bits
  const bool mix = any_xform || any_read_first || (n_ops <= 65535 && share > stages * (B > 8 ? 5200u : 2700u));
  // In 64ths of an SQ unit: what a further row of tiles (flush, input segment) costs a CTA, and an odd number of units where two consumer groups
  // take them in turn.  A segment that the CTA mixes itself weighs more.
  const uint64_t kRunCost = mix ? 16u : 64u, kOddCost = 32u;
  info->mix = any_xform || any_read_first ? 2 : mix ? 1 : 0;      // the kernel's MIX
  const uint32_t nbp = (uint32_t)((B + 1) & ~1);

  info->n_stages = n_stages;
  info->n_barriers = ((uint32_t)n_stages + 1) * (mix ? 2u : 1u);   // the pre-pass has a barrier of its own per stage

  // Stages of squared inputs alone (no token shift, no gain): up to kSquaresShare inputs a CTA it squares what it reads itself, behind the stage's
  // barrier, and the stage needs neither the pre-pass nor its barrier.  Four blocks, pre-pass / so, us, at `inputs a CTA`: d 512, batch 1, 256, 100.1 / 94.3;
  // d 2048, batch 1, 512, 123.5 / 117.1; batch 2, 1024, 125.0 / 119.1; d 3072, batch 1, 1024, 151.7 / 145.6; d 4096, batch 1, 1792, 190.6 / 186.7; batch 8, 2048,
  // d 512 106.7 / 103.1, d 1024 115.0 / 112.0, d 1536 125.4 / 121.8; d 3072, batch 3, 3072, 164.3 / 161.9; d 4096, batch 2, 3584, 192.7 / 192.5; d 2048, batch 8,
  // 4096, 150.4 / 146.1; d 4096, batch 3, 5376, 205.0 / 208.6; batch 4, 7168, 211.6 / 213.0.  (What it takes depends on the rows and on the CTA's columns, too: 3584 is
  // even and 4096 a gain.)
  constexpr uint64_t kSquaresShare = 4200u;
  std::vector<char> squares(n_stages, 0);
  for (int s = 0; s < n_stages && any_xform && B <= 8; ++s) {
    uint64_t n = 0;
    bool all = true;
    for (int o = stage_ranges[s].first; o < stage_ranges[s].second; ++o) {
      const rwkvq_gemv_op& op = ops[o];
      n += (uint64_t)((op.W_desc.oc_pad + 255) / 256) * (uint64_t)(op.W_desc.ic_pad / 256);
      all = all && op.in.kind == RWKVQ_IN_RELU2 && !op.mu_image_dev && !op.in.xprev_out_fp16 && !op.in.scale_f32;
    }
    squares[s] = all && !read_first[s] && (n + (uint64_t)P - 1) / (uint64_t)P * 256u * (uint64_t)B <= kSquaresShare;
  }

  size_t deepest = 0;      // units of the CTA that has most, over all stages
  std::vector<std::vector<HostUnit>> cta_units(P);
  std::vector<std::vector<StepEvent>> cta_arrivals(P);      // arrival events, one per barrier
  bool too_many_ranges = false;
  auto make_arrival = [&](int c, int stage_idx_to_clear, int barrier) {
    StepEvent ev;
    std::memset(&ev, 0, sizeof(ev));
    ev.kind = EV_ARRIVE; ev.barrier = (uint32_t)barrier;
    if (barrier > 0 && barrier < n_stages && read_first[barrier - 1]) ev.flags |= EF_READ_FIRST;
    if (stage_idx_to_clear < n_stages) {
      uint64_t total = 0;
      for (int o = stage_ranges[stage_idx_to_clear].first; o < stage_ranges[stage_idx_to_clear].second; ++o)
        total += (uint64_t)B * ops[o].W_desc.oc;
      const uint64_t lo = total * (uint64_t)c / P, hi = total * (uint64_t)(c + 1) / P;
      uint64_t base = 0;
      int k = 0;
      for (int o = stage_ranges[stage_idx_to_clear].first; o < stage_ranges[stage_idx_to_clear].second; ++o) {
        const uint64_t n = (uint64_t)B * ops[o].W_desc.oc;
        const uint64_t a0 = std::max(lo, base), a1 = std::min(hi, base + n);
        if (a1 > a0) {
          if (k >= 3) { too_many_ranges = true; break; }
          ev.arr.zptr[k] = (uint64_t)(uintptr_t)ops[o].y_dev + (a0 - base) * 4;
          ev.arrd.zcount[k] = (uint32_t)(a1 - a0);
          ++k;
        }
        base += n;
      }
    }
    if (mix && barrier < n_stages && squares[barrier]) {
      ev.flags |= EF_SQUARES;
    } else if (mix && barrier < n_stages) {
      // this CTA's share of the pre-pass of stage `barrier`
      uint64_t G = 0;
      for (int o = stage_ranges[barrier].first; o < stage_ranges[barrier].second; ++o) G += (uint64_t)B * (ops[o].W_desc.ic_pad / 128);
      // counted from the first product that the share falls in: whoever looks for an item's product passes over those of the share only (192
      // products in one stage, batch 1: 303 us when every item was looked for from the stage's first product)
      const uint64_t lo = G * (uint64_t)c / P, hi = G * (uint64_t)(c + 1) / P;
      int first = stage_ranges[barrier].first;
      uint64_t base = 0;
      auto groups = [&](int o) { return (uint64_t)B * (ops[o].W_desc.ic_pad / 128); };
      while (lo < hi && lo >= base + groups(first)) base += groups(first++);
      int end = first;
      for (uint64_t b = base; lo < hi && b < hi; ++end) b += groups(end);
      ev.arr.grp_lo = (uint32_t)(lo - base); ev.arr.grp_hi = (uint32_t)(lo < hi ? hi - base : lo - base);
      ev.arrd.op_first = (uint16_t)first; ev.arrd.op_count = (uint16_t)(end - first);
    }
    cta_arrivals[c].push_back(ev);
  };
  for (int c = 0; c < P; ++c) make_arrival(c, 0, 0);   // barrier 0: the first stage's outputs are clear

  for (int s = 0; s < n_stages; ++s) {
    std::vector<HostUnit> units;
    for (int o = stage_ranges[s].first; o < stage_ranges[s].second; ++o) {
      const rwkvq_desc& d = ops[o].W_desc;
      const uint8_t* img = static_cast<const uint8_t*>(ops[o].W_image_dev);
      const uint8_t* payload = img + RWKVQ_HEADER_BYTES;
      const int KT = d.ic_pad / 256, MB = d.oc_pad / 128;
      const bool vq = d.method != RWKVQ_SQ;
      const uint32_t rb = vq ? rwkvq_vq_record_bytes(d.bits) : (uint32_t)RWKVQ_SQ_RECORD_BYTES;
      const uint32_t cb = 8u * rb;
      const uint8_t* aux = vq ? img + matrix_aux_offset(&d) : nullptr;
      for (int tr = 0; tr < (MB + 1) / 2; ++tr)
        for (int kt = 0; kt < KT; ++kt) {
          HostUnit h;
          std::memset(&h, 0, sizeof(h));
          h.u.flags = vq ? (UF_VQ | (d.bits == 8 ? UF_BITS8 : 0)) : 0;
          h.u.src0 = (uint64_t)(uintptr_t)(payload + (size_t)((2 * tr) * KT + kt) * cb);
          h.u.bytes0 = cb;
          if (2 * tr + 1 < MB) { h.u.src1 = (uint64_t)(uintptr_t)(payload + (size_t)((2 * tr + 1) * KT + kt) * cb); h.u.bytes1 = cb; }
          if (vq) {
            h.u.cb_src = (uint64_t)(uintptr_t)(aux + (size_t)(tr * KT + kt) * d.entries * 4);
            h.u.cb_bytes = (uint32_t)d.entries * 4u;
          }
          h.u.chunk_bytes = cb; h.u.rec_bytes = rb;
          h.u.row0 = (uint32_t)tr * 256u; h.u.oc = (uint32_t)d.oc; h.u.y = (uint64_t)(uintptr_t)ops[o].y_dev;
          h.u.stage = (uint32_t)s;
          h.op = o; h.tr = tr; h.kt = kt; h.stage = s;
          units.push_back(h);
        }
    }
    // The cost of a unit is what a record of its format costs the consumer warps, so that the CTAs that get a stage's VQ matrix do not finish
    // last.  A unit of the last 128 rows of an odd number takes the warps as long as a whole one (d 3712, batch 1, twelve layers: 403 us so, 572 when it
    // counted half; d 2944, batch 12, twenty layers: 793, 955).
    auto cost_of = [&](const HostUnit& h) -> uint64_t {
      // in twentieths of an SQ record, from stacks of one format and one stage (52 MB a layer, four layers, us: SQ / 64 / 256 entries at batch 1
      // 88, 121, 128; 8: 99, 135, 143; 16: 146, 177, 189), and the best of 24 to 34 for whole steps (14B-class, batch 16: 24 3416 us, 26 3420, 30 3427,
      // 34 3475; 7B-class, batch 1: 24 to 28 1153, 30 1162, 33 1185; batch 8: 24 1367, 27 1358, 33 1367)
      const uint64_t vq6 = B > 8 ? 26u : 27u, vq8 = B > 8 ? 26u : 28u;
      const uint64_t wgt = !(h.u.flags & UF_VQ) ? 20u : (h.u.flags & UF_BITS8) ? vq8 : vq6;
      return 16u * wgt * 64u;
    };
    // Units are dealt WHOLE (a consumer group spends about the same time on a piece of a unit as on a whole one, the warps
    // without a record idle), in runs of neighbouring units, by the smallest estimated time of the slowest CTA.  The estimate
    // of a run of units: their costs, kRunCost for every row of tiles it touches, and kOddCost.  Against rows cut into whole
    // numbers of runs alone: 14B-class stack B=16 4212 -> 4085 us (a stage of 64 rows x 16 tiles: seven units per CTA instead of
    // eight), 7B-class B=1 1277 -> 1254.
    const uint64_t whole = 16u * 20u * 64u;                      // an SQ unit
    std::vector<uint64_t> before(units.size() + 1, 0);
    for (size_t i = 0; i < units.size(); ++i) before[i + 1] = before[i] + cost_of(units[i]);
    auto new_row = [&](size_t i) { return units[i].op != units[i - 1].op || units[i].tr != units[i - 1].tr; };
    // most units from `first` on whose estimate stays within `limit`
    auto take = [&](size_t first, uint64_t limit) {
      size_t best = 0;
      uint64_t extra = kRunCost * whole / 64u;
      for (size_t n = 1; first + n <= units.size(); ++n) {
        const size_t i = first + n - 1;
        if (n > 1 && new_row(i)) extra += kRunCost * whole / 64u;
        const uint64_t sum = before[i + 1] - before[first] + extra;
        const uint64_t est = sum + (kGroups == 2 && (n & 1) ? cost_of(units[i]) * kOddCost / 64u : 0u);
        if (est <= limit) best = n;
        if (sum > limit) break;
      }
      return best;
    };
    typedef std::vector<std::pair<size_t, size_t>> Deal;         // (first unit, units) of consecutive CTAs
    auto pack = [&](uint64_t limit, Deal* deal) {
      if (deal) deal->clear();
      size_t i = 0;
      for (int c = 0; c < P && i < units.size(); ++c) {
        const size_t n = take(i, limit);
        if (n == 0) return false;
        if (deal) deal->push_back({i, n});
        i += n;
      }
      return i == units.size();
    };
    // runs that ignore the ends of rows
    uint64_t lo = 0, hi = before.back() + (uint64_t)(units.size() + 1) * (2u * whole);
    while (lo + whole / 64u < hi) {
      const uint64_t mid = lo + (hi - lo) / 2;
      if (pack(mid, nullptr)) hi = mid; else lo = mid;
    }
    Deal deal;
    pack(hi, &deal);
    // rows of tiles cut into a number of runs each, greedily the row with the largest cost per CTA first: taken where it is no worse (one
    // input segment and one flush per CTA; small stages leave some CTAs idle)
    {
      struct Row { size_t first, count; uint64_t cost; size_t k; };
      std::vector<Row> rows;
      for (size_t i = 0; i < units.size();) {
        size_t j = i + 1;
        while (j < units.size() && !new_row(j)) ++j;
        rows.push_back(Row{i, j - i, before[j] - before[i], 1});
        i = j;
      }
      if (rows.size() <= (size_t)P) {
        for (size_t spare = (size_t)P - rows.size(); spare > 0; --spare) {
          Row* best = nullptr;
          for (Row& r : rows)
            if (r.k < r.count && (!best || r.cost / r.k > best->cost / best->k)) best = &r;
          if (!best) break;
          ++best->k;
        }
        Deal by_row;
        bool fits = true;
        for (const Row& r : rows)
          for (size_t q = 0; q < r.k && fits; ++q) {
            const size_t a = r.first + r.count * q / r.k, b = r.first + r.count * (q + 1) / r.k;
            by_row.push_back({a, b - a});
            fits = take(a, hi + whole / 64u) >= b - a;
          }
        if (fits) deal.swap(by_row);
      }
    }
    size_t most = 0;
    for (const auto& d : deal) most = std::max(most, d.second);
    deepest += most;
    // start at a CTA that moves with the stage, so that idle CTAs are not always the same SMs
    size_t c = ((size_t)s * 37u) % (size_t)P;
    for (const auto& d : deal) {
      for (size_t i = d.first; i < d.first + d.second; ++i) cta_units[c].push_back(units[i]);
      c = (c + 1) % (size_t)P;
    }
    for (int c = 0; c < P; ++c) make_arrival(c, s + 1, s + 1);
  }
  // Units unpacked ahead of their inputs (consumer_role): they take about 1000 of the 2700 cycles of a group's first unit out of a stage's chain; a launch takes no
  // longer by itself (one layer of d 512: 17.5 us either way).  It gains where most groups have one unit a stage.  Eight layers where nothing else is said, without / with, us,
  // at `units of the CTA that has most, mean over the stages`: batch 1, d 512, 1, 104.3 / 96.3; d 1536, 1.25, 118.3 / 108.7; d 2048, 1.75, twelve layers, 203.0 / 176.5; d 2304,
  // 2.25, 148.4 / 144.5, but batch 4, d 2176, 2.25, twelve layers, 278.0 / 282.4; batch 1, d 2560, 2.75, 170.2 / 172.2; d 3072, 3.75, 194.7 / 192.5; d 4096, 6, 271.2 / 279.0;
  // batch 2, d 2048, 149.6 / 136.3; batch 8, d 2048, 200.9 / 189.2, d 4096, 324.7 / 325.7; four blocks of d 2048, batch 2, 114.8 / 108.7.  (One line for all batches
  // and for the whole plan: d 2304 and 3072 are on the wrong side of it.)  Above eight rows two warps a scheduler do not hide the trips to tensor memory (14B-class stack, batch
  // 16: 3330 / 3554).
  info->park = B <= 8 && deepest <= 2 * (size_t)n_stages;
  if (info->park) info->smem_bytes = std::max(info->smem_bytes, kSmemAlone);
  if (too_many_ranges) return RWKVQ_EUNSUPPORTED;   // a CTA's slice of a stage's outputs may touch at most three products

  // pre-pass outputs: one region, reused by every stage (a stage's pre-pass starts only after the
  // previous stage, and with it every copy out of the region, has finished everywhere)
  std::vector<uint64_t> mix_x_off(n_ops, 0), mix_sums_off(n_ops, 0);
  std::vector<StepMixOp> mixops(mix ? n_ops : 0);
  std::vector<StepMixX> mixx(mix ? n_ops : 0);
  uint64_t scratch_bytes = 0;
  if (mix) {
    for (int st_i = 0; st_i < n_stages; ++st_i) {
      uint64_t off = 0;
      for (int o = stage_ranges[st_i].first; o < stage_ranges[st_i].second; ++o) {
        const rwkvq_gemv_op& op = ops[o];
        mix_x_off[o] = off; off += round_up_sz((size_t)B * op.W_desc.ic_pad * 2, 256);
        mix_sums_off[o] = off; off += round_up_sz((size_t)(op.W_desc.ic_pad / 128) * 3 * nbp * 4, 256);
        StepMixOp& m = mixops[o];
        std::memset(&m, 0, sizeof(m));
        m.x = (uint64_t)(uintptr_t)op.x_fp16_dev;
        if (op.mu_image_dev) {
          const uint8_t* mi = static_cast<const uint8_t*>(op.mu_image_dev);
          m.xprev = (uint64_t)(uintptr_t)op.xprev_fp16_dev;
          m.mu = (uint64_t)(uintptr_t)(mi + RWKVQ_HEADER_BYTES);
          m.mu_aux = (uint64_t)(uintptr_t)(mi + vector_aux_offset(&op.mu_desc));
          m.mu_bits = (uint16_t)op.mu_desc.bits; m.mu_entries = (uint16_t)op.mu_desc.entries;
        }
        m.kind = (uint16_t)(op.in.kind | ((op.in.kind == RWKVQ_IN_F32 && (op.in.flags & RWKVQ_INF_RMSNORM)) ? 0x100 : 0) |
                            (op.in.xprev_out_fp16 ? 0x200 : 0));
        StepMixX& mx = mixx[o];
        std::memset(&mx, 0, sizeof(mx));
        mx.src = (uint64_t)(uintptr_t)op.in.src_f32;
        mx.k = (uint64_t)(uintptr_t)(op.in.kind == RWKVQ_IN_F32 ? op.in.gate_f32 : op.in.k_f32);
        mx.v = (uint64_t)(uintptr_t)op.in.v_f32;
        mx.state_a = (uint64_t)(uintptr_t)op.in.state_a; mx.state_b = (uint64_t)(uintptr_t)op.in.state_b;
        mx.state_p = (uint64_t)(uintptr_t)op.in.state_p;
        mx.u = (uint64_t)(uintptr_t)op.in.u_f32; mx.w = (uint64_t)(uintptr_t)op.in.w_f32;
        mx.xprev_out = (uint64_t)(uintptr_t)op.in.xprev_out_fp16;
        mx.scale = (uint64_t)(uintptr_t)op.in.scale_f32;
        m.dst_x = mix_x_off[o]; m.dst_sums = mix_sums_off[o];
        m.ic = (uint32_t)op.W_desc.ic; m.ic_pad = (uint32_t)op.W_desc.ic_pad;
        m.sums = op.W_desc.method == RWKVQ_SQ ? 1 : 0;
      }
      bool stage_norm = false;
      for (int o = stage_ranges[st_i].first; o < stage_ranges[st_i].second; ++o) stage_norm = stage_norm || (mixops[o].kind & 0x100);
      bool stage_plain = true;
      for (int o = stage_ranges[st_i].first; o < stage_ranges[st_i].second; ++o) stage_plain = stage_plain && mixops[o].kind == 0;
      for (int o = stage_ranges[st_i].first; o < stage_ranges[st_i].second; ++o) mixops[o].kind |= (stage_norm ? 0x400 : 0) | (stage_plain ? 0x800 : 0);
      scratch_bytes = std::max(scratch_bytes, off);
    }
  }
  std::vector<uint32_t> unit_off(P + 1, 0), event_off(P + 1, 0);
  std::vector<StepUnit> all_units;
  std::vector<StepEvent> all_events;
  for (int c = 0; c < P; ++c) {
    std::vector<HostUnit>& L = cta_units[c];
    unit_off[c] = (uint32_t)all_units.size();
    event_off[c] = (uint32_t)all_events.size();
    const size_t n = L.size();
    // a group accumulates along K in registers while its consecutive units stay on the same rows
    for (size_t i = 0; i < n; ++i) {
      const size_t j = i + (size_t)kGroups;
      const bool same_run = j < n && L[j].stage == L[i].stage && L[j].op == L[i].op && L[j].tr == L[i].tr;
      if (!same_run) L[i].u.flags |= UF_FLUSH;
    }
    all_events.push_back(cta_arrivals[c][0]);
    uint32_t seg_no = 0, heads[2] = {0, 0};
    bool squared[2] = {false, false};      // the segment last put into the buffer
    static_assert(XBufs<2, 1>::kCount == 2u, "segments take the buffers in turn");
    size_t i = 0;
    for (int s = 0; s < n_stages; ++s) {
      // segments: maximal runs of units of one product whose column span fits the buffer
      bool first_of_stage = true;
      while (i < n && L[i].stage == s) {
        const int op = L[i].op;
        const bool sums = ops[op].W_desc.method == RWKVQ_SQ;
        const bool has_mu = !mix && ops[op].mu_image_dev != nullptr;   // copied segments carry no mu row
        int kmin = L[i].kt, kmax = L[i].kt + 1;
        size_t j = i + 1, last = i;
        // A segment is a contiguous run of column tiles (a range that wraps from the end of one row
        // pair to the start of the next starts a new segment) that fits the buffer.
        while (j < n && L[j].op == op && L[j].stage == s) {
          if (L[j].kt < kmin || L[j].kt > kmax) break;
          const int nmax = std::max(kmax, L[j].kt + 1);
          if (xseg_bytes(B, (nmax - kmin) * 256, sums, has_mu) > xbuf_bytes) break;
          kmax = nmax; last = j; ++j;
        }
        const int ncols = (kmax - kmin) * 256;
        if (xseg_bytes(B, ncols, sums, has_mu) > xbuf_bytes) return RWKVQ_EUNSUPPORTED;
        StepEvent ev;
        std::memset(&ev, 0, sizeof(ev));
        const rwkvq_gemv_op& o = ops[op];
        ev.kind = EV_SEGMENT;
        ev.seg.x = (uint64_t)(uintptr_t)o.x_fp16_dev;
        ev.segd.ic = (uint32_t)o.W_desc.ic; ev.segd.col0 = (uint32_t)kmin * 256u; ev.segd.ncols = (uint32_t)ncols;
        const uint32_t xstride = (uint32_t)ncols * 2u + 32u;
        ev.xstride_sums = xstride | (sums ? 0x80000000u : 0u);
        ev.mu_off16 = (uint16_t)(xseg_mu_off(B, ncols, sums) / 16u);
        ev.barrier = (uint32_t)s + 1u;   // stage s reads its inputs after barrier s
        if (squares[s]) {
          ev.flags |= EF_SQUARES;
          ev.seg.x = (uint64_t)(uintptr_t)o.in.src_f32;
        } else if (mix) {
          if (squared[seg_no & 1u]) ev.flags |= EF_BEHIND_SQUARES;
          ev.seg.x = mix_x_off[op] + (uint64_t)kmin * 512u;
          ev.seg.xprev = mix_sums_off[op] + (uint64_t)(kmin * 2) * 3u * nbp * 4u;
          ev.segd.ic = (uint32_t)o.W_desc.ic_pad * 2u;
        } else if (has_mu) {
          const uint8_t* m = static_cast<const uint8_t*>(o.mu_image_dev);
          ev.seg.xprev = (uint64_t)(uintptr_t)o.xprev_fp16_dev;
          ev.seg.mu = (uint64_t)(uintptr_t)(m + RWKVQ_HEADER_BYTES);
          ev.seg.mu_aux = (uint64_t)(uintptr_t)(m + vector_aux_offset(&o.mu_desc));
          ev.segd.mu_bits = (uint16_t)o.mu_desc.bits; ev.segd.mu_entries = (uint16_t)o.mu_desc.entries;
        }
        for (size_t k = i; k <= last; ++k) {
          L[k].u.seg = seg_no;
          L[k].u.ev_index = (uint32_t)(all_events.size() - event_off[c]);
          L[k].u.xcol0 = (uint32_t)(L[k].kt - kmin) * 256u;
          L[k].u.xstride = xstride; L[k].u.gs_off = (uint32_t)B * xstride; L[k].u.nbp = nbp;
        }
        // One row that the CTA mixes itself, large stages: the head of a stage's first segment, the tiles of its groups' first units, is announced by itself
        // where at least as many follow, and the rest is mixed while those are at work.  Eight layers, batch 1, without / with, us: d 3072 202.9 / 198.9, d 3584
        // 246.6 / 239.7, d 4096 287.3 / 274.8.  (Copies of the pre-pass's results gain nothing by it, and what a unit's question for its barrier costs is
        // lost: batch 8, d 4096, 334 / 338; batch 16 445 / 455.  As a segment of its own the head cost more than it gave: batch 1, d 4096, 304.)
        bool in_order = first_of_stage && !mix && B == 1 && !info->park && kmax - kmin >= 2 * kHeadTiles && last + 1 - i >= 2 * (size_t)kHeadTiles;
        for (int k = 0; k < kHeadTiles && in_order; ++k) in_order = L[i + k].kt == kmin + k;
        if (in_order) {
          ev.flags |= EF_HEAD;
          const uint32_t phase = heads[seg_no & 1u]++ & 1u;
          for (int k = 0; k < kHeadTiles; ++k) {
            L[i + k].u.flags |= UF_HEAD | (phase ? UF_PHASE : 0u);
            L[i + kHeadTiles + k].u.flags |= UF_REST;      // every group waits for either
          }
        }
        first_of_stage = false;
        squared[seg_no & 1u] = squares[s] != 0;
        all_events.push_back(ev);
        ++seg_no;
        i = last + 1;
      }
      all_events.push_back(cta_arrivals[c][s + 1]);
    }
    // what each group has to pass between its consecutive segments, and after its last unit of a stage
    uint32_t prev_ev[2] = {0, 0};
    const StepEvent* evs = all_events.data() + event_off[c];
    const uint32_t n_ev = (uint32_t)(all_events.size() - event_off[c]);
    std::vector<uint32_t> arr_idx(n_stages, 0);
    for (uint32_t e = 0; e < n_ev; ++e)
      if (evs[e].kind == EV_ARRIVE && evs[e].barrier > 0u) arr_idx[evs[e].barrier - 1u] = e;
    auto mask_of = [&](uint32_t first, uint32_t last_excl) {
      uint32_t mask = 0;
      for (uint32_t e = first; e < last_excl; ++e)
        if (evs[e].kind == EV_ARRIVE && evs[e].barrier > 0u) mask |= 1u << (e - first);
      return mask;
    };
    for (size_t k = 0; k < n; ++k) {
      const int gidx = (int)(k % kGroups);
      const uint32_t target = L[k].u.ev_index;
      L[k].u.between_mask = (target > prev_ev[gidx] && target - prev_ev[gidx] - 1u <= 32u) ? mask_of(prev_ev[gidx] + 1u, target) : 0u;
      prev_ev[gidx] = target;
      const bool last_of_stage = k + kGroups >= n || L[k + kGroups].stage != L[k].stage;
      const uint32_t arr = arr_idx[L[k].stage];
      if (last_of_stage && arr > target && arr - target <= 32u) {
        L[k].u.after_count = arr - target;
        L[k].u.after_mask = mask_of(target + 1u, arr + 1u);
        prev_ev[gidx] = arr;
      }
    }
    for (size_t k = 0; k < n; ++k) all_units.push_back(L[k].u);
  }
  unit_off[P] = (uint32_t)all_units.size();
  event_off[P] = (uint32_t)all_events.size();

  info->n_units = (uint32_t)all_units.size();
  info->n_events = (uint32_t)all_events.size();
  size_t off = 256;
  info->off_unit_off = off; off += round_up_sz((size_t)(P + 1) * 4, 256);
  info->off_event_off = off; off += round_up_sz((size_t)(P + 1) * 4, 256);
  info->off_units = off; off += round_up_sz(std::max<size_t>(1, all_units.size()) * sizeof(StepUnit), 256);
  info->off_events = off; off += round_up_sz(all_events.size() * sizeof(StepEvent), 256);
  info->off_counter = off; off += round_up_sz((size_t)info->n_barriers * 4, 256);
  info->off_mixops = off; off += round_up_sz(mixops.size() * sizeof(StepMixOp), 256);
  info->off_mixx = off; off += round_up_sz(mixx.size() * sizeof(StepMixX), 256);
  info->off_scratch = off; off += round_up_sz((size_t)scratch_bytes, 256);
  info->total_bytes = off;
  if (out) {
    out->assign(off, 0);
    memcpy(out->data() + info->off_unit_off, unit_off.data(), (size_t)(P + 1) * 4);
    memcpy(out->data() + info->off_event_off, event_off.data(), (size_t)(P + 1) * 4);
    if (!all_units.empty()) memcpy(out->data() + info->off_units, all_units.data(), all_units.size() * sizeof(StepUnit));
    memcpy(out->data() + info->off_events, all_events.data(), all_events.size() * sizeof(StepEvent));
    if (!mixops.empty()) memcpy(out->data() + info->off_mixops, mixops.data(), mixops.size() * sizeof(StepMixOp));
    if (!mixx.empty()) memcpy(out->data() + info->off_mixx, mixx.data(), mixx.size() * sizeof(StepMixX));
  }
  return RWKVQ_OK;
}

}  // namespace rwkvq

using namespace rwkvq;

extern "C" {

size_t rwkvq_step_plan_bytes(const rwkvq_gemv_op* ops, int n_ops, int B) {
  PlanInfo info;
  if (build_plan(ops, n_ops, B, sm_count(), nullptr, &info) != RWKVQ_OK) return 0;
  return info.total_bytes;
}

rwkvq_status rwkvq_step_plan(const rwkvq_gemv_op* ops, int n_ops, int B, void* plan_dev, size_t plan_bytes, void* stream) {
  if (!plan_dev) return RWKVQ_EINVAL;
  if (!aligned16(plan_dev)) return RWKVQ_EALIGN;
  PlanInfo info;
  std::vector<uint8_t> image;
  rwkvq_status st = build_plan(ops, n_ops, B, sm_count(), &image, &info);
  if (st != RWKVQ_OK) return st;
  if (plan_bytes < info.total_bytes) return RWKVQ_ENOMEM;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaMemcpyAsync(plan_dev, image.data(), image.size(), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);   // `image` is a pageable temporary
  if (e != cudaSuccess) return cuda_status(e);
  info.runs = 0;
  info.captured = false;
  info.abort_epoch = abort_epoch();   // the image just copied holds zeroed counters
  for (int i = 0; i < n_ops; ++i) {
    if (i == 0 || ops[i].stage != ops[i - 1].stage) { info.y_lo.push_back(~0ull); info.y_hi.push_back(0ull); }
    const uint64_t lo = (uint64_t)(uintptr_t)ops[i].y_dev, hi = lo + (uint64_t)B * (uint64_t)ops[i].W_desc.oc * 4u;
    info.y_lo.back() = std::min(info.y_lo.back(), lo);
    info.y_hi.back() = std::max(info.y_hi.back(), hi);
  }
  std::lock_guard<std::mutex> lock(g_plan_mutex);
  g_plans[plan_dev] = info;
  return RWKVQ_OK;
}

}  // extern "C"

namespace {
// Inputs that arrive while the step runs (see StepArgs::in_flag).
struct HostRun {
  const unsigned* in_flag = nullptr;
  unsigned in_base = 0, in_shift = 0;
  uint64_t in_lo = 0, in_hi = 0;
};

// Every arrival counter that is short of `target` (a run that gave up) is raised to it, so that
// nothing ordered behind a counter waits for ever and the next run starts from a consistent state.
__global__ void step_finish_kernel(unsigned* counter, int n, unsigned target) {
  const int k = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (k < n && (int)(counter[k] - target) < 0) counter[k] = target;
}

unsigned* counters_of(const void* plan_dev, const PlanInfo& info) {
  return reinterpret_cast<unsigned*>(static_cast<uint8_t*>(const_cast<void*>(plan_dev)) + info.off_counter);
}
unsigned target_of(const PlanInfo& info) { return info.runs * (unsigned)info.P; }

bool is_capturing(cudaStream_t s) {
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &status) != cudaSuccess) { cudaGetLastError(); return false; }      // the default stream beside another thread's capture
  return status == cudaStreamCaptureStatusActive;
}

// A run that was counted but will never arrive: have the next one clear the counters.
void forget_run(const void* plan_dev) {
  std::lock_guard<std::mutex> lock(g_plan_mutex);
  auto it = g_plans.find(plan_dev);
  if (it != g_plans.end()) it->second.abort_epoch = abort_epoch() - 1u;
}

// Counts one more run of the plan and, where it is due, clears the arrival counters on the caller's stream.  Whatever waits for the counters of
// this run on another stream is ordered behind this call.
rwkvq_status begin_run(const void* plan_dev, size_t plan_bytes, cudaStream_t s, PlanInfo* info) {
  if (!plan_dev) return RWKVQ_EINVAL;
  bool clear_counters = false;
  {
    std::lock_guard<std::mutex> lock(g_plan_mutex);
    auto it = g_plans.find(plan_dev);
    if (it == g_plans.end()) return RWKVQ_EINVAL;   // not a plan written by rwkvq_step_plan in this process
    if (plan_bytes < it->second.total_bytes) return RWKVQ_ENOMEM;
    // The arrival counters only ever grow: run r opens a barrier at r * CTAs arrivals, so a launch
    // needs no clearing pass.  A run that gave up leaves them short; start over after one.  A captured run is launched any number of times
    // with the target it was captured with: it clears them itself, and so does every other run of the plan from then on, which cannot know
    // what the graph's launches left.
    const unsigned epoch = abort_epoch();
    it->second.captured = it->second.captured || is_capturing(s);
    if (it->second.abort_epoch != epoch || it->second.captured) { it->second.abort_epoch = epoch; it->second.runs = 0; clear_counters = true; }
    it->second.runs += 1;
    *info = it->second;
  }
  if (clear_counters) {
    const cudaError_t e = cudaMemsetAsync(counters_of(plan_dev, *info), 0, round_up_sz((size_t)info->n_barriers * 4, 256), s);
    if (e != cudaSuccess) { forget_run(plan_dev); return cuda_status(e); }
  }
  return RWKVQ_OK;
}

rwkvq_status launch_run(const void* plan_dev, const PlanInfo& info, cudaStream_t s, const HostRun* hr) {
  const uint8_t* p = static_cast<const uint8_t*>(plan_dev);
  StepArgs a;
  a.units = reinterpret_cast<const StepUnit*>(p + info.off_units);
  a.events = reinterpret_cast<const StepEvent*>(p + info.off_events);
  a.unit_off = reinterpret_cast<const uint32_t*>(p + info.off_unit_off);
  a.event_off = reinterpret_cast<const uint32_t*>(p + info.off_event_off);
  a.counter = counters_of(plan_dev, info);
  a.status = device_status_ptr();
  if (!a.status) { forget_run(plan_dev); return RWKVQ_ECUDA; }
  a.B = info.B; a.n_slots = info.n_slots; a.n_stages = info.n_stages;
  a.mix = info.mix; a.mixops = reinterpret_cast<const StepMixOp*>(p + info.off_mixops);
  a.mixx = reinterpret_cast<const StepMixX*>(p + info.off_mixx);
  a.scratch = const_cast<uint8_t*>(p) + info.off_scratch;
  a.slot_bytes = info.slot_bytes; a.replica_bytes = info.replica_bytes;
  a.target = target_of(info);
  a.poll_limit = info.poll_limit; a.wait_skew = info.wait_skew;
  a.in_flag = nullptr; a.in_base = 0; a.in_shift = 0; a.in_lo = 0; a.in_hi = 0;
  if (hr) { a.in_flag = hr->in_flag; a.in_base = hr->in_base; a.in_shift = hr->in_shift; a.in_lo = hr->in_lo; a.in_hi = hr->in_hi; }
  static const void* const kernels[3][3] = {{(const void*)step_kernel<1, 0, false>, (const void*)step_kernel<1, 1, false>, (const void*)step_kernel<1, 2, false>},
                                            {(const void*)step_kernel<2, 0, false>, (const void*)step_kernel<2, 1, false>, (const void*)step_kernel<2, 2, false>},
                                            {(const void*)step_kernel<1, 0, true>, (const void*)step_kernel<1, 1, true>, (const void*)step_kernel<1, 2, true>}};
  static const void* const one_row[2] = {(const void*)step_kernel<1, 0, false, true>, (const void*)step_kernel<1, 0, true, true>};
  const void* fn = info.B == 1 && info.mix == 0 ? one_row[info.park] : kernels[info.park ? 2 : info.NB - 1][info.mix];
  void* params[] = {&a};
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)info.smem_bytes);
  // Cooperative launch: all CTAs must be resident at once because they meet at the stage barrier.
  if (e == cudaSuccess) e = cudaLaunchCooperativeKernel(fn, dim3(info.P), dim3(threads_of(info.NB)), params, info.smem_bytes, s);
  if (e != cudaSuccess) { forget_run(plan_dev); return cuda_status(e); }
  if (hr) {
    step_finish_kernel<<<(info.n_barriers + 255u) / 256u, 256, 0, s>>>(a.counter, (int)info.n_barriers, a.target);
    e = cudaGetLastError();
  }
  return cuda_status(e);
}
}  // namespace

extern "C" {

rwkvq_status rwkvq_step_run(const void* plan_dev, size_t plan_bytes, void* stream) {
  PlanInfo info;
  const rwkvq_status st = begin_run(plan_dev, plan_bytes, static_cast<cudaStream_t>(stream), &info);
  return st != RWKVQ_OK ? st : launch_run(plan_dev, info, static_cast<cudaStream_t>(stream), nullptr);
}

rwkvq_status rwkvq_step_plan_release(const void* plan_dev) {
  if (!plan_dev) return RWKVQ_EINVAL;
  std::lock_guard<std::mutex> lock(g_plan_mutex);
  return g_plans.erase(plan_dev) ? RWKVQ_OK : RWKVQ_EINVAL;
}

rwkvq_status rwkvq_step_set_wait(const void* plan_dev, uint32_t poll_limit, uint32_t wait_skew) {
  if (!plan_dev) return RWKVQ_EINVAL;
  std::lock_guard<std::mutex> lock(g_plan_mutex);
  auto it = g_plans.find(plan_dev);
  if (it == g_plans.end()) return RWKVQ_EINVAL;
  it->second.poll_limit = poll_limit ? poll_limit : kDefaultPollLimit;
  it->second.wait_skew = wait_skew;
  return RWKVQ_OK;
}

rwkvq_status rwkvq_step_reciprocal(const float* y_dev, float* out_dev, size_t n, void* stream) {
  if (!y_dev || !out_dev || n == 0) return RWKVQ_EINVAL;
  if (n > (size_t)1 << 31) return RWKVQ_EUNSUPPORTED;
  reciprocal_kernel<<<(unsigned)((n + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(y_dev, out_dev, n);
  return cuda_status(cudaGetLastError());
}

rwkvq_status rwkvq_step_plan_cover(const rwkvq_gemv_op* ops, int n_ops, int B, int n_ctas, uint32_t* counts_host,
                                   size_t n_counts, uint32_t* cta_items_host) {
  if (!counts_host || n_ctas <= 0) return RWKVQ_EINVAL;
  PlanInfo info;
  std::vector<uint8_t> image;
  rwkvq_status st = build_plan(ops, n_ops, B, n_ctas, &image, &info);
  if (st != RWKVQ_OK) return st;
  // cell of (product, 16-row slice, column tile) in counts_host
  std::vector<size_t> base(n_ops + 1, 0);
  for (int i = 0; i < n_ops; ++i) base[i + 1] = base[i] + (size_t)(ops[i].W_desc.oc / 16) * (size_t)(ops[i].W_desc.ic_pad / 256);
  if (n_counts < base[n_ops]) return RWKVQ_ENOMEM;
  std::unordered_map<uint64_t, int> op_of_y;
  for (int i = 0; i < n_ops; ++i) op_of_y[(uint64_t)(uintptr_t)ops[i].y_dev] = i;
  const uint32_t* unit_off = reinterpret_cast<const uint32_t*>(image.data() + info.off_unit_off);
  const StepUnit* units = reinterpret_cast<const StepUnit*>(image.data() + info.off_units);
  for (int c = 0; c < n_ctas; ++c) {
    uint32_t items = 0;
    for (uint32_t k = unit_off[c]; k < unit_off[c + 1]; ++k) {
      const StepUnit& u = units[k];
      auto it = op_of_y.find(u.y);
      if (it == op_of_y.end()) return RWKVQ_EINVAL;     // the walk needs distinct output buffers
      const int o = it->second;
      const rwkvq_desc& d = ops[o].W_desc;
      const uint32_t KT = (uint32_t)d.ic_pad / 256u, slices = (uint32_t)d.oc / 16u;
      const uint8_t* payload = static_cast<const uint8_t*>(ops[o].W_image_dev) + RWKVQ_HEADER_BYTES;
      // the unit's chunks: warp w of the group takes record w of chunk A (and of chunk B, 128 rows below)
      const uint64_t src[2] = {u.src0, u.src1};
      const uint32_t bytes[2] = {u.bytes0, u.bytes1};
      for (int h = 0; h < 2; ++h) {
        if (!bytes[h]) continue;
        if (bytes[h] != 8u * u.rec_bytes) return RWKVQ_EINVAL;
        const uint64_t rel = src[h] - (uint64_t)(uintptr_t)payload;
        if (rel % u.chunk_bytes) return RWKVQ_EINVAL;
        const uint64_t chunk = rel / u.chunk_bytes;       // mb * KT + kt
        const uint32_t mb = (uint32_t)(chunk / KT), kt = (uint32_t)(chunk % KT);
        if (mb * 128u != u.row0 + 128u * (uint32_t)h) return RWKVQ_EINVAL;
        for (uint32_t w = 0; w < 8u; ++w) {
          const uint32_t slice = mb * 8u + w;
          if (slice >= slices) continue;                  // padding rows of the last chunk
          counts_host[base[o] + (size_t)slice * KT + kt] += 1u;
          ++items;
        }
      }
    }
    if (cta_items_host) cta_items_host[c] = items;
  }
  return RWKVQ_OK;
}

rwkvq_status rwkvq_step_plan_forms(const rwkvq_gemv_op* ops, int n_ops, int B, int n_ctas, rwkvq_step_forms* forms_host) {
  if (!forms_host || n_ctas <= 0) return RWKVQ_EINVAL;
  PlanInfo info;
  std::vector<uint8_t> image;
  const rwkvq_status st = build_plan(ops, n_ops, B, n_ctas, &image, &info);
  if (st != RWKVQ_OK) return st;
  rwkvq_step_forms f;
  std::memset(&f, 0, sizeof(f));
  f.pre_pass = info.mix; f.unpacked_ahead = info.park ? 1 : 0; f.smem_bytes = info.smem_bytes;
  const uint32_t* event_off = reinterpret_cast<const uint32_t*>(image.data() + info.off_event_off);
  const StepEvent* events = reinterpret_cast<const StepEvent*>(image.data() + info.off_events);
  for (int c = 0; c < n_ctas; ++c) {
    uint32_t heads = 0;
    for (uint32_t e = event_off[c]; e < event_off[c + 1]; ++e) {
      if (events[e].kind != EV_SEGMENT) continue;
      ++f.segments;
      heads += (events[e].flags & EF_HEAD) != 0;
      f.squared += (events[e].flags & EF_SQUARES) != 0;
      f.behind_squared += (events[e].flags & EF_BEHIND_SQUARES) != 0;
    }
    f.announced_heads += heads;
    f.most_heads = std::max(f.most_heads, heads);
  }
  *forms_host = f;
  return RWKVQ_OK;
}

}  // extern "C"

namespace {
// Streams, events and the arrival word of host-buffer runs, one set per context (context_id; what cudaDeviceReset ended
// leaves an empty entry behind).  The stream memory operations come from the driver through the runtime's entry-point query (no link to the driver library).
typedef CUresult (*StreamValueFn)(CUstream, CUdeviceptr, cuuint32_t, unsigned int);
struct HostPipe {
  bool tried = false, ok = false;
  cudaStream_t h2d = nullptr, d2h = nullptr;
  cudaEvent_t start = nullptr, h2d_done = nullptr, d2h_done = nullptr;
  unsigned* flag = nullptr;      // device word: chunks arrived so far, over all runs
  unsigned chunks = 0;           // the host's copy of its final value after the last run enqueued
  StreamValueFn wait_value = nullptr, write_value = nullptr;
  bool used = false;             // the last run came on the stream of number `user`
  unsigned long long user = 0;
};
std::mutex g_pipe_mutex;
std::unordered_map<unsigned long long, HostPipe> g_pipes;
// Activations arrive in pieces of 256 KB, then twice as much each time up to 4 MB: the step begins behind the first piece (5 us instead of 80)
// and most of the bytes go in copies long enough for the link's rate.  Outputs leave in groups of whole stages of at least a quarter
// of what is still to come, 2 MB at most, so that little is left to copy when the step ends.  73 MB both ways, 32 layers: 1606 us, 1646 with
// pieces of 4 MB and groups of 2 MB, 2795 in the plain order.
constexpr unsigned kChunkShift = 18, kMaxChunks = 16;
constexpr size_t kOutGroupBytes = (size_t)2 << 20, kMinOutGroupBytes = (size_t)128 << 10;
// Steps that copy less run the plain order: overlapped, 0.4 MB took 93 us against 92.  From there on it gains: 0.57 MB 147 against 150,
// 1.1 MB 149 and 164, 2.3 MB 176 and 204, 4.6 MB 220 and 288.
constexpr size_t kOverlapMinBytes = (size_t)512 << 10;

HostPipe* host_pipe() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
  unsigned long long id = context_id();
  if (id == 0 && cudaFree(nullptr) == cudaSuccess) id = context_id();      // a thread's first call
  HostPipe& hp = g_pipes[id != 0 ? id : ~(unsigned long long)dev];
  if (hp.tried) return hp.ok ? &hp : nullptr;
  hp.tried = true;
  // allocations are no concern of another thread's capture
  struct Relaxed {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    Relaxed() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~Relaxed() { cudaThreadExchangeStreamCaptureMode(&mode); }
  } relaxed;
  cudaDriverEntryPointQueryResult q1, q2;
  void *f1 = nullptr, *f2 = nullptr;
  if (cudaGetDriverEntryPoint("cuStreamWaitValue32", &f1, cudaEnableDefault, &q1) != cudaSuccess || q1 != cudaDriverEntryPointSuccess || !f1) return nullptr;
  if (cudaGetDriverEntryPoint("cuStreamWriteValue32", &f2, cudaEnableDefault, &q2) != cudaSuccess || q2 != cudaDriverEntryPointSuccess || !f2) return nullptr;
  hp.wait_value = reinterpret_cast<StreamValueFn>(f1);
  hp.write_value = reinterpret_cast<StreamValueFn>(f2);
  if (cudaStreamCreateWithFlags(&hp.h2d, cudaStreamNonBlocking) != cudaSuccess) return nullptr;
  if (cudaStreamCreateWithFlags(&hp.d2h, cudaStreamNonBlocking) != cudaSuccess) return nullptr;
  if (cudaEventCreateWithFlags(&hp.start, cudaEventDisableTiming) != cudaSuccess) return nullptr;
  if (cudaEventCreateWithFlags(&hp.h2d_done, cudaEventDisableTiming) != cudaSuccess) return nullptr;
  if (cudaEventCreateWithFlags(&hp.d2h_done, cudaEventDisableTiming) != cudaSuccess) return nullptr;
  if (cudaMalloc(&hp.flag, 256) != cudaSuccess) return nullptr;
  if (cudaMemset(hp.flag, 0, 256) != cudaSuccess) return nullptr;
  // one write and one wait that is already satisfied: if the driver refuses either, stay on the plain path
  if (hp.write_value(hp.h2d, (CUdeviceptr)(uintptr_t)hp.flag, 0u, 0u) != CUDA_SUCCESS) return nullptr;
  if (hp.wait_value(hp.h2d, (CUdeviceptr)(uintptr_t)hp.flag, 0u, CU_STREAM_WAIT_VALUE_GEQ) != CUDA_SUCCESS) return nullptr;
  if (cudaStreamSynchronize(hp.h2d) != cudaSuccess) return nullptr;
  hp.ok = true;
  return &hp;
}

// Whether a run on stream s may take the copy streams: its copies must not lie behind those of another stream's run, which wait for that stream's
// work, while its step already occupies every SM and waits for them.  Behind a run on the same stream they do not wait longer than the step.
bool pipe_free(HostPipe& hp, cudaStream_t s) {
  unsigned long long id = 0;
  const bool known = cudaStreamGetId(s, &id) == cudaSuccess;
  if (hp.used && !(known && id == hp.user)) {
    const bool idle = cudaStreamQuery(hp.h2d) == cudaSuccess && cudaStreamQuery(hp.d2h) == cudaSuccess;
    if (!idle) { cudaGetLastError(); return false; }
  }
  hp.used = true;
  hp.user = known ? id : ~0ull;
  return true;
}

rwkvq_status run_host_plain(const void* plan_dev, size_t plan_bytes, const void* act_host, void* act_dev, size_t act_bytes,
                            const void* y_dev, void* y_host, size_t y_bytes, void* stream) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (act_bytes) {
    cudaError_t e = cudaMemcpyAsync(act_dev, act_host, act_bytes, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return cuda_status(e);
  }
  rwkvq_status st = rwkvq_step_run(plan_dev, plan_bytes, stream);
  if (st != RWKVQ_OK) return st;
  if (y_bytes) {
    cudaError_t e = cudaMemcpyAsync(y_host, y_dev, y_bytes, cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) return cuda_status(e);
  }
  return RWKVQ_OK;
}
}  // namespace

extern "C" {

rwkvq_status rwkvq_step_run_host(const void* plan_dev, size_t plan_bytes, const void* act_host, void* act_dev,
                                 size_t act_bytes, const void* y_dev, void* y_host, size_t y_bytes, void* stream) {
  if ((act_bytes && (!act_host || !act_dev)) || (y_bytes && (!y_dev || !y_host))) return RWKVQ_EINVAL;
  // Small steps: the copies are short and the plain order (copy in, run, copy out on one stream) is best.
  const char* ov = std::getenv("RWKVQ_HOST_OVERLAP");      // "0": always the plain order
  if ((ov && ov[0] == '0') || act_bytes + y_bytes < kOverlapMinBytes)
    return run_host_plain(plan_dev, plan_bytes, act_host, act_dev, act_bytes, y_dev, y_host, y_bytes, stream);
  // A captured call stays on its stream: a graph would keep this call's numbers for the words that the overlapped order waits for.
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (is_capturing(s)) return run_host_plain(plan_dev, plan_bytes, act_host, act_dev, act_bytes, y_dev, y_host, y_bytes, stream);
  std::lock_guard<std::mutex> lock(g_pipe_mutex);
  HostPipe* hp = host_pipe();
  if (!hp || !pipe_free(*hp, s)) return run_host_plain(plan_dev, plan_bytes, act_host, act_dev, act_bytes, y_dev, y_host, y_bytes, stream);
  PlanInfo info;
  rwkvq_status st = begin_run(plan_dev, plan_bytes, s, &info);
  if (st != RWKVQ_OK) return st;
  // Both side streams start behind everything already enqueued on the caller's stream, the clearing of the counters among it: the output
  // copies wait for this run's arrivals, which the counters of earlier runs would seem to be.
  cudaError_t e = cudaEventRecord(hp->start, s);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(hp->h2d, hp->start, 0);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(hp->d2h, hp->start, 0);
  if (e != cudaSuccess) { forget_run(plan_dev); return cuda_status(e); }
  // Activations: chunk by chunk on the copy stream; the word counts the chunks that have arrived.
  // They are enqueued BEFORE the launch: streams share a limited number of hardware queues, and a copy
  // enqueued behind the running step in the same queue would start only when the step, which waits for it, ends.
  HostRun hr;
  const unsigned n_in = (unsigned)((act_bytes + ((size_t)1 << kChunkShift) - 1) >> kChunkShift);
  if (n_in) {
    hr.in_flag = hp->flag; hr.in_base = hp->chunks; hr.in_shift = kChunkShift;
    hr.in_lo = (uint64_t)(uintptr_t)act_dev; hr.in_hi = hr.in_lo + act_bytes;
    for (unsigned i = 0; i < n_in;) {
      const unsigned upto = std::min(n_in, i + std::min(kMaxChunks, std::max(1u, i)));
      const size_t off = (size_t)i << kChunkShift, len = std::min((size_t)upto << kChunkShift, act_bytes) - off;
      e = cudaMemcpyAsync(static_cast<uint8_t*>(act_dev) + off, static_cast<const uint8_t*>(act_host) + off, len, cudaMemcpyHostToDevice, hp->h2d);
      if (e != cudaSuccess) break;
      if (hp->write_value(hp->h2d, (CUdeviceptr)(uintptr_t)hp->flag, hp->chunks + upto, 0u) != CUDA_SUCCESS) { e = cudaErrorUnknown; break; }
      i = upto;
    }
    // Whatever happened, the word reaches its final value, so that no stager waits for a chunk in vain.
    if (e != cudaSuccess) hp->write_value(hp->h2d, (CUdeviceptr)(uintptr_t)hp->flag, hp->chunks + n_in, 0u);
    hp->chunks += n_in;
    if (e != cudaSuccess) { forget_run(plan_dev); cudaStreamSynchronize(hp->h2d); return cuda_status(e); }
  }
  // The step itself, on the caller's stream, at once: its stagers wait for the chunks they read.
  st = launch_run(plan_dev, info, s, &hr);
  if (st != RWKVQ_OK) { cudaStreamSynchronize(hp->h2d); return st; }
  // Outputs: stage by stage behind the stage barriers (the arrival counters of the plan), in groups of
  // whole stages, as long as the stages' outputs lie one behind the other in [y_dev, y_dev + y_bytes).
  if (y_bytes) {
    unsigned* counter = counters_of(plan_dev, info);
    const unsigned target = target_of(info);
    const uint64_t y0 = (uint64_t)(uintptr_t)y_dev, y1 = y0 + y_bytes;
    bool ordered = !info.y_lo.empty();
    uint64_t prev = y0;
    for (size_t k = 0; k < info.y_lo.size() && ordered; ++k) {
      if (info.y_lo[k] < prev || info.y_hi[k] > y1 || info.y_hi[k] < info.y_lo[k]) ordered = false;
      prev = info.y_hi[k];
    }
    const int n_st = info.n_stages;
    size_t done = 0;                               // bytes of the output buffer already handed to copies
    for (int k = 0; k < n_st && e == cudaSuccess; ++k) {
      const bool last = k + 1 == n_st;
      const size_t upto = last || !ordered ? (last ? y_bytes : done) : (size_t)(info.y_hi[k] - y0);
      if (!last && upto - done < std::min(kOutGroupBytes, std::max(kMinOutGroupBytes, (y_bytes - done) / 4))) continue;
      if (upto == done) continue;
      // barrier k + 1 closes stage k: every CTA has arrived behind its reductions into these outputs
      if (hp->wait_value(hp->d2h, (CUdeviceptr)(uintptr_t)(counter + (k + 1)), target, CU_STREAM_WAIT_VALUE_GEQ) != CUDA_SUCCESS) { e = cudaErrorUnknown; break; }
      e = cudaMemcpyAsync(static_cast<uint8_t*>(y_host) + done, static_cast<const uint8_t*>(y_dev) + done, upto - done, cudaMemcpyDeviceToHost, hp->d2h);
      done = upto;
    }
  }
  // The caller's stream ends behind both side streams: synchronizing it covers the whole step.
  if (e == cudaSuccess) e = cudaEventRecord(hp->h2d_done, hp->h2d);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(s, hp->h2d_done, 0);
  if (e == cudaSuccess) e = cudaEventRecord(hp->d2h_done, hp->d2h);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(s, hp->d2h_done, 0);
  return cuda_status(e);
}

}  // extern "C"
