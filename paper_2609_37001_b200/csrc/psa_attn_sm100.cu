// psa_attn_fwd for sm_100a: stripe-masked flash attention forward.
//
// A work item is up to two query slabs (<= 128 rows each) of one query block (PSABlock); both slabs share the block's key
// list (GetKVBlocks, Algorithm 2), which the load warp enumerates in ascending block id (edge blocks last) straight from
// the six stripe parameters (Algorithm 1) -- no mask or index list is read from memory.
// How items reach CTAs depends on how many there are (Mode; the choice is in the host file): with more items than SMs, one
// persistent CTA per SM draws them from a global ticket, stored heaviest first (by the number of attended key blocks) and
// head-major by a planning kernel; when all of them run at once, CTA i takes item i and nothing is planned; when they are
// few or some are long, a cluster of 2, 4 or 8 CTAs shares each item.
// A single-slab item runs in split-KV mode: both softmax warpgroups work on that one slab, on
// the even and the odd key slabs, and their partial results are merged in the epilogue.
//
// Roles (384 threads = 3 warpgroups):
//   warp  0    tcgen05.mma issue: S_i = Q_i K^T (SS form), O_i += P_i V (P read from TMEM).  Its
//              own instruction stream is on the critical path, so it probes two barriers per
//              shared-memory round trip and divides nothing inside the loop
//   warp  1    scheduler + TMA loads: Q slabs once per item, K and V slabs through a 5-slot ring
//              (V_j travels with K_{j+1} under one barrier)
//   warps 2-3  idle; they only exist so that the first warpgroup can hand its registers
//              to the softmax warpgroups (setmaxnreg)
//   warps 4-7  softmax / correction / epilogue of tile 0 = (S0, O0)   (TMEM lanes 0..127)
//   warps 8-11 the same for tile 1 = (S1, O1)
// TMEM (512 columns): S0 | S1 | O0 | O1, 128 fp32 columns each; the bf16 probabilities
// P_i overwrite the first columns of S_i.  A key slab has 128 keys, or 112/96/64 for the last
// slab of a block whose token count is not a multiple of 128.
// Every meeting point inside the kernel's loops is an mbarrier wait with a time limit (2 s of
// %globaltimer): producer / consumer hand-offs, the merge of a split-KV item, and the gathering
// of a staged output slab before its TMA store.  On expiry the waiter sets a CTA-wide abort
// flag; every other waiter sees the flag at its next poll and returns, all roles leave their
// loops, the load warp waits (bounded) for its TMA loads in flight, the MMA warp waits (bounded)
// for its MMAs in flight, all threads meet at the one __syncthreads of the teardown, TMEM is
// freed and the status word reports the timeout.  Not bounded by the kernel: the wait for the kernel
// before it in the stream (griddepcontrol.wait); the two cluster barriers of shared items, which every
// thread reaches, since all loops before them are left in bounded time; and the TMEM allocation
// at start-up, which blocks while another resident CTA holds tensor memory -- this kernel takes a
// whole SM (226 KB of shared memory, 512 TMEM columns), so a caller must not run other
// TMEM-using kernels on the same device concurrently with it.
// Build-time knob: PSA_EMU_PAIRS (share of exponentials computed by a polynomial on the FMA
// pipe, default 0).
#include <cuda.h>
#include <cuda_bf16.h>

#include "psa_common.cuh"

namespace psa {

constexpr int kThreads = 384;                       // 3 warpgroups; register budgets are re-split below
constexpr int kWarpMma = 0, kWarpLoad = 1, kUtilGroup = 0, kFirstSoftmaxWarp = 4;   // warp roles
constexpr int kNumSlots = 5;                       // K/V ring slots of one 128 x 128 bf16 slab
constexpr uint32_t kSlabBytes = 128 * 128 * 2;     // 32 KB
constexpr uint32_t kHalfBytes = kSlabBytes / 2;    // one 64-column swizzled half
// Register budgets after the re-split (setmaxnreg).  The CTA's pool is what it was launched with
// (kRegsAtLaunch per thread: the compiler's figure under the launch bound of 384 threads);
// setmaxnreg.inc blocks until the pool has room, so a split that does not fit would never start.
constexpr int kRegsAtLaunch = 168, kRegsUtil = 72, kRegsSoftmax = 216;
static_assert(128 * kRegsUtil + 256 * kRegsSoftmax <= kThreads * kRegsAtLaunch, "register re-split exceeds the CTA's pool");
constexpr int kMetaRing = 8;
constexpr float kRescaleThreshold = 8.0f;          // log2 units; lazy rescale of O
constexpr unsigned long long kTimeoutNs = 2000000000ull;

// shared memory map (offsets from a 1024-byte aligned base)
constexpr uint32_t kOffQ = 0;                                   // 2 slabs
constexpr uint32_t kOffRing = 2 * kSlabBytes;                   // kNumSlots slabs
constexpr uint32_t kOffBar = kOffRing + kNumSlots * kSlabBytes; // mbarriers
// One load barrier per ring slot: a barrier is armed again only after as many further tiles as
// there are slots have been issued, i.e. after the tiles of its previous phase were consumed
// (tiles that travel alone -- the first K and the last V of an item -- each take a barrier).
constexpr int kNumPairBars = kNumSlots;
constexpr int kBarQFull = 0, kBarQEmpty = 2, kBarPairFull = 4, kBarSlotEmpty = kBarPairFull + kNumPairBars,
              kBarSFull = kBarSlotEmpty + kNumSlots, kBarPHalf = kBarSFull + 2, kBarPReady = kBarPHalf + 2,
              kBarOFull = kBarPReady + 2, kBarOEmpty = kBarOFull + 2, kBarSchedFull = kBarOEmpty + 2,
              kBarSchedEmpty = kBarSchedFull + 2, kBarStage = kBarSchedEmpty + 2, kBarMerge = kBarStage + 2,
              kBarDrain = kBarMerge + 1, kNumBars = (kBarDrain + 1 + 1) & ~1;
constexpr uint32_t kOffMeta = kOffBar + kNumBars * 8;           // kMetaRing x 8 words
constexpr uint32_t kOffMaskT = kOffMeta + kMetaRing * 32;       // [2][kMaxTp / 32] words (key_block_sets)
constexpr uint32_t kOffMaskS = kOffMaskT + 2 * (kMaxTp / 32) * 4;   // [2][kMaxSp / 32] words, or [4][kMaxSp / 64]
constexpr uint32_t kOffSched = kOffMaskS + 2 * (kMaxSp / 32) * 4;   // two published work items
constexpr uint32_t kOffMisc = kOffSched + 32;                   // tmem base, abort flag
constexpr uint32_t kOffXchg = kOffMisc + 16;                    // split-KV merge: (m, l) of 128 rows
static_assert(256 * 128 * 4 <= kNumSlots * kSlabBytes, "the partial outputs do not fit into the ring");
constexpr uint32_t kOffPartTmp = kOffQ + 16384;                 // cluster mode: (m, l, lr) of the two tiles of one query slab
constexpr uint32_t kOffRowTok = kOffXchg;                       // cluster mode: token of every row that this CTA merges
// Grids with edge blocks: boxes of a slab, {w, h, t, first row / 8 << 8 | map}, as loaded for K and, up to two slabs later, for V.
constexpr int kLists = 3, kMaxListed = 16;
constexpr uint32_t kOffLists = kOffXchg + 128 * 8;
constexpr uint32_t kSmemBytes = kOffLists + kLists * kMaxListed * 16;
constexpr uint32_t kSmemAlloc = kSmemBytes;                     // base alignment comes from the declaration
static_assert(kSmemAlloc <= kMaxSmemBytes, "exceeds the shared memory a CTA may use");

// ----------------------------------------------------------------------------- PTX
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait.  Returns false once the CTA-wide abort flag is set (by this or another
// waiter); `code` names the wait for the status word.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int code,
                                          unsigned long long limit_ns = kTimeoutNs) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = globaltimer_ns();
  uint32_t n = 0;
  while (!mbar_try_wait(bar, parity)) {
    if ((++n & 255u) == 0u) {
      if (*abort_flag != 0) return false;
      if (globaltimer_ns() - t0 > limit_ns) {
        atomicCAS((int*)abort_flag, 0, code);
        return false;
      }
    }
  }
  return true;
}
// warp-uniform variant: every lane waits, the warp agrees on the outcome
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag, int code) {
  const bool ok = mbar_wait(bar, parity, abort_flag, code);
  return __all_sync(0xffffffffu, ok);
}

// Two barriers at once: both probes are issued before either result is used, so a wait that is
// already satisfied costs one shared-memory round trip instead of two.
__device__ __forceinline__ bool mbar_wait2_warp(uint32_t bar_a, uint32_t par_a, uint32_t bar_b, uint32_t par_b,
                                                volatile int* abort_flag, int code_a, int code_b) {
  uint32_t ra, rb;
  asm volatile(
      "{\n\t.reg .pred pa, pb;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 pa, [%2], %3;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 pb, [%4], %5;\n\t"
      "selp.u32 %0, 1, 0, pa;\n\t"
      "selp.u32 %1, 1, 0, pb;\n\t}"
      : "=r"(ra), "=r"(rb) : "r"(bar_a), "r"(par_a), "r"(bar_b), "r"(par_b) : "memory");
  bool ok = true;
  if (!ra) ok = mbar_wait(bar_a, par_a, abort_flag, code_a);
  if (ok && !rb) ok = mbar_wait(bar_b, par_b, abort_flag, code_b);
  return __all_sync(0xffffffffu, ok);
}

// Waits on barrier a and, in the same shared-memory round trip, probes barrier b once;
// *b_done tells whether b's phase was already complete (warp-uniform).
__device__ __forceinline__ bool mbar_wait_probe_warp(uint32_t bar_a, uint32_t par_a, uint32_t bar_b, uint32_t par_b,
                                                     volatile int* abort_flag, int code_a, bool* b_done) {
  uint32_t ra, rb;
  asm volatile(
      "{\n\t.reg .pred pa, pb;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 pa, [%2], %3;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 pb, [%4], %5;\n\t"
      "selp.u32 %0, 1, 0, pa;\n\t"
      "selp.u32 %1, 1, 0, pb;\n\t}"
      : "=r"(ra), "=r"(rb) : "r"(bar_a), "r"(par_a), "r"(bar_b), "r"(par_b) : "memory");
  bool ok = true;
  if (!ra) ok = mbar_wait(bar_a, par_a, abort_flag, code_a);
  *b_done = __all_sync(0xffffffffu, rb != 0u);
  return __all_sync(0xffffffffu, ok);
}

// Programmatic dependent launch: the next kernel of the stream may start once every block has triggered; it sees this
// kernel's results after its own wait.  Both do nothing in a launch without the attribute.  No role waits on a barrier
// before that: a predecessor may run for longer than the barriers' time limit after it has triggered.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// words of an axis' set of attended differences
__host__ __device__ constexpr int axis_words(int n) { return (2 * n - 1 + 31) / 32; }

// Cluster: rank and size, the shared::cluster address of a CTA's shared memory, a barrier over all threads.
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ void st_cluster_u4(uint32_t addr, const uint32_t* v) {
  asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
}
__device__ __forceinline__ void st_cluster_f4(uint32_t addr, float4 v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap* tm, uint32_t bar,
                                            int c0, int c1, int c2, int c3, int c4) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5, %6, %7}], [%2];"
      ::"r"(dst), "l"(tm), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4) : "memory");
}
__device__ __forceinline__ void tma_store_5d(const CUtensorMap* tm, uint32_t src,
                                             int c0, int c1, int c2, int c3, int c4) {
  asm volatile(
      "cp.async.bulk.tensor.5d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5, %6}], [%1];"
      ::"l"(tm), "r"(src), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4) : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// D[tmem] (+)= A[smem desc] * B[smem desc]
__device__ __forceinline__ void tc_mma_ss(uint32_t d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc) : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem desc]
__device__ __forceinline__ void tc_mma_ts(uint32_t d, uint32_t a, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d), "r"(a), "l"(bdesc), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void tc_ld32(uint32_t addr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(addr) : "memory");
}
__device__ __forceinline__ void tc_st32(uint32_t addr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
      ::"r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
        "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
        "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
__device__ __forceinline__ void tc_ld16(uint32_t addr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(addr) : "memory");
}
__device__ __forceinline__ void tc_st8(uint32_t addr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
      ::"r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
      : "memory");
}
__device__ __forceinline__ void tc_st16(uint32_t addr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
// 32 bytes to a 32-byte aligned address: whole sectors even when every lane writes a row of its own
__device__ __forceinline__ void st_global_v8(void* p, const uint32_t* v) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]),
               "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
}
__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// packed fp32 pairs (one instruction for two lanes of work on sm_100)
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
// 2^x for a pair on the FMA/ALU pipes: x = n + f with n = rint(x), f in [-0.5, 0.5];
// 2^f by a cubic (relative error < 8e-5, far below the bf16 rounding of the result), and
// 2^n by adding n to the exponent field.  x is clamped at -125 so the exponent cannot wrap.
__device__ __forceinline__ void exp2_poly_pair(uint64_t x2, float& p0, float& p1) {
  float x0, x1;
  unpack2(x2, x0, x1);
  x0 = fmaxf(x0, -125.f);
  x1 = fmaxf(x1, -125.f);
  const uint64_t xc = pack2(x0, x1);
  const uint64_t magic = pack2(12582912.f, 12582912.f);       // 1.5 * 2^23: rounds to integer
  const uint64_t t2 = add2(xc, magic);
  const uint64_t n2 = add2(t2, pack2(-12582912.f, -12582912.f));
  const uint64_t f2 = fma2(n2, pack2(-1.f, -1.f), xc);
  uint64_t q2 = fma2(f2, pack2(0.05508868396282196f, 0.05508868396282196f), pack2(0.24260404706001282f, 0.24260404706001282f));
  q2 = fma2(q2, f2, pack2(0.6932762265205383f, 0.6932762265205383f));
  q2 = fma2(q2, f2, pack2(0.9999289512634277f, 0.9999289512634277f));
  float q0, q1, t0, t1;
  unpack2(q2, q0, q1);
  unpack2(t2, t0, t1);
  p0 = __int_as_float(__float_as_int(q0) + (__float_as_int(t0) << 23));
  p1 = __int_as_float(__float_as_int(q1) + (__float_as_int(t1) << 23));
}
#ifndef PSA_EMU_PAIRS
#define PSA_EMU_PAIRS 0   // of every 4 pairs of probabilities, this many use exp2_poly_pair (0: all ex2.approx)
#endif


__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

// Instruction descriptor: bf16 x bf16 -> fp32, M = 128, N columns (multiple of 16); A is K-major.
__host__ __device__ constexpr uint32_t instr_desc(bool b_mn_major, uint32_t n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((b_mn_major ? 1u : 0u) << 16) | ((n >> 3) << 17) | ((128u >> 4) << 24);
}
// One elected lane of a converged warp (keeps the branch warp-uniform for the compiler).
__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(pred));
  return pred != 0;
}

// First error of API call `call_id` into the status words.  Nothing clears them: the host takes them as an answer only
// if they carry the id of the call that it asks about.
__device__ __forceinline__ void report_status(int* ws_header, int call_id, int status, int detail) {
  if (atomicExch(ws_header + kWsCallId, call_id) != call_id) {
    ws_header[kWsDetail] = detail;
    ws_header[kWsStatus] = status;
  }
}

// Checked build (-DPSA_DEBUG_CHECKS; the stand-in for a memory checker): every global store index,
// TMA coordinate, ring / table index and TMEM column range computed by the kernel is verified before
// use.  A violation records PSA_ERR_INTERNAL with a code naming the site in the status word and the
// access is skipped -- nothing traps.  In the regular build the checks compile to `true`.
#ifdef PSA_DEBUG_CHECKS
__device__ __noinline__ bool dbg_fail(int* ws_header, int call_id, int code) {
  report_status(ws_header, call_id, PSA_ERR_INTERNAL, code);
  return false;
}
#define PSA_CHECKED(cond, code) ((cond) ? true : dbg_fail(prm.ws_header, prm.call_id, (code)))
#else
#define PSA_CHECKED(cond, code) true
#endif

// The lowest n bits, none if n < 0.
__device__ __forceinline__ uint32_t low_bits(int n) { return n >= 32 ? 0xffffffffu : (n <= 0 ? 0u : (1u << n) - 1u); }

// Class of the block at block coordinates (t, s) (EdgeClass).
__device__ __forceinline__ int block_class(const Geom& g, int t, int s) {
  int c = 0;
  if ((g.edge_axes & 1) && t == g.Tp - 1) c |= 1;
  if ((g.edge_axes & 2) && s >= g.s_edge) c |= 2;
  if ((g.edge_axes & 4) && s % g.Wp == g.Wp - 1) c |= 4;
  return c;
}
// Of spatial block coordinates b .. b + 31, those in the last row, if its blocks are edge blocks.
__device__ __forceinline__ uint32_t last_row_word(const Geom& g, int b) {
  const int d = g.s_edge - b;
  return !(g.edge_axes & 2) || d >= 32 ? 0u : (d <= 0 ? 0xffffffffu : 0xffffffffu << d);
}

// ----------------------------------------------------------------------------- planning
// Work order: heads by descending number of attended pairs (`place`, from the host; heads stay together so that
// concurrently running CTAs share K/V in L2), within a head query blocks by descending number of attended key blocks.
// Heaviest first keeps the last wave short.  Bound by latency (one block per head): axis sets by ballot, counts as
// popcounts of windows of the sets, ranks by counting larger keys, four per shared-memory load.  2.0 us for 40 heads
// of 315 blocks (one thread per pair of coordinates and a compare of two words per pair of blocks: 11.7 us), most of
// it hidden behind the attention kernel's prologue, which starts when every block has reached the trigger.
constexpr int kPlanThreads = 512;
__host__ __device__ __forceinline__ int plan_key_words(const Geom& g) {
  const int sets = axis_words(g.Tp) + axis_words(g.Sp);
  return g.NB > sets ? g.NB : sets;
}
__global__ void __launch_bounds__(kPlanThreads)
plan_kernel(const __grid_constant__ PlanParams hp, const Geom g, int* __restrict__ ws_header,
            psa_head_params* __restrict__ hp_dev, WorkItem* __restrict__ items) {
  // key[NB], cntT[Tp], cntS[Sp]; the axis sets stand where the keys are written later (2n - 1 bits of n coordinates: as many
  // words as the grid has blocks are enough, but for a grid of one block)
  extern __shared__ __align__(16) uint32_t sm[];
  pdl_trigger();
  uint32_t* key = sm;
  uint32_t* cntT = sm + plan_key_words(g);
  uint32_t* cntS = cntT + g.Tp;
  uint32_t* setT = sm;
  uint32_t* setS = setT + axis_words(g.Tp);
  const int h = blockIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const psa_head_params p = hp.p[h];
  // The previous launch on this workspace may still be running; nothing is written before it has finished.
  pdl_wait();
  if (h == 0 && threadIdx.x == 0) ws_header[kWsCounter] = 0;   // the scheduler ticket restarts with every launch
  if (threadIdx.x == 0) hp_dev[h] = p;
  // attended differences, bit d + n - 1 for difference d
  const int wT = axis_words(g.Tp), wS = axis_words(g.Sp);
  for (int w = warp; w < wT + wS; w += kPlanThreads / 32) {
    const bool is_t = w < wT;
    const int i = (is_t ? w : w - wT) * 32 + lane, n = is_t ? g.Tp : g.Sp;
    const bool att = i < 2 * n - 1 && (is_t ? axis_attends(i - (n - 1), p.Tw, p.To, p.Ts) : axis_attends(i - (n - 1), p.Sw, p.So, p.Ss));
    const unsigned m = __ballot_sync(0xffffffffu, att);
    if (lane == 0) setT[w] = m;   // setS follows setT
  }
  __syncthreads();
  // row count of coordinate x: bits n - 1 - x .. 2n - 2 - x of its set
  for (int a = threadIdx.x; a < g.Tp + g.Sp; a += kPlanThreads) {
    const bool is_t = a < g.Tp;
    const uint32_t* set = is_t ? setT : setS;
    const int n = is_t ? g.Tp : g.Sp, x = is_t ? a : a - g.Tp;
    const int lo = n - 1 - x, hi = lo + n;   // [lo, hi)
    int c = 0;
    for (int w = lo >> 5; w <= (hi - 1) >> 5; ++w) {
      uint32_t m = set[w];
      if (w == lo >> 5) m &= 0xffffffffu << (lo & 31);
      if (w == (hi - 1) >> 5) m &= 0xffffffffu >> (31 - ((hi - 1) & 31));
      c += __popc(m);
    }
    cntT[a] = (uint32_t)c;   // cntS follows cntT
  }
  __syncthreads();
  // unique keys: larger count first, then smaller block id (counts are at most NB < 2^16 here)
  for (int qb = threadIdx.x; qb < g.NB; qb += kPlanThreads)
    key[qb] = cntT[qb / g.Sp] * cntS[qb % g.Sp] * (uint32_t)g.NB + (uint32_t)(g.NB - 1 - qb);
  __syncthreads();
  const int ipb = g.items_per_block;
  // Text-query items of all heads first: they attend every key block, so they are the heaviest (behind the lighter
  // items of earlier heads the last one alone kept the launch running: 825 instead of 783 us for 7 heads of 150 blocks).
  // Two text slabs per item; a single one runs in split-KV mode.  Flag in bit 25.
  WorkItem* head_items = items + (size_t)hp.place[h] * g.n_titems;
  for (int it = threadIdx.x; it < g.n_titems; it += kPlanThreads) {
    const int sub0 = 2 * it;
    const int nq = (g.n_ts - sub0) >= 2 ? 2 : 1;
    head_items[it] = make_int4(h, 0, g.NB, sub0 | (nq << 16) | ((nq == 1 ? 1 : 0) << 24) | (1 << 25));
  }
  WorkItem* out = items + (size_t)gridDim.x * g.n_titems + (size_t)hp.place[h] * (g.items_per_head - g.n_titems);
  for (int qb = threadIdx.x; qb < g.NB; qb += kPlanThreads) {
    const uint32_t mine = key[qb];
    int pos = 0, j = 0;
    for (; j + 4 <= g.NB; j += 4) {
      const uint4 k4 = *reinterpret_cast<const uint4*>(key + j);
      pos += (int)(k4.x > mine) + (int)(k4.y > mine) + (int)(k4.z > mine) + (int)(k4.w > mine);
    }
    for (; j < g.NB; ++j) pos += (int)(key[j] > mine);
    const int c = (int)(mine / (uint32_t)g.NB);
    const int n_sub = g.slabs_of[block_class(g, qb / g.Sp, qb % g.Sp)];
    // two-slab items first (heavier), then the odd single-slab items, each in rank order
    for (int it = 0; it < ipb; ++it) {
      const int sub0 = 2 * it;
      if (sub0 >= n_sub) break;
      if (it == 1 && g.items_per_head - g.n_titems != 2 * g.NB) {   // some blocks have no second item: the rank among those that have one
        pos = j = 0;
        for (int tj = 0; tj < g.Tp; ++tj)
          for (int sj = 0, wj = 0; sj < g.Sp; ++sj, ++j) {
            const int cj = g.edge_axes & ((tj == g.Tp - 1 ? 1 : 0) | (sj >= g.s_edge ? 2 : 0) | (wj == g.Wp - 1 ? 4 : 0));
            pos += (int)(g.slabs_of[cj] > 2 && key[j] > mine);
            wj = wj == g.Wp - 1 ? 0 : wj + 1;
          }
      }
      const int nq = (n_sub - sub0) >= 2 ? 2 : 1;
      // A single-slab item runs in split-KV mode: both softmax warpgroups work on that one
      // query slab, one on the even and one on the odd key slabs (flag in bit 24).
      out[(size_t)it * g.NB + pos] = make_int4(h, qb, c, sub0 | (nq << 16) | ((nq == 1 ? 1 : 0) << 24));
    }
  }
}

// ----------------------------------------------------------------------------- attention
// Extents and token count of slab `sub` of a block; `last` selects the tensor-map set.
__device__ __forceinline__ void slab_shape(const Geom& g, int sub, int& et, int& eh, int& ew, int& ntok, int& last) {
  last = (sub == g.n_sub - 1) ? 1 : 0;
  et = g.ct; eh = g.ch; ew = g.cw;
  if (last) {
    if (g.sub_axis == 0) et = g.c_last;
    else if (g.sub_axis == 1) eh = g.c_last;
    else ew = g.c_last;
  }
  ntok = last ? g.n_last : kSlabTokens;
}

__device__ __forceinline__ void slab_origin(const Geom& g, int qb, int sub, int& t0, int& h0, int& w0) {
  const int tb = qb / g.Sp, sb = qb % g.Sp;
  t0 = tb * g.bt;
  h0 = (sb / g.Wp) * g.bh;
  w0 = (sb % g.Wp) * g.bw;
  if (g.sub_axis == 0) t0 += sub * g.ct;
  else if (g.sub_axis == 1) h0 += sub * g.ch;
  else w0 += sub * g.cw;
}

// Descriptor halves.  Only the low word (start address, leading byte offset) changes
// between MMAs; the high word (stride byte offset 1024, version, 128-byte swizzle) is fixed.
constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr, uint32_t lbo_bytes) {
  return ((addr >> 4) & 0x3FFFu) | ((lbo_bytes >> 4) << 16);
}
__device__ __forceinline__ uint64_t make_desc(uint32_t lo) { return ((uint64_t)kDescHi << 32) | lo; }

// Online-softmax step of one query row (one thread) for one key slab of NK keys.
//   tS: TMEM address of the row's scores (fp32, NK columns); the bf16 probabilities are written
//       back over the first NK/2 columns.  tO: the row's output accumulator (128 fp32 columns).
//   meta: validity bits of the slab's keys (bit c of word c/32); all ones when nothing is padded.
//   m_ref / l: running reference maximum (scaled log2 domain) and running sum.
// The reference maximum is lazy: it moves only when the slab's maximum exceeds it by more than
// kRescaleThreshold, so exponentials stay below 2^threshold and O is rarely rescaled.
//   lr (kRounded): running sum of the probabilities as rounded to bf16 for P V.  A shared item's partial results are
// weighted by it, so that the rounding of a dominant probability cancels in out = O / lr; lse comes from l.
template <int NK, bool kRounded>
__device__ __forceinline__ void softmax_slab(uint32_t tS, uint32_t tO, const uint4 meta, bool first,
                                             float scale_log2, float& m_ref, float& l, float& lr, uint32_t bar_half,
                                             uint32_t bar_ready) {
  constexpr int NFULL = NK / 32, REM = NK % 32;
  static_assert(NK % 16 == 0 && NK >= 64 && NK <= 128 && (REM == 0 || REM == 16), "unsupported slab width");
  const float neg_inf = __int_as_float(0xff800000);
  uint32_t s[NK];  // raw scores of this row (fp32 bit patterns), kept in registers
#pragma unroll
  for (int c4 = 0; c4 < NFULL; ++c4) tc_ld32(tS + c4 * 32, s + c4 * 32);
  if (REM) tc_ld16(tS + NFULL * 32, s + NFULL * 32);
  tc_wait_ld();
  if ((meta.x & meta.y & meta.z & meta.w) != 0xffffffffu) {  // 3D-padding: padded key positions score -inf
    // by groups of 32 keys: padding of the slab's outer axes touches few of them
    const uint32_t v[4] = {meta.x, meta.y, meta.z, meta.w};
#pragma unroll
    for (int c4 = 0; c4 < (NK + 31) / 32; ++c4) {
      if (v[c4] != 0xffffffffu) {
#pragma unroll
        for (int c = c4 * 32; c < NK && c < c4 * 32 + 32; ++c)
          if (!((v[c4] >> (c & 31)) & 1u)) s[c] = 0xff800000u;
      }
    }
  }
  // eight independent chains (NK is a multiple of 16): shorter dependency depth
  float a[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) a[i] = fmaxf(__uint_as_float(s[2 * i]), __uint_as_float(s[2 * i + 1]));
#pragma unroll
  for (int c = 16; c < NK; c += 16) {
#pragma unroll
    for (int i = 0; i < 8; ++i) a[i] = max3(a[i], __uint_as_float(s[c + 2 * i]), __uint_as_float(s[c + 2 * i + 1]));
  }
  const float ms = fmaxf(fmaxf(max3(a[0], a[1], a[2]), max3(a[3], a[4], a[5])), fmaxf(a[6], a[7])) * scale_log2;
  if (first) {
    m_ref = ms;  // first slab of the item: nothing accumulated yet
  } else {
    float alpha = 1.f;
    const bool grow = ms > m_ref + kRescaleThreshold;  // also true when m_ref == -inf
    if (grow) {
      alpha = fast_exp2(m_ref - ms);  // 0 when m_ref == -inf
      m_ref = ms;
    }
    if (__any_sync(0xffffffffu, grow)) {
      l *= alpha;
      if (kRounded) lr *= alpha;
#pragma unroll
      for (int c4 = 0; c4 < 4; ++c4) {
        uint32_t o[32];
        tc_ld32(tO + c4 * 32, o);
        tc_wait_ld();
#pragma unroll
        for (int c = 0; c < 32; ++c) o[c] = __float_as_uint(__uint_as_float(o[c]) * alpha);
        tc_st32(tO + c4 * 32, o);
      }
    }
  }
  const float m_use = (m_ref == neg_inf) ? 0.f : m_ref;
  const uint64_t sc2 = pack2(scale_log2, scale_log2), negm2 = pack2(-m_use, -m_use);
  uint64_t sum2 = pack2(0.f, 0.f), sumr2 = pack2(0.f, 0.f);
  // probabilities exp2(scale*s - m_use), bf16, written over the scores in chunks of 32 keys
  auto exp_chunk = [&](int base, int npairs, uint32_t* pk) {
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      if (c >= npairs) break;
      const uint64_t x2 = fma2(pack2(__uint_as_float(s[base + 2 * c]), __uint_as_float(s[base + 2 * c + 1])), sc2, negm2);
      float p0, p1;
      if ((c & 3) < PSA_EMU_PAIRS) {
        exp2_poly_pair(x2, p0, p1);
      } else {
        float x0, x1;
        unpack2(x2, x0, x1);
        p0 = fast_exp2(x0);
        p1 = fast_exp2(x1);
      }
      sum2 = add2(sum2, pack2(p0, p1));
      pk[c] = pack_bf16(p0, p1);
      if (kRounded) sumr2 = add2(sumr2, pack2(__uint_as_float(pk[c] << 16), __uint_as_float(pk[c] & 0xffff0000u)));
    }
  };
#pragma unroll
  for (int c4 = 0; c4 < NFULL; ++c4) {
    uint32_t pk[16];
    exp_chunk(c4 * 32, 16, pk);
    tc_st16(tS + c4 * 16, pk);
    if (c4 == 1) {  // the first 64 keys are final: their P V MMAs may start
      tc_wait_st();
      tc_fence_before();
      mbar_arrive(bar_half);
    }
  }
  if (REM) {
    uint32_t pk[16];
    exp_chunk(NFULL * 32, 8, pk);
    tc_st8(tS + NFULL * 16, pk);
  }
  float sum0, sum1;
  unpack2(sum2, sum0, sum1);
  l += sum0 + sum1;
  if (kRounded) {
    unpack2(sumr2, sum0, sum1);
    lr += sum0 + sum1;
  }
  tc_wait_st();
  tc_fence_before();
  mbar_arrive(bar_ready);
}

// Token (within the head) of row `row` of a query slab, or -1 if the row is padding.
template <bool kBoxes, class Params>
__device__ __forceinline__ long long row_token(const Params& prm, bool textq, int qb, int sub, int row) {
  const Geom& g = prm.g;
  if (textq) {   // text slab: rows are consecutive text tokens; they follow the L video tokens
    const int i = sub * kSlabTokens + row;
    return i < g.n_text ? g.L + i : -1;
  }
  if constexpr (kBoxes) {
    const int tb = qb / g.Sp, sb = qb % g.Sp;
    const EdgeClass& e = prm.cls[block_class(g, tb, sb)];
    const int r = sub * e.step + row;
    if (row >= e.step || r >= e.rows) return -1;
    const int f = r / e.frame, y = r - f * e.frame;
    const int t = tb * g.bt + f, hh = (sb / g.Wp) * g.bh + (y >> e.lw), ww = (sb % g.Wp) * g.bw + (y & ((1 << e.lw) - 1));
    return t < g.T && hh < g.H && ww < g.W ? ((long long)t * g.H + hh) * g.W + ww : -1;
  }
  int t0, h0, w0, et, eh, ew, ntok, last;
  slab_origin(g, qb, sub, t0, h0, w0);
  slab_shape(g, sub, et, eh, ew, ntok, last);
  const int t = t0 + (row >> g.pos_ts), hh = h0 + ((row >> g.pos_ws) & (g.ch - 1)), ww = w0 + (row & (g.cw - 1));
  return (row < ntok && t < g.T && hh < g.H && ww < g.W) ? ((long long)t * g.H + hh) * g.W + ww : -1;
}

// Item i of a launch without planning (every item runs at once, so their order does not matter), by a whole warp; its numbers
// of attended key blocks are left to key_block_sets.
template <bool kEdge>
__device__ __forceinline__ WorkItem direct_item(const Geom& g, int i, int lane) {
  const int n_text_items = g.n_heads * g.n_titems;
  if (i < n_text_items) {
    const int head = i / g.n_titems, sub0 = 2 * (i % g.n_titems);
    const int nq = (g.n_ts - sub0) >= 2 ? 2 : 1;
    return make_int4(head, 0, 0, sub0 | (nq << 16) | ((nq == 1 ? 1 : 0) << 24) | (1 << 25));
  }
  i -= n_text_items;
  const int per_head = g.items_per_head - g.n_titems;
  const int head = i / per_head, r = i - head * per_head;
  int qb = r, sub0 = 0;
  if (r >= g.NB) {   // second items of the blocks that have three slabs
    sub0 = 2;
    qb = r - g.NB;
    if (kEdge) {
      int skip = qb;   // such blocks in front of it
      for (int b = 0; b < g.NB; b += 32) {
        const int j = b + lane;
        uint32_t m = __ballot_sync(0xffffffffu, j < g.NB && g.slabs_of[block_class(g, j / g.Sp, j % g.Sp)] > 2);
        if (skip >= __popc(m)) { skip -= __popc(m); continue; }
        for (; skip > 0; --skip) m &= m - 1;
        qb = b + __ffs(m) - 1;
        break;
      }
    }
  }
  const int n_sub = kEdge ? g.slabs_of[block_class(g, qb / g.Sp, qb % g.Sp)] : g.n_sub;
  const int nq = (n_sub - sub0) >= 2 ? 2 : 1;
  return make_int4(head, qb, 0, sub0 | (nq << 16) | ((nq == 1 ? 1 : 0) << 24));
}

// Numbers of attended block coordinates, packed: temporal ones without and with the edge one (16 bits each); spatial ones of classes
// 0 and 2, and of classes 4 and 6.
struct Attended {
  uint32_t t, s, s4;
  __device__ __forceinline__ int blocks(int c) const {
    const uint32_t x = c & 4 ? s4 : s;
    return (int)((c & 1 ? t >> 16 : t & 0xffffu) * (c & 2 ? x >> 16 : x & 0xffffu));
  }
};

// Words in front of the set of class c's spatial coordinates: two sets, or four of a grid that is cut along both h and w, whose spatial
// blocks are at most half as many (cut_edges).
__device__ __forceinline__ int spatial_set(const Geom& g, int c) { return (g.edge_axes & 6) == 6 ? (c >> 1) * (kMaxSp / 64) : (c > 1 ? kMaxSp / 32 : 0); }

// Attended key-block coordinates of an item's query block (all of them for text queries), one bit per block coordinate, by a
// whole warp: temporal ones without and with the edge one, spatial ones of classes 0, 2, 4 and 6 (those that the grid has).
// (With one set each, and its classes told apart in the loop over the key blocks, edge slabs took the load warp 10,000 clocks of
// its CTA's time instead of 7,000: 3 heads of 22x11x12 with 1x12x16 blocks, all dense, 74 us instead of 58.)
template <bool kEdge>
__device__ __forceinline__ Attended key_block_sets(const Geom& g, bool textq, int qb, const psa_head_params& p, int lane, uint32_t* maskT,
                                                   uint32_t* maskS) {
  const int tq = qb / g.Sp, sq = qb % g.Sp;
  Attended a = {0u, 0u, 0u};
  for (int b = 0; b < g.Tp; b += 32) {
    const int tk = b + lane;
    const unsigned m = __ballot_sync(0xffffffffu, tk < g.Tp && (textq || axis_attends(tk - tq, p.Tw, p.To, p.Ts)));
    const unsigned last = kEdge && (g.edge_axes & 1) && b == ((g.Tp - 1) & ~31) ? m & 1u << ((g.Tp - 1) & 31) : 0u;
    if (lane == 0) {
      maskT[b >> 5] = m & ~last;
      if (kEdge && (g.edge_axes & 1)) maskT[kMaxTp / 32 + (b >> 5)] = last;
    }
    a.t += (uint32_t)(__popc(m & ~last) | __popc(last) << 16);
  }
  for (int b = 0; b < g.Sp; b += 32) {
    const int sk = b + lane;
    const unsigned m = __ballot_sync(0xffffffffu, sk < g.Sp && (textq || axis_attends(sk - sq, p.Sw, p.So, p.Ss)));
    if (!kEdge) {
      if (lane == 0) maskS[b >> 5] = m;
      a.s += (uint32_t)__popc(m);
      continue;
    }
    const unsigned col = g.edge_axes & 4 ? __ballot_sync(0xffffffffu, sk % g.Wp == g.Wp - 1) : 0u, row = last_row_word(g, b);
    if (lane == 0) {
      uint32_t* to = maskS + (b >> 5);
      to[0] = m & ~col & ~row;
      if (g.edge_axes & 2) to[spatial_set(g, 2)] = m & ~col & row;
      if (g.edge_axes & 4) to[spatial_set(g, 4)] = m & col & ~row;
      if ((g.edge_axes & 6) == 6) to[spatial_set(g, 6)] = m & col & row;
    }
    a.s += (uint32_t)(__popc(m & ~col & ~row) | __popc(m & ~col & row) << 16);
    a.s4 += (uint32_t)(__popc(m & col & ~row) | __popc(m & col & row) << 16);
  }
  __syncwarp();
  return a;
}

// Slabs of `n` edge blocks of a class.
__device__ __forceinline__ int class_slabs(const EdgeClass& e, int n) { return e.together > 1 ? (n + e.together - 1) / e.together : n * e.n_slabs; }

// Cluster mode: CTA d of the cluster merges query rows d * rpc .. (d + 1) * rpc - 1 of the item (rpc = nq * 128 /
// cluster size), and every CTA pushes its partial results of those rows into d's shared memory: (m, l, lr) to
// kOffQ [source][row], O as fp32 to kOffRing [source][32 groups of 4 columns][row].  Remote stores are posted; reading
// the partial results from where they were computed took 5 to 9 us at 8 x 128 rows, against 2 for pushing them.
struct Share {
  uint32_t ml, o, step;   // shared::cluster addresses of this thread's row in the merging CTA, bytes between column groups
};
__device__ __forceinline__ Share share_of_row(uint32_t sbase, int r, int nq) {
  const int rpc = nq * 128 / (int)cluster_size(), i = r & (rpc - 1);
  const uint32_t d = (uint32_t)(r / rpc), src = cluster_rank();
  return Share{map_rank(sbase + kOffQ + (src * (uint32_t)rpc + (uint32_t)i) * 16u, d),
               map_rank(sbase + kOffRing + (src * 32u * (uint32_t)rpc + (uint32_t)i) * 16u, d), (uint32_t)rpc * 16u};
}

// The merge itself, by the softmax warpgroups, once all partial results have arrived: sums over the sources in a fixed
// order, out and lse written.
template <class Params>
__device__ __forceinline__ void merge_cluster(const Params& prm, const uint8_t* smem) {
  const Geom& g = prm.g;
  const int4 wi = *reinterpret_cast<const int4*>(smem + kOffSched);   // the item as the load warp published it
  const int head = wi.x & 0xff, nq = (wi.w >> 16) & 0xff;
  const int csize = (int)cluster_size();
  constexpr int kMergeThreads = kThreads - 32 * kFirstSoftmaxWarp;
  const int tid = (int)threadIdx.x - 32 * kFirstSoftmaxWarp;
  const int rpc = nq * 128 / csize;    // 16, 32, 64 or 128
  const int i = tid & (rpc - 1);       // this thread's row
  const int tok = *reinterpret_cast<const int*>(smem + kOffRowTok + i * 4);
  if (tok < 0) return;
  const float neg_inf = __int_as_float(0xff800000);
  const float4* ml = reinterpret_cast<const float4*>(smem + kOffQ) + i;
  float m_all = neg_inf, l_all = 0.f, lr_all = 0.f;
  for (int p = 0; p < csize; ++p) m_all = fmaxf(m_all, ml[p * rpc].x);
  for (int p = 0; p < csize; ++p) {
    const float4 v = ml[p * rpc];
    const float w = (v.x == neg_inf) ? 0.f : fast_exp2(v.x - m_all);
    l_all += w * v.y;
    lr_all += w * v.z;
  }
  const bool empty = !(l_all > 0.f);
  const float inv = empty ? 0.f : 1.f / lr_all;
  if (tid < rpc && PSA_CHECKED(head >= 0 && head < g.n_heads && tok < g.Lt, 0xD15))
    prm.lse[(long long)head * g.Lt + tok] = empty ? neg_inf : (m_all + log2f(l_all)) * 0.6931471805599453f;
  // units of 8 columns of the row; the lanes of a warp read consecutive rows
  for (int cg = tid / rpc; cg < 16; cg += kMergeThreads / rpc) {
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const float4* o = reinterpret_cast<const float4*>(smem + kOffRing) + 2 * cg * rpc + i;
#pragma unroll 4
    for (int p = 0; p < csize; ++p, o += 32 * rpc) {
      const float m = ml[p * rpc].x;
      if (m == neg_inf) continue;   // a share without keys left nothing behind
      const float w = fast_exp2(m - m_all);
      const float4 a = o[0], b = o[rpc];
      acc[0] = fmaf(w, a.x, acc[0]); acc[1] = fmaf(w, a.y, acc[1]); acc[2] = fmaf(w, a.z, acc[2]); acc[3] = fmaf(w, a.w, acc[3]);
      acc[4] = fmaf(w, b.x, acc[4]); acc[5] = fmaf(w, b.y, acc[5]); acc[6] = fmaf(w, b.z, acc[6]); acc[7] = fmaf(w, b.w, acc[7]);
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = empty ? 0.f : acc[e] * inv;   // (empty: no key, or a sum that is not a number)
    if (PSA_CHECKED(head >= 0 && head < g.n_heads && tok < g.Lt, 0xD16))
      *reinterpret_cast<uint4*>(reinterpret_cast<uint16_t*>(prm.out) + (long long)head * prm.out_head + (long long)tok * prm.out_token + cg * 8) =
          make_uint4(pack_bf16(acc[0], acc[1]), pack_bf16(acc[2], acc[3]), pack_bf16(acc[4], acc[5]), pack_bf16(acc[6], acc[7]));
  }
}

// How a launch hands out its work items (Mode).
//   kTicket   persistent CTAs draw planned items (heaviest first) from a ticket
//   kDirect   CTA i runs item i: all items run at once, nothing is planned
//   kShared   cluster i (2, 4 or 8 CTAs) runs planned item i, each CTA taking its share of the attended key blocks
//   kSharedDirect   the same without planning
// (Separate instantiations: the ticket kernel's slab loop is sensitive to what else is compiled with it -- one kernel
// with the mode as an argument was 1.5 to 2 % slower on the 720p layers.)
//   kTicketShort  kTicket for short items of blocks of one slab: bound by what lies between two
//                 items, so the next item's loads and Q K^T run while the last one is still being written out.  The query
//                 buffers are released by the MMAs that read them last (a commit), the output goes from registers to
//                 memory instead of through those buffers, and the accumulators are waited for at the first P V only.
//                 12 heads of 1x8x16 blocks attending 19.5 of them, 8x32x48 grid: 221 -> 198 us
// (A slab of a cut grid goes through a list of boxes, which costs the load warp some 700 clocks: more than it has in split-KV mode.
// 2 heads of 5x16x63 with 1x30x8 blocks, one slab each, took 28.6 us as a cut grid and take 23.6 as a padded one.)
template <int kGrid> struct ArgsOf { typedef TensorMaps maps; typedef AttnParams params; };
template <> struct ArgsOf<kCut> { typedef TensorMapsCut maps; typedef AttnParamsCut params; };
template <int kMode, int kGrid>
__global__ void __launch_bounds__(kThreads, 1)
attn_fwd_kernel(const __grid_constant__ typename ArgsOf<kGrid>::maps tms, const __grid_constant__ HeadParamsArray heads,
                const __grid_constant__ typename ArgsOf<kGrid>::params prm) {
  // 128-byte swizzled slabs need a 1024-byte aligned base; the declaration asks for it and the
  // kernel checks it (a misaligned base is reported through the status word, no work is done).
  constexpr bool kCluster = kMode == kShared || kMode == kSharedDirect, kShort = kMode == kTicketShort;
  constexpr bool kEdge = kGrid != kWhole, kBoxes = kGrid == kCut;
  constexpr bool kDraws = kMode == kTicket || kShort;
  constexpr bool kPlanned = kDraws || kMode == kShared;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = smem_raw;
  const uint32_t sbase = smem_u32(smem);
  const Geom& g = prm.g;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  auto bar = [&](int idx) -> uint32_t { return sbase + kOffBar + 8u * (uint32_t)idx; };
  uint32_t* meta = reinterpret_cast<uint32_t*>(smem + kOffMeta);
  // attended key-block coordinates of the item being loaded
  uint32_t* maskT = reinterpret_cast<uint32_t*>(smem + kOffMaskT);
  uint32_t* maskS = reinterpret_cast<uint32_t*>(smem + kOffMaskS);
  volatile int4* sched = reinterpret_cast<volatile int4*>(smem + kOffSched);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + kOffMisc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kOffMisc + 4);

  // A short query slab leaves its last rows of the Q buffer unwritten; keep them finite.
  if (kDraws || kBoxes || g.n_last != kSlabTokens) {   // (the test alone costs the ticket kernel 2 %: see Mode)
    for (uint32_t off = threadIdx.x * 16u; off < 2u * kSlabBytes; off += kThreads * 16u)
      *reinterpret_cast<uint4*>(smem + kOffQ + off) = make_uint4(0u, 0u, 0u, 0u);
    fence_async_smem();
  }
  if (threadIdx.x == 0) {
    *abort_flag = 0;
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar(kBarQFull + i), 1);
      mbar_init(bar(kBarQEmpty + i), 1);
      mbar_init(bar(kBarSFull + i), 1);
      mbar_init(bar(kBarPHalf + i), 128);
      mbar_init(bar(kBarPReady + i), 128);
      mbar_init(bar(kBarOFull + i), 1);
      mbar_init(bar(kBarOEmpty + i), 128);
      mbar_init(bar(kBarStage + i), 128);
      mbar_init(bar(kBarSchedFull + i), 1);
      mbar_init(bar(kBarSchedEmpty + i), 9);  // the MMA warp and the eight softmax warps
    }
    mbar_init(bar(kBarMerge), 128);
    mbar_init(bar(kBarDrain), 1);
    for (int s = 0; s < kNumPairBars; ++s) mbar_init(bar(kBarPairFull + s), 1);
    for (int s = 0; s < kNumSlots; ++s) mbar_init(bar(kBarSlotEmpty + s), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kWarpMma) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sbase + kOffMisc), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 0) pdl_trigger();
  // Without planning the load warp works its item out here, alongside the rest of the set-up (1.5 us earlier).
  WorkItem first_item = make_int4(-1, 0, 0, 0);
  Attended attended = {0u, 0u, 0u};   // (load warp) by the item's query block
  if constexpr (!kPlanned) {
    if (warp == kWarpLoad) {
      first_item = direct_item<kEdge>(g, (int)(blockIdx.x / cluster_size()), lane);
      attended = key_block_sets<kEdge>(g, ((first_item.w >> 25) & 1) != 0, first_item.y, heads.p[first_item.x], lane, maskT, maskS);
    }
  }
  // A persistent CTA has one idle thread wait for the kernel before, on behalf of every role behind the barrier.  (Waits in
  // the roles, or by more threads here, made launches of many items 0.5 % slower: 33 heads of 147 blocks of 240 tokens 16.10
  // ms without, 16.11 with one thread, 16.19 with a wait in every role.)  Launches of few items wait in the roles, behind
  // their own set-up.
  if constexpr (kDraws) {
    if (threadIdx.x == 64) pdl_wait();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // The CTA owns all 512 TMEM columns, so the allocation starts at column 0, lane 0; using
  // the constant keeps every TMEM address of the MMA stream in uniform registers.  Checked:
  // any other base is reported through the status word and the CTA does no work.
  constexpr uint32_t tmem = 0u;
  const bool tmem_ok = (*tmem_slot == 0u) && ((sbase & 1023u) == 0u);
  if (!tmem_ok && threadIdx.x == 0) atomicCAS((int*)abort_flag, 0, (*tmem_slot == 0u) ? 0x501 : 0x500);

  // Work items are handed out through a two-entry ring: the load warp draws a ticket from
  // a global counter (items are stored heaviest first), publishes the item, and the other
  // roles pick it up.  A negative head ends the kernel.
  auto next_item = [&](uint32_t n, WorkItem& wi) -> bool {
    const uint32_t slot = n & 1u;
    if (!tmem_ok) return false;
    if (!mbar_wait_warp(bar(kBarSchedFull + slot), (n >> 1) & 1u, abort_flag, 0x400)) return false;
    // broadcast from lane 0 so that the compiler knows the item (and every loop bound
    // derived from it) is warp-uniform
    wi.x = __shfl_sync(0xffffffffu, sched[slot].x, 0);
    wi.y = __shfl_sync(0xffffffffu, sched[slot].y, 0);
    wi.z = __shfl_sync(0xffffffffu, sched[slot].z, 0);
    wi.w = __shfl_sync(0xffffffffu, sched[slot].w, 0);
    __syncwarp();
    if (lane == 0) mbar_arrive(bar(kBarSchedEmpty + slot));
    return wi.x >= 0;
  };

  if ((warp >> 2) == kUtilGroup) {
  // Utility warpgroup: give registers away (the budget is re-split per warpgroup).
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsUtil));
  if (warp == kWarpLoad) {
    // ======================================================================= load warp
    // Ring tiles are issued in the order K_0, V_0, K_1, V_1, ...; the MMA warp needs V_j and
    // K_{j+1} at the same moment, so those two travel under one "pair" barrier
    // (K_0 and the last V of an item travel alone).
    uint32_t slot_i = 0, slot_ph = 1;   // ring slot of the next tile and the parity its wait needs; pair barrier of the next arrival
    uint32_t pair_i = 0;
    uint32_t pair_g = 0;       // pair barriers armed so far
    uint32_t kv_g = 0;         // key slabs issued so far
    uint32_t it_q0 = 0, it_q1 = 0; // items in which query slab i was active
    // block -> row of the spatial block grid without a division: sk, Wp <= 2^11
    const uint32_t magic_w = ((1u << 22) + (uint32_t)g.Wp - 1u) / (uint32_t)g.Wp;
    auto class_at = [&](int i) -> int {
      if constexpr (kBoxes) return prm.order[i];
      return i == 0 ? 0 : g.edge_axes;
    };
    int n_classes = 1;
    bool late = !kDraws;   // an item is published when its classes of key blocks have been counted
    if constexpr (kBoxes) {
      n_classes = prm.n_classes;
      late = late || !prm.planned;
    } else if constexpr (kEdge) {
      n_classes = g.edge_axes != 0 ? 2 : 1;
      late = late || g.edge_axes != 0;
    }
    bool ok = tmem_ok;
    pdl_wait();   // the work items are written by the planning kernel, q, k and v by whatever ran before
    for (uint32_t n = 0; ok; ++n) {
      const uint32_t sslot = n & 1u;
      ok = mbar_wait_warp(bar(kBarSchedEmpty + sslot), ((n >> 1) & 1u) ^ 1u, abort_flag, 0x401);
      if (!ok) break;
      WorkItem wi = make_int4(-1, 0, 0, 0);
      int skip = 0, left = 0x7fffffff;   // attended key blocks before this CTA's share, and those still to load (kBoxes: of a class)
      // kBoxes: the attended blocks of class c that are this CTA's (all of them, or its share: by rows, cut between blocks), and how
      // many others come before them.  `before`: rows of the classes before, carried along.
      // (32 bits hold 8 times the rows of the largest block grid, 58,112 x 384)
      auto blocks_of = [&](int c, int all, int& before, int* skip) -> int {
        const int n = attended.blocks(c);
        *skip = 0;
        if constexpr (kCluster && kBoxes) {
          const int per = prm.cls[c].rows, r = (int)cluster_rank(), size = (int)cluster_size();
          auto upto = [&](int rows) -> int { return rows <= before ? 0 : min((rows - before) / per, n); };
          const int from = upto(all * r / size), to = upto(all * (r + 1) / size);
          before += n * per;
          *skip = from;
          return to - from;
        }
        return n;
      };
      int all = 0;   // rows of the attended blocks
      auto take_share = [&]() {   // (every lane)
        // (this CTA's share of the item's key blocks; the text keys go with the last share)
        if (kCluster && cluster_rank() + 1 < cluster_size()) wi.w |= 1 << 26;
        if constexpr (kBoxes) {
          if constexpr (kCluster) {
            for (int i = 0; i < n_classes; ++i) all += attended.blocks(class_at(i)) * prm.cls[class_at(i)].rows;
          }
          int before = 0, edge_slabs = 0;
          wi.z = 0;
#pragma unroll 1
          for (int i = 0; i < n_classes; ++i) {
            const int c = class_at(i), n = blocks_of(c, all, before, &skip);
            if (prm.cls[c].in_pattern) wi.z += n;
            else edge_slabs += n ? class_slabs(prm.cls[c], n) : 0;
          }
          wi.x |= edge_slabs << 8;
        } else {   // whole blocks, those of fewer slabs last
          wi.z = attended.blocks(0);
          const int main = wi.z, edge = n_classes > 1 ? attended.blocks(g.edge_axes) : 0, edge_slabs = kEdge ? g.slabs_of[g.edge_axes] : 0;
          left = main + edge;
          if constexpr (kCluster) {   // by slabs, cut between blocks
            const int slabs = kEdge && edge != 0 ? g.main_slabs : 1, all = main * slabs + edge * edge_slabs, r = (int)cluster_rank();
            auto by = [](int n, int d) -> int { return d == 1 ? n : (d == 2 ? n >> 1 : n / 3); };   // (a division costs this warp some 400 clocks)
            auto upto = [&](int n) -> int { return n <= main * slabs ? by(n, slabs) : main + by(n - main * slabs, edge_slabs); };
            const int shift = 31 - __clz((int)cluster_size());   // 2, 4 or 8 CTAs
            skip = upto(all * r >> shift);
            left = upto(all * (r + 1) >> shift) - skip;
            wi.z = max(min(skip + left, main) - skip, 0);
          }
          if (edge != 0) wi.x |= (left - wi.z) * edge_slabs << 8;
        }
      };
      auto publish = [&]() {   // by lane 0
        sched[sslot].x = wi.x; sched[sslot].y = wi.y; sched[sslot].z = wi.z; sched[sslot].w = wi.w;
        mbar_arrive(bar(kBarSchedFull + sslot));
      };
      if constexpr (kDraws) {
        if (lane == 0) {
          const int ticket = atomicAdd(prm.ws_header + kWsCounter, 1);
          if (ticket < prm.n_items) wi = prm.items[ticket];
          if (!late) publish();
        }
        wi.x = __shfl_sync(0xffffffffu, wi.x, 0);
        wi.y = __shfl_sync(0xffffffffu, wi.y, 0);
        wi.w = __shfl_sync(0xffffffffu, wi.w, 0);
      } else if (n == 0) {
        wi = kPlanned ? prm.items[blockIdx.x / cluster_size()] : first_item;
      }
      if (kPlanned && wi.x >= 0) attended = key_block_sets<kEdge>(g, ((wi.w >> 25) & 1) != 0, wi.y, prm.hp_dev[wi.x], lane, maskT, maskS);
      if (late) {
        if (wi.x >= 0) take_share();
        if (lane == 0) publish();
      }
      if (wi.x < 0) break;
      const int head = kEdge ? wi.x & 0xff : wi.x, qb = wi.y, sub0 = wi.w & 0xffff, nq = (wi.w >> 16) & 0xff;
      if (!PSA_CHECKED(head < g.n_heads && qb >= 0 && qb <= g.NB && nq >= 1 && nq <= 2 &&
                       sub0 + nq <= ((wi.w >> 25) & 1 ? g.n_ts : g.n_sub), 0xD04)) {
        if (lane == 0) atomicCAS((int*)abort_flag, 0, 0xD04);   // a malformed item: stop this CTA through the abort path
        ok = false;
        break;
      }
      const int lag = ((wi.w >> 24) & 1) ? 2 : 1;   // V_j travels with K_{j+lag} (2 in split-KV mode)
      const bool textq = ((wi.w >> 25) & 1) != 0;   // the queries are text tokens: every key is attended
      const int head_ld = prm.shared_qkv ? 0 : head;   // head coordinate of the q, k, v loads
      // A box into a tile, at a multiple of 8 rows.
      auto load_box = [&](uint32_t dst, const CUtensorMap* map, uint32_t pb, int t, int h, int w) {
        tma_load_5d(dst, map, pb, 0, w, h, t, head_ld);
        tma_load_5d(dst + kHalfBytes, map, pb, 64, w, h, t, head_ld);
      };
      // kBoxes: every slab is a list of boxes; list `list` is the one being made.
      int4* lists = reinterpret_cast<int4*>(smem + kOffLists);
      int list = 0;
      // The first nv boxes of list lv into a tile of V, the first nk of list lk into one of K (or of Q), by a whole warp.  The lists
      // are read at once, by box_of: a shared-memory round trip takes 150 to 450 clocks while the tensor core is busy.
      auto box_of = [&](int lv, int lk) -> int4 { return lists[(lane < kMaxListed ? lv : lk) * kMaxListed + (lane & (kMaxListed - 1))]; };
      auto load_lists = [&](const int4& mine, uint32_t pb, const CUtensorMap* maps_v, uint32_t dv, int nv, const CUtensorMap* maps_k, uint32_t dk, int nk) {
#pragma unroll 1
        for (int b = 0; b < nv + nk; ++b) {
          const int from = b < nv ? b : kMaxListed + b - nv;
          const int w = __shfl_sync(0xffffffffu, mine.x, from), h = __shfl_sync(0xffffffffu, mine.y, from), t = __shfl_sync(0xffffffffu, mine.z, from),
                    to = __shfl_sync(0xffffffffu, mine.w, from);
          if (lane == 0 && PSA_CHECKED(nv <= kMaxListed && nk <= kMaxListed && (to & 255) < kMaxMaps && (to >> 8) < 16 && w >= 0 && h >= 0 && t >= 0 && t <= g.T, 0xD07))
            load_box((b < nv ? dv : dk) + ((uint32_t)to >> 8) * 1024u, (b < nv ? maps_v : maps_k) + (to & 255), pb, t, h, w);
        }
      };
      // The boxes of slab `sub` of a block; their number.
      auto list_boxes = [&](const EdgeClass& e, int sub, int t0, int h0, int w0) -> int {
        const int first = e.first_box[sub], n = e.first_box[sub + 1] - first;
        if (lane < n) {
          const EdgeBox x = e.box[first + lane];
          const int4 zeros = make_int4(0, 0, g.T, x.row8 << 8 | x.map);
          lists[list * kMaxListed + lane] = x.t == kZeros ? zeros : make_int4(w0 + x.w, h0 + x.h, t0 + x.t, zeros.w);
        }
        __syncwarp();
        return n;
      };
      const int qcls = kBoxes && !textq ? block_class(g, qb / g.Sp, qb % g.Sp) : 0;
      // query slabs
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        if (i >= nq) break;
        const uint32_t itq = i == 0 ? it_q0 : it_q1;
        ok = mbar_wait_warp(bar(kBarQEmpty + i), (itq & 1u) ^ 1u, abort_flag, 0x100 + i);
        if (!ok) break;
        int t0, h0, w0, et, eh, ew, ntok, last, n_boxes = 0;
        if constexpr (kBoxes) {
          if (!textq) {
            const EdgeClass& e = prm.cls[qcls];
            slab_origin(g, qb, 0, t0, h0, w0);
            n_boxes = list_boxes(e, sub0 + i, t0, h0, w0);
            const bool whole = sub0 + i + 1 < e.n_slabs || !(e.in_pattern || e.together > 1);
            if (e.together > 1) n_boxes = 1;   // (a block alone: no box of zeros)
            if (lane == 0) mbar_expect_tx(bar(kBarQFull + i), whole ? kSlabBytes : (uint32_t)(e.together > 1 ? e.rows : g.main_last) * 256u);
            load_lists(box_of(list, list), bar(kBarQFull + i), tms.q, 0u, 0, tms.q, sbase + kOffQ + (uint32_t)i * kSlabBytes, n_boxes);
          }
        }
        if (lane == 0 && n_boxes == 0) {   // (n_boxes: kBoxes, video queries)
          if (textq) {   // text slab: 128 tokens from the text map, token index in the second coordinate
            t0 = 0; h0 = 0; w0 = (sub0 + i) * kSlabTokens; ntok = kSlabTokens; last = 2;
          } else {
            slab_origin(g, qb, sub0 + i, t0, h0, w0);
            slab_shape(g, sub0 + i, et, eh, ew, ntok, last);
          }
          const uint32_t dst = sbase + kOffQ + (uint32_t)i * kSlabBytes;
          if (PSA_CHECKED(w0 >= 0 && h0 >= 0 && t0 >= 0 && head_ld >= 0 && head_ld < g.n_heads && last >= 0 && last <= 2 &&
                          ntok > 0 && ntok <= kSlabTokens &&
                          (textq || (w0 < g.Wp * g.bw && h0 < g.Hp * g.bh && t0 < g.Tp * g.bt)), 0xD01)) {   // inside the padded grid
            mbar_expect_tx(bar(kBarQFull + i), (uint32_t)ntok * 256u);
            load_box(dst, &tms.q[last], bar(kBarQFull + i), t0, h0, w0);
          }
        }
        if (i == 0) ++it_q0; else ++it_q1;
      }
      if (!ok) break;
      // key / value slabs in ascending key-block id.  Up to `lag` slabs wait for their V load.
      int npend = 0;
      int at0 = 0, ah0 = 0, aw0 = 0, alast = 0, antok = kSlabTokens;  // oldest pending slab (kBoxes: at0 boxes)
      int bt0 = 0, bh0 = 0, bw0 = 0, blast = 0, bntok = kSlabTokens;  // newer pending slab (lag 2)
      // Slots of the next tiles, V of the oldest pending slab (if it is due) and K of the new one.
      bool with_v;
      uint32_t v_slot, k_slot, k_par;
      auto slot_next = [&](uint32_t sl, uint32_t& ph) -> uint32_t {
        ph ^= sl + 1u == (uint32_t)kNumSlots ? 1u : 0u;
        return sl + 1u == (uint32_t)kNumSlots ? 0u : sl + 1u;
      };
      auto wait_slots = [&]() {
        with_v = npend == lag;
        const uint32_t v_par = slot_ph;
        v_slot = k_slot = slot_i;
        k_par = slot_ph;
        if (with_v) k_slot = slot_next(k_slot, k_par);
        ok = with_v ? mbar_wait2_warp(bar(kBarSlotEmpty + v_slot), v_par, bar(kBarSlotEmpty + k_slot), k_par, abort_flag, 0x111, 0x110)
                    : mbar_wait_warp(bar(kBarSlotEmpty + k_slot), k_par, abort_flag, 0x110);
      };
      // The tiles are on their way: queue this slab's V.
      auto issued = [&](int t0, int h0, int w0, int last, int ntok) {
        slot_ph = k_par;
        slot_i = slot_next(k_slot, slot_ph);
        ++pair_g;
        pair_i = pair_i + 1u == (uint32_t)kNumPairBars ? 0u : pair_i + 1u;
        ++kv_g;
        if (with_v) {
          if (lag == 2) { at0 = bt0; ah0 = bh0; aw0 = bw0; alast = blast; antok = bntok; }
          --npend;
        }
        if (npend == 0) { at0 = t0; ah0 = h0; aw0 = w0; alast = last; antok = ntok; }
        else { bt0 = t0; bh0 = h0; bw0 = w0; blast = last; bntok = ntok; }
        ++npend;
      };
      // One key slab: K now, V of the slab issued `lag` slabs earlier under the same barrier.
      auto issue_slab = [&](int t0, int h0, int w0, int last, int ntok, uint32_t vw0, uint32_t vw1, uint32_t vw2,
                            uint32_t vw3) {
        wait_slots();
        if (!ok) return;
        if (lane == 0 && PSA_CHECKED(v_slot < (uint32_t)kNumSlots && k_slot < (uint32_t)kNumSlots && t0 >= 0 && h0 >= 0 && w0 >= 0 &&
                                     last >= 0 && last <= 2 && ntok > 0 && ntok <= kSlabTokens &&
                                     (!with_v || (at0 >= 0 && ah0 >= 0 && aw0 >= 0 && alast >= 0 && alast <= 2)), 0xD02)) {
          uint32_t* m = meta + (kv_g % kMetaRing) * 8;
          m[0] = vw0; m[1] = vw1; m[2] = vw2; m[3] = vw3;
          const uint32_t pb = bar(kBarPairFull + pair_i);
          mbar_expect_tx(pb, (uint32_t)((with_v ? antok : 0) + ntok) * 256u);
          if (with_v) load_box(sbase + kOffRing + v_slot * kSlabBytes, &tms.v[alast], pb, at0, ah0, aw0);
          load_box(sbase + kOffRing + k_slot * kSlabBytes, &tms.k[last], pb, t0, h0, w0);
        }
        issued(t0, h0, w0, last, ntok);
      };
      // The same for the slab of the n boxes of the list; vw: word `lane` of its validity bits, in lanes 0 to 3.
      auto issue_list = [&](int n, int ntok, uint32_t vw) {
        __syncwarp();
        const int4 mine = box_of(list < lag ? list + kLists - lag : list - lag, list);
        wait_slots();
        if (!ok) return;
        if (lane < 4) meta[(kv_g % kMetaRing) * 8 + lane] = vw;
        __syncwarp();
        if (PSA_CHECKED(v_slot < (uint32_t)kNumSlots && k_slot < (uint32_t)kNumSlots && ntok > 0 && ntok <= kSlabTokens, 0xD09)) {
          const uint32_t pb = bar(kBarPairFull + pair_i);
          if (lane == 0) mbar_expect_tx(pb, (uint32_t)((with_v ? antok : 0) + ntok) * 256u);
          load_lists(mine, pb, tms.v, sbase + kOffRing + v_slot * kSlabBytes, with_v ? at0 : 0, tms.k, sbase + kOffRing + k_slot * kSlabBytes, n);
        }
        issued(n, 0, 0, 0, ntok);
        list = list == kLists - 1 ? 0 : list + 1;
      };
      // classes in turn
      int before = 0;
#pragma unroll 1
      for (int ci = 0; ok && ci < n_classes; ++ci) {
      const int c = class_at(ci);
      if constexpr (kBoxes) left = blocks_of(c, all, before, &skip);
      const uint32_t *mask_t = maskT + (c & 1) * (kMaxTp / 32), *mask_s = maskS + spatial_set(g, c);
      int listed = 0;
      // The class in registers (constants by a computed index are slow): lane b holds box b, lane 4 s + i word i of slab s's validity.
      int rows = 0, n_slabs = 1, together = 1, n_full = 0;
      uint32_t first_box = 0, valid = 0, last_keys = kSlabTokens;
      EdgeBox mine_box = {};
      n_slabs = kEdge ? g.slabs_of[c] : g.n_sub;
      if constexpr (kBoxes) {
        const EdgeClass& e = prm.cls[c];
        rows = e.rows;
        together = e.together;
        n_full = e.together + e.n_boxes - 1;
        first_box = *reinterpret_cast<const uint32_t*>(e.first_box);
        if (e.in_pattern) last_keys = (uint32_t)g.main_last;
        if (lane < 12) valid = e.valid[lane >> 2][lane & 3];
        if (lane < kMaxEdgeBoxes) mine_box = e.box[lane];
      }
      for (int tw = 0; ok && left > 0 && tw < g.Tp; tw += 32) {
        uint32_t mt = mask_t[tw >> 5];
        while (ok && left > 0 && mt) {
          const int tk = tw + __ffs(mt) - 1;
          mt &= mt - 1;
          for (int sw = 0; ok && left > 0 && sw < g.Sp; sw += 32) {
            uint32_t ms = mask_s[sw >> 5];
            while (ok && ms) {
              const int sk = sw + __ffs(ms) - 1;
              ms &= ms - 1;
              if constexpr (kCluster) {
                if (skip > 0) { --skip; continue; }
                if (left == 0) break;
              }
              if (kCluster || kBoxes) --left;
              const int hb = (int)(((unsigned long long)(uint32_t)sk * magic_w) >> 22);
              int t0 = tk * g.bt, h0 = hb * g.bh, w0 = (sk - hb * g.Wp) * g.bw;
              if constexpr (kBoxes) {
                int4* const to = lists + list * kMaxListed;
                if (together > 1) {
                  if (lane == 0 && PSA_CHECKED(listed < kMaxListed && list < kLists, 0xD06)) to[listed] = make_int4(w0, h0, t0, listed * rows << 5 | mine_box.map);
                  if (++listed < together && left > 0) continue;
                  // zeros in the place of what a full slab has more of
                  const int map0 = __shfl_sync(0xffffffffu, (int)mine_box.map, 0);
                  if (lane >= listed && lane < together) to[lane] = make_int4(0, 0, g.T, lane * rows << 5 | map0);
                  if (lane == 1 && n_full > together) to[together] = make_int4(0, 0, g.T, mine_box.row8 << 8 | mine_box.map);
                }
#pragma unroll 1
                for (int sub = 0; ok && sub < n_slabs; ++sub) {
                  const int first = (int)(first_box >> (8 * sub) & 255u);
                  int n = (int)(first_box >> (8 * sub + 8) & 255u) - first;
                  uint32_t vw = __shfl_sync(0xffffffffu, valid, 4 * sub + (lane & 3));
                  if (together > 1) {
                    n = n_full;
                    vw &= low_bits(listed * rows - 32 * (lane & 3));
                    listed = 0;
                  } else if (lane >= first && lane < first + n) {
                    const bool zeros = mine_box.t == kZeros;
                    lists[list * kMaxListed + lane - first] = make_int4(zeros ? 0 : w0 + mine_box.w, zeros ? 0 : h0 + mine_box.h, zeros ? g.T : t0 + mine_box.t,
                                                                        mine_box.row8 << 8 | mine_box.map);
                  }
                  issue_list(n, sub + 1 == n_slabs ? (int)last_keys : kSlabTokens, vw);
                }
              } else {
              for (int sub = 0; ok && sub < n_slabs; ++sub) {
                const int last = (sub == g.n_sub - 1) ? 1 : 0, ntok = last ? g.n_last : kSlabTokens;
                // validity of the slab's key positions (3D-padding): bit c of word c/32; ones beyond a short slab
                uint32_t vw0 = 0xffffffffu, vw1 = 0xffffffffu, vw2 = 0xffffffffu, vw3 = 0xffffffffu;
                if constexpr (kGrid == kPadded) {
                  const int et = last && g.sub_axis == 0 ? g.c_last : g.ct, eh = last && g.sub_axis == 1 ? g.c_last : g.ch,
                            ew = last && g.sub_axis == 2 ? g.c_last : g.cw;
                  const int rt = g.T - t0, rh = g.H - h0, rw = g.W - w0;
                  if (et > rt || eh > rh || ew > rw) {
                    auto valid = [&](int i) -> bool {
                      const int x = lane + 32 * i;
                      return ((x >> g.pos_ts) < rt && ((x >> g.pos_ws) & (g.ch - 1)) < rh && (x & (g.cw - 1)) < rw) || x >= ntok;
                    };
                    vw0 = __ballot_sync(0xffffffffu, valid(0));
                    vw1 = __ballot_sync(0xffffffffu, valid(1));
                    vw2 = __ballot_sync(0xffffffffu, valid(2));
                    vw3 = __ballot_sync(0xffffffffu, valid(3));
                  }
                }
                issue_slab(t0, h0, w0, last, ntok, vw0, vw1, vw2, vw3);
                if (g.sub_axis == 0) t0 += g.ct;
                else if (g.sub_axis == 1) h0 += g.ch;
                else w0 += g.cw;
              }
              }
            }
          }
        }
      }
      }
      // text key slabs: attended by every query; tokens beyond n_text are zero-filled and masked
      const int n_ts = kCluster && ((wi.w >> 26) & 1) ? 0 : g.n_ts;
      for (int ts = 0; ok && ts < n_ts; ++ts) {
        const int tok0 = ts * kSlabTokens;
        const int nvalid = g.n_text - tok0;   // >= 1
        if constexpr (kBoxes) {
          if (lane == 0) lists[list * kMaxListed] = make_int4(tok0, 0, 0, 2);
          issue_list(1, kSlabTokens, low_bits(nvalid - 32 * (lane & 3)));
        } else issue_slab(0, 0, tok0, 2, kSlabTokens, low_bits(nvalid), low_bits(nvalid - 32), low_bits(nvalid - 64), low_bits(nvalid - 96));
      }
      while (ok && npend > 0) {  // V of the item's last slab(s), one pair barrier each
        const uint32_t v_slot = slot_i;
        ok = mbar_wait_warp(bar(kBarSlotEmpty + v_slot), slot_ph, abort_flag, 0x112);
        if (!ok) break;
        const uint32_t pb = bar(kBarPairFull + pair_i), dv = sbase + kOffRing + v_slot * kSlabBytes;
        if (PSA_CHECKED(v_slot < (uint32_t)kNumSlots && at0 >= 0 && ah0 >= 0 && aw0 >= 0 && alast >= 0 && alast <= 2 && antok > 0 &&
                        antok <= kSlabTokens, 0xD03)) {
          if (lane == 0) mbar_expect_tx(pb, (uint32_t)antok * 256u);
          if constexpr (kBoxes) {
            const int vl = list < npend ? list + kLists - npend : list - npend;
            load_lists(box_of(vl, vl), pb, tms.v, dv, at0, tms.v, dv, 0);
          } else if (lane == 0) {
            load_box(dv, &tms.v[alast], pb, at0, ah0, aw0);
          }
        }
        slot_i = slot_next(slot_i, slot_ph);
        ++pair_g;
        pair_i = pair_i + 1u == (uint32_t)kNumPairBars ? 0u : pair_i + 1u;
        at0 = bt0; ah0 = bh0; aw0 = bw0; alast = blast; antok = bntok;
        --npend;
      }
      if (!ok) break;
    }
    // Let every load that was issued land before the CTA retires: wait for the last armed
    // phase of each pair barrier and of the Q barriers (bounded; the abort flag no longer
    // cuts these short).
    if (lane == 0) {
      for (uint32_t back = 0; back < (uint32_t)kNumPairBars && back < pair_g; ++back) {
        const uint32_t pg = pair_g - 1 - back;
        const unsigned long long t0 = globaltimer_ns();
        while (!mbar_try_wait(bar(kBarPairFull + pg % kNumPairBars), (pg / kNumPairBars) & 1u)) {
          if (globaltimer_ns() - t0 > kTimeoutNs) break;
        }
      }
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const uint32_t itq = i == 0 ? it_q0 : it_q1;
        if (itq == 0) continue;
        const unsigned long long t0 = globaltimer_ns();
        while (!mbar_try_wait(bar(kBarQFull + i), (itq - 1) & 1u)) {
          if (globaltimer_ns() - t0 > kTimeoutNs) break;
        }
      }
    }
    __syncwarp();
  } else if (warp == kWarpMma) {
    // ======================================================================= MMA warp
    constexpr uint32_t kIdescPV = instr_desc(true, 128);  // N = head_dim
    // ring slot of the next tile and pair barrier of the next arrival: wrapping index + phase bit
    uint32_t slot_i = 0, pair_i = 0, pair_ph = 0;
    auto slot_next = [&](uint32_t sl) -> uint32_t { return sl + 1u == (uint32_t)kNumSlots ? 0u : sl + 1u; };
    auto pair_adv = [&]() { if (++pair_i == (uint32_t)kNumPairBars) { pair_i = 0; pair_ph ^= 1u; } };
    uint32_t it_q0 = 0, it_q1 = 0;
    uint32_t cnt_s0 = 0, cnt_s1 = 0;  // P_i tiles consumed so far
    bool ok = true;
    const uint32_t q_lo = desc_lo(sbase + kOffQ, 16);
    const uint32_t ring_lo_k = desc_lo(sbase + kOffRing, 16);
    const uint32_t ring_lo_v = desc_lo(sbase + kOffRing, kHalfBytes);
    constexpr uint32_t kSlabStep = kSlabBytes >> 4;  // descriptor address units per slab

    // S_i = Q_i K^T over head_dim = 128: 8 MMAs of K = 16; both operands K-major, SW128.
    // nk = keys of the slab (N of the instruction): 128, or fewer for a block's last slab.
    // iq: Q buffer; it: S tile written (they differ only in split-KV items).
    auto issue_qk = [&](int iq, uint32_t kslot, int nk, int it) {
      if (!PSA_CHECKED(iq >= 0 && iq < 2 && it >= 0 && it < 2 && kslot < (uint32_t)kNumSlots && nk >= 16 && nk <= 128 && (nk & 15) == 0, 0xD20))
        return;
      const uint32_t a0 = q_lo + (uint32_t)iq * kSlabStep, b0 = ring_lo_k + kslot * kSlabStep;
      const uint32_t idesc = instr_desc(false, (uint32_t)nk);
#pragma unroll
      for (int kk = 0; kk < 8; ++kk) {
        const uint32_t off = (uint32_t)(kk >> 2) * (kHalfBytes >> 4) + (uint32_t)(kk & 3) * 2u;
        tc_mma_ss(tmem + (uint32_t)it * 128u, make_desc(a0 + off), make_desc(b0 + off), idesc, kk > 0 ? 1u : 0u);
      }
    };
    // O_i (+)= P_i V over 128 keys: 8 MMAs of K = 16; A = bf16 P in TMEM (8 columns per
    // step), B = V slab as loaded (keys x head_dim, head_dim contiguous) = MN-major SW128:
    // 16 keys advance 2048 bytes, the second 64 columns of head_dim sit one half slab
    // further (leading byte offset).
    auto issue_pv_half = [&](int i, uint32_t vslot, int half, bool accumulate, int nk) {
      if (!PSA_CHECKED(i >= 0 && i < 2 && half >= 0 && half < 2 && vslot < (uint32_t)kNumSlots && nk >= 16 && nk <= 128, 0xD21)) return;
      const uint32_t b0 = ring_lo_v + vslot * kSlabStep;
#pragma unroll
      for (int k4 = 0; k4 < 4; ++k4) {
        const int kk = half * 4 + k4;
        if (kk * 16 >= nk) break;   // a short slab has fewer 16-key steps
        tc_mma_ts(tmem + 256u + (uint32_t)i * 128u, tmem + (uint32_t)i * 128u + (uint32_t)kk * 8u,
                  make_desc(b0 + (uint32_t)kk * (2048u >> 4)), kIdescPV, (accumulate || kk > 0) ? 1u : 0u);
      }
    };

    uint32_t it_o0 = 0, it_o1 = 0;    // items in which accumulator O_i was used
    if constexpr (!kDraws) pdl_wait();   // (see pdl_wait)
    // keys of a slab from its index within its block (r = j mod n_sub, carried along: no division)
    const int n_sub = kEdge ? g.main_slabs : g.n_sub, n_last = kEdge ? g.main_last : g.n_last;
    const int r_last = n_sub - 1;
    auto nk_at = [&](int r) -> int { return r == r_last ? n_last : kSlabTokens; };
    auto r_inc = [&](int r) -> int { return r == r_last ? 0 : r + 1; };

    for (uint32_t n = 0; ok; ++n) {
      WorkItem wi;
      if (!next_item(n, wi)) break;
      const int nq = (wi.w >> 16) & 0xff;
      const bool split = ((wi.w >> 24) & 1) != 0;
      const int n_vid = wi.z * n_sub;            // key slabs in the pattern, then others and those of text (always 128 wide)
      const int n_kv = n_vid + (kEdge ? wi.x >> 8 : 0) + (kCluster && ((wi.w >> 26) & 1) ? 0 : g.n_ts);
      auto nk_j = [&](int j, int r) -> int { return j >= n_vid ? kSlabTokens : nk_at(r); };
      // which accumulators this item uses: both for a two-slab item, and for a split-KV item
      // with at least two key slabs (even slabs -> O_0, odd slabs -> O_1)
      const bool use_o1 = (nq > 1) || (split && n_kv > 1);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        if (i < nq) {
          const uint32_t itq = i == 0 ? it_q0 : it_q1;
          ok = mbar_wait_warp(bar(kBarQFull + i), itq & 1u, abort_flag, 0x200 + i);
          if (!ok) break;
        }
        if ((i == 0 || use_o1) && (!kShort || n_kv == 0)) {
          // the epilogue of the previous item must have drained O_i before it is overwritten
          const uint32_t ito = i == 0 ? it_o0 : it_o1;
          ok = mbar_wait_warp(bar(kBarOEmpty + i), (ito & 1u) ^ 1u, abort_flag, 0x202 + i);
          if (!ok) break;
        }
      }
      if (!ok) break;
      if (n_kv > 0 && split) {
        // ---- split-KV item: one query slab (Q buffer 0); key slab j feeds tile (j & 1).
        // Ring order (see the load warp): K_0, K_1, (V_0, K_2), (V_1, K_3), ..., V_{n-2}, V_{n-1}.
        int r0 = 0;   // residue of the slab whose scores are issued next
        for (int j = 0; ok && j < 2 && j < n_kv; ++j) {
          ok = mbar_wait_warp(bar(kBarPairFull + pair_i), pair_ph, abort_flag, 0x230);
          if (!ok) break;
          pair_adv();
          const uint32_t slot = slot_i;
          slot_i = slot_next(slot_i);
          tc_fence_after();
          if (elect_one()) {
            issue_qk(0, slot, nk_j(j, r0), j);
            tc_commit(bar(kBarSFull + j));
            tc_commit(bar(kBarSlotEmpty + slot));
            if (kShort && j + 1 == n_kv) tc_commit(bar(kBarQEmpty + 0));
          }
          __syncwarp();
          r0 = r_inc(r0);
        }
        int rj = 0;   // residue of slab j; r0 is that of slab j + 2 from here on
        for (int j = 0; ok && j < n_kv; ++j) {
          const int i = j & 1;
          const uint32_t cs = i == 0 ? cnt_s0 : cnt_s1;
          ok = mbar_wait2_warp(bar(kBarPairFull + pair_i), pair_ph, bar(kBarPHalf + i), cs & 1u, abort_flag, 0x231, 0x234 + i);
          if (!ok) break;
          pair_adv();
          const bool more = (j + 2 < n_kv);
          const uint32_t vslot = slot_i;
          const uint32_t kslot = slot_next(slot_i);
          slot_i = more ? slot_next(kslot) : kslot;
          const int nk_cur = nk_j(j, rj);
          rj = r_inc(rj);
          if (kShort && j < 2) {   // the previous item's O_i has been read
            ok = mbar_wait_warp(bar(kBarOEmpty + i), ((i == 0 ? it_o0 : it_o1) & 1u) ^ 1u, abort_flag, 0x202 + i);
            if (!ok) break;
          }
          tc_fence_after();
          if (elect_one()) issue_pv_half(i, vslot, 0, j > 1, nk_cur);
          ok = mbar_wait_warp(bar(kBarPReady + i), cs & 1u, abort_flag, 0x232 + i);
          if (!ok) break;
          if (i == 0) ++cnt_s0; else ++cnt_s1;
          tc_fence_after();
          if (elect_one()) {
            issue_pv_half(i, vslot, 1, true, nk_cur);
            tc_commit(bar(kBarSlotEmpty + vslot));
            if (more) {
              issue_qk(0, kslot, nk_j(j + 2, r0), i);
              r0 = r_inc(r0);
              tc_commit(bar(kBarSFull + i));
              tc_commit(bar(kBarSlotEmpty + kslot));
              if (kShort && j + 3 == n_kv) tc_commit(bar(kBarQEmpty + 0));
            } else {
              tc_commit(bar(kBarOFull + i));
            }
          }
          __syncwarp();
        }
        if (!ok) break;
      } else if (n_kv > 0) {
        // first key slab: both S tiles (a two-slab item: nq == 2)
        {
          ok = mbar_wait_warp(bar(kBarPairFull + pair_i), pair_ph, abort_flag, 0x210);
          if (!ok) break;
          pair_adv();
          const uint32_t slot = slot_i;
          slot_i = slot_next(slot_i);
          tc_fence_after();
          if (elect_one()) {
            issue_qk(0, slot, nk_j(0, 0), 0);
            tc_commit(bar(kBarSFull + 0));
            issue_qk(1, slot, nk_j(0, 0), 1);
            tc_commit(bar(kBarSFull + 1));
            tc_commit(bar(kBarSlotEmpty + slot));
            if (kShort && n_kv == 1) {
              tc_commit(bar(kBarQEmpty + 0));
              tc_commit(bar(kBarQEmpty + 1));
            }
          }
          __syncwarp();
        }
        // Per key slab j: P_0's first half -> P V (4 MMAs); all of P_0 -> the other 4 + next scores of
        // tile 0; the same for tile 1.  The barrier of V_j / K_{j+1} (loaded long before) is waited for
        // together with another wait, never on its own, and the bookkeeping for the next slab runs
        // while the queued MMAs drain.
        int rj = 0;
        bool pair_seen = false;   // V_j / K_{j+1} already known to have arrived
        for (int j = 0; ok && j < n_kv; ++j) {
          const int nk_cur = nk_j(j, rj);
          rj = r_inc(rj);
          const int nk_next = nk_j(j + 1, rj);
          const bool more = (j + 1 < n_kv);
          const uint32_t vslot = slot_i;
          const uint32_t kslot = slot_next(slot_i);
          slot_i = more ? slot_next(kslot) : kslot;
          if (pair_seen) ok = mbar_wait_warp(bar(kBarPHalf + 0), cnt_s0 & 1u, abort_flag, 0x224);
          else ok = mbar_wait2_warp(bar(kBarPairFull + pair_i), pair_ph, bar(kBarPHalf + 0), cnt_s0 & 1u, abort_flag, 0x211, 0x224);
          if (!ok) break;
          pair_adv();
          if (kShort && j == 0) {
            ok = mbar_wait2_warp(bar(kBarOEmpty + 0), (it_o0 & 1u) ^ 1u, bar(kBarOEmpty + 1), (it_o1 & 1u) ^ 1u, abort_flag, 0x202, 0x203);
            if (!ok) break;
          }
          tc_fence_after();
          if (elect_one()) issue_pv_half(0, vslot, 0, j > 0, nk_cur);
          bool half1_done = false;   // first half of P_1 already seen complete
          ok = mbar_wait_probe_warp(bar(kBarPReady + 0), cnt_s0 & 1u, bar(kBarPHalf + 1), cnt_s1 & 1u, abort_flag, 0x220,
                                    &half1_done);
          if (!ok) break;
          ++cnt_s0;
          tc_fence_after();
          if (elect_one()) {
            issue_pv_half(0, vslot, 1, true, nk_cur);
            if (more) {
              issue_qk(0, kslot, nk_next, 0);
              tc_commit(bar(kBarSFull + 0));
              if (kShort && j + 2 == n_kv) tc_commit(bar(kBarQEmpty + 0));
            } else {
              tc_commit(bar(kBarOFull + 0));
            }
          }
          __syncwarp();
          if (!half1_done) {
            ok = mbar_wait_warp(bar(kBarPHalf + 1), cnt_s1 & 1u, abort_flag, 0x225);
            if (!ok) break;
          }
          tc_fence_after();
          if (elect_one()) issue_pv_half(1, vslot, 0, j > 0, nk_cur);
          // all of P_1, and (one round trip) the loads of the next slab
          pair_seen = false;
          if (more) {
            ok = mbar_wait_probe_warp(bar(kBarPReady + 1), cnt_s1 & 1u, bar(kBarPairFull + pair_i), pair_ph, abort_flag, 0x221,
                                      &pair_seen);
          } else {
            ok = mbar_wait_warp(bar(kBarPReady + 1), cnt_s1 & 1u, abort_flag, 0x221);
          }
          if (!ok) break;
          ++cnt_s1;
          tc_fence_after();
          if (elect_one()) {
            issue_pv_half(1, vslot, 1, true, nk_cur);
            tc_commit(bar(kBarSlotEmpty + vslot));
            if (more) {
              issue_qk(1, kslot, nk_next, 1);
              tc_commit(bar(kBarSFull + 1));
              tc_commit(bar(kBarSlotEmpty + kslot));
              if (kShort && j + 2 == n_kv) tc_commit(bar(kBarQEmpty + 1));
            } else {
              tc_commit(bar(kBarOFull + 1));
            }
          }
          __syncwarp();
        }
        if (!ok) break;
      } else {
        if (elect_one()) {
          tc_commit(bar(kBarOFull + 0));
          if (nq > 1) tc_commit(bar(kBarOFull + 1));
          if (kShort) {
            tc_commit(bar(kBarQEmpty + 0));
            if (nq > 1) tc_commit(bar(kBarQEmpty + 1));
          }
        }
        __syncwarp();
      }
      ++it_q0;
      if (nq > 1) ++it_q1;
      ++it_o0;
      if (use_o1) ++it_o1;
    }
    // Every MMA issued so far must have completed before the TMEM allocation is released (after
    // a timeout some may still be in flight): one more commit, awaited with a bound of its own.
    if (elect_one()) {
      tc_commit(bar(kBarDrain));
      const unsigned long long t0 = globaltimer_ns();
      while (!mbar_try_wait(bar(kBarDrain), 0u)) {
        if (globaltimer_ns() - t0 > kTimeoutNs) break;
      }
    }
    __syncwarp();
  } else if constexpr (kCluster) {
    // ======================================================================= idle warps: tokens of the rows to merge
    // (the divisions take a microsecond, which the merge need not wait for)
    pdl_wait();
    if (tmem_ok && mbar_wait_warp(bar(kBarSchedFull), 0u, abort_flag, 0x402)) {
      const int4 wi = *reinterpret_cast<const int4*>(smem + kOffSched);
      const int nq = (wi.w >> 16) & 0xff, rpc = nq * 128 / (int)cluster_size(), r0 = (int)cluster_rank() * rpc;
      for (int i = (int)threadIdx.x - 64; i < rpc; i += 64)
        *reinterpret_cast<int*>(smem + kOffRowTok + (uint32_t)i * 4u) =
            (int)row_token<kBoxes>(prm, ((wi.w >> 25) & 1) != 0, wi.y, (wi.w & 0xffff) + ((r0 + i) >> 7), (r0 + i) & 127);
    }
    __syncwarp();
  }
  if constexpr (kCluster) cluster_sync_all();   // the barrier that the softmax warps meet at before they push
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsSoftmax));
    // ======================================================================= softmax warps
    const int qi = (warp - kFirstSoftmaxWarp) >> 2;   // tile (S_i, O_i) handled by this warpgroup
    const int row = (warp & 3) * 32 + lane;       // row of the slab == TMEM lane
    const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t tS = tmem + lane_addr + (uint32_t)qi * 128u;
    const uint32_t tO = tmem + lane_addr + 256u + (uint32_t)qi * 128u;
    uint32_t it_o0 = 0, it_o1 = 0, cnt_s = 0, kv_g = 0;
    uint32_t n_stage = 0;   // output slabs staged by this warpgroup so far
    uint32_t n_merge = 0;   // split-KV merges so far
    bool ok = true, met = false;   // met: cluster mode's first barrier passed
    const float neg_inf = __int_as_float(0xff800000);
    float2* xchg = reinterpret_cast<float2*>(smem + kOffXchg);
    const int n_sub = kEdge ? g.main_slabs : g.n_sub, n_last = kEdge ? g.main_last : g.n_last;
    if constexpr (!kDraws) pdl_wait();   // (see pdl_wait)

    for (uint32_t n = 0; ok; ++n) {
      WorkItem wi;
      if (!next_item(n, wi)) break;
      const int head = kEdge ? wi.x & 0xff : wi.x, qb = wi.y, sub0 = wi.w & 0xffff, nq = (wi.w >> 16) & 0xff;
      const bool split = ((wi.w >> 24) & 1) != 0;
      const bool textq = ((wi.w >> 25) & 1) != 0;
      const int n_vid = wi.z * n_sub;            // key slabs in the pattern, then others and those of text (always 128 wide)
      const int n_kv = n_vid + (kEdge ? wi.x >> 8 : 0) + (kCluster && ((wi.w >> 26) & 1) ? 0 : g.n_ts);
      const bool use_o1 = (nq > 1) || (split && n_kv > 1);
      const bool active = (qi == 0) || use_o1;
      float m_ref = neg_inf;  // running reference maximum, scaled log2 domain
      float l = 0.f;          // running sum of exp2(s - m_ref)
      float lr = 0.f;         // cluster mode: the same of the rounded probabilities
      if (active) {
        // key slabs of this tile: all of them, or every second one in a split-KV item
        const int j0 = split ? qi : 0, dj = split ? 2 : 1;
        const int r_last = n_sub - 1;
        int rj = (j0 > r_last) ? 0 : j0;   // j mod n_sub, carried along (no division in the loop)
        for (int j = j0; ok && j < n_kv; j += dj) {
          const int nk = (rj == r_last && j < n_vid) ? n_last : kSlabTokens;
          rj = (rj == r_last) ? 0 : rj + 1;
          if (dj == 2) rj = (rj == r_last) ? 0 : rj + 1;
          ok = mbar_wait_warp(bar(kBarSFull + qi), cnt_s & 1u, abort_flag, 0x300 + qi);
          if (!ok) break;
          ++cnt_s;
          tc_fence_after();
          // Read the slab's validity words first: shared memory is busy feeding the tensor core,
          // so the load's latency is overlapped with the TMEM loads that follow.
          const uint4 m = *reinterpret_cast<const uint4*>(meta + ((kv_g + (uint32_t)j) % kMetaRing) * 8);
          const uint32_t bh = bar(kBarPHalf + qi), br = bar(kBarPReady + qi);
          const bool first = (j == j0);
          if (nk == 128) softmax_slab<128, kCluster>(tS, tO, m, first, g.scale_log2, m_ref, l, lr, bh, br);
          else if (nk == 112) softmax_slab<112, kCluster>(tS, tO, m, first, g.scale_log2, m_ref, l, lr, bh, br);
          else if (nk == 96) softmax_slab<96, kCluster>(tS, tO, m, first, g.scale_log2, m_ref, l, lr, bh, br);
          else softmax_slab<64, kCluster>(tS, tO, m, first, g.scale_log2, m_ref, l, lr, bh, br);
        }
      }
      kv_g += (uint32_t)n_kv;
      if (!ok) break;
      const uint32_t par_o0 = it_o0 & 1u, par_o1 = it_o1 & 1u;
      ++it_o0;
      if (use_o1) ++it_o1;
      if constexpr (kCluster) {
        // Push this CTA's partial results to the CTAs that merge them.  The receiving Q buffers and K/V ring are idle
        // once every MMA of the cluster has completed: the first cluster barrier.  A share without keys is marked by
        // m = -inf.  The two tiles of a single query slab (even / odd key slabs) are merged here first: each warpgroup
        // takes 64 columns of both.
        ok = mbar_wait_warp(bar(kBarOFull + 0), par_o0, abort_flag, 0x310);
        if (!ok) break;
        if (use_o1) {
          ok = mbar_wait_warp(bar(kBarOFull + 1), par_o1, abort_flag, 0x311);
          if (!ok) break;
        }
        const bool has = active && n_kv > 0;
        cluster_sync_all();
        met = true;
        tc_fence_after();
        const float4 mine = has ? make_float4(m_ref, l, lr, 0.f) : make_float4(neg_inf, 0.f, 0.f, 0.f);
        if (split) {
          float4* tmp = reinterpret_cast<float4*>(smem + kOffPartTmp) + row;   // [2][128]
          tmp[qi * 128] = mine;
          mbar_arrive(bar(kBarStage + qi));
          ok = mbar_wait_warp(bar(kBarStage + (qi ^ 1)), 0u, abort_flag, 0x313);
          if (!ok) break;
          const float4 a = tmp[0], b = tmp[128];
          const float m_all = fmaxf(a.x, b.x);
          const float wa = (a.x == neg_inf) ? 0.f : fast_exp2(a.x - m_all), wb = (b.x == neg_inf) ? 0.f : fast_exp2(b.x - m_all);
          const Share sh = share_of_row(sbase, row, 1);
          if (qi == 0) st_cluster_f4(sh.ml, make_float4(m_all, wa * a.y + wb * b.y, wa * a.z + wb * b.z, 0.f));
          const uint32_t tO0 = tmem + lane_addr + 256u;
          if (n_kv > 0) {
#pragma unroll 1
            for (int c4 = 2 * qi; c4 < 2 * qi + 2; ++c4) {
              uint32_t o[32], o1[32];
              tc_ld32(tO0 + c4 * 32, o);
              tc_ld32(tO0 + 128u + c4 * 32, o1);
              tc_wait_ld();
#pragma unroll
              for (int c = 0; c < 32; ++c)   // (an accumulator without keys holds left-overs)
                o[c] = __float_as_uint((wa != 0.f ? wa * __uint_as_float(o[c]) : 0.f) + (wb != 0.f ? wb * __uint_as_float(o1[c]) : 0.f));
#pragma unroll
              for (int e = 0; e < 8; ++e)
                st_cluster_u4(sh.o + (uint32_t)(c4 * 8 + e) * sh.step, o + 4 * e);
            }
          }
        } else {
          const Share sh = share_of_row(sbase, qi * 128 + row, 2);
          st_cluster_f4(sh.ml, mine);
          if (n_kv > 0) {
#pragma unroll 1
            for (int c4 = 0; c4 < 4; ++c4) {
              uint32_t o[32];
              tc_ld32(tO + c4 * 32, o);
              tc_wait_ld();
#pragma unroll
              for (int e = 0; e < 8; ++e)
                st_cluster_u4(sh.o + (uint32_t)(c4 * 8 + e) * sh.step, o + 4 * e);
            }
          }
        }
        tc_fence_before();
        continue;
      }
      if (!active) continue;

      // ---- epilogue: out = O / l, lse = ln2 * (m_ref + log2 l).  In a split-KV item the two
      // partial results (even / odd key slabs) of each row are merged by warpgroup 0, which can
      // read both accumulators because they sit in the same TMEM lanes.
      float scale0 = 1.f, scale1 = 0.f;   // weights of O_0 and O_1 in the merged output
      if (split && qi == 1) {
        // hand (m, l) of the odd key slabs to warpgroup 0 (release / acquire through the barrier)
        if constexpr (kShort) {   // which may still be merging the previous item: it has read that one's by then
          ok = mbar_wait_warp(bar(kBarOEmpty + 1), par_o1 ^ 1u, abort_flag, 0x315);
          if (!ok) break;
        }
        xchg[row] = make_float2(m_ref, l);
        mbar_arrive(bar(kBarMerge));
        // This warpgroup has no use for O_1 itself, but must not fall a phase behind its barrier: a following two-slab
        // item without keys waits for nothing else, and would take the phase before last for its own.
        ok = mbar_wait_warp(bar(kBarOFull + 1), par_o1, abort_flag, 0x314);
        if (!ok) break;
        continue;
      }
      ok = mbar_wait_warp(bar(kBarOFull + qi), (qi == 0 ? par_o0 : par_o1), abort_flag, 0x310 + qi);
      if (!ok) break;
      if (split && use_o1) {
        ok = mbar_wait_warp(bar(kBarOFull + 1), par_o1, abort_flag, 0x312);
        if (!ok) break;
        ok = mbar_wait_warp(bar(kBarMerge), n_merge & 1u, abort_flag, 0x313);
        if (!ok) break;
        ++n_merge;
        const float2 other = xchg[row];
        const float m_all = fmaxf(m_ref, other.x);
        scale0 = (m_ref == neg_inf) ? 0.f : fast_exp2(m_ref - m_all);
        scale1 = (other.x == neg_inf) ? 0.f : fast_exp2(other.x - m_all);
        l = scale0 * l + scale1 * other.y;
        m_ref = m_all;
      }
      tc_fence_after();
      const bool empty = (n_kv == 0) || !(l > 0.f);
      const float inv = empty ? 0.f : 1.f / l;
      scale0 *= inv;
      scale1 *= inv;
      uint8_t* stage = smem + kOffQ + (uint32_t)qi * kSlabBytes;
      long long out_tok = -1;        // kShort: this row's token, and where its output goes
      uint4* out_row = nullptr;
      if constexpr (kShort) {
        out_tok = row_token<false>(prm, textq, qb, sub0 + qi, row);
        if (out_tok >= 0)
          out_row = reinterpret_cast<uint4*>(reinterpret_cast<uint16_t*>(prm.out) + (long long)head * prm.out_head + out_tok * prm.out_token);
      }
#pragma unroll
      for (int c4 = 0; c4 < 4; ++c4) {
        uint32_t o[32];
        if (n_kv > 0) {
          tc_ld32(tO + c4 * 32, o);
          tc_wait_ld();
        } else {
#pragma unroll
          for (int c = 0; c < 32; ++c) o[c] = 0u;
        }
        if (split && use_o1) {   // qi == 0 here: add the odd-slab accumulator
          uint32_t o1[32];
          tc_ld32(tO + 128u + c4 * 32, o1);
          tc_wait_ld();
#pragma unroll
          for (int c = 0; c < 32; ++c)
            o[c] = __float_as_uint(__uint_as_float(o[c]) * scale0 + __uint_as_float(o1[c]) * scale1);
        } else {
#pragma unroll
          for (int c = 0; c < 32; ++c) o[c] = __float_as_uint(__uint_as_float(o[c]) * scale0);
        }
        if constexpr (kShort) {
          if (out_row != nullptr && PSA_CHECKED(head >= 0 && head < g.n_heads && out_tok < g.Lt, 0xD17)) {
            uint32_t w[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) w[e] = empty ? 0u : pack_bf16(__uint_as_float(o[2 * e]), __uint_as_float(o[2 * e + 1]));
            if ((reinterpret_cast<uintptr_t>(out_row) & 31u) == 0u) {
              st_global_v8(out_row + c4 * 4, w);
              st_global_v8(out_row + c4 * 4 + 2, w + 8);
            } else {
#pragma unroll
              for (int e = 0; e < 4; ++e) out_row[c4 * 4 + e] = make_uint4(w[4 * e], w[4 * e + 1], w[4 * e + 2], w[4 * e + 3]);
            }
          }
          continue;
        }
#pragma unroll
        for (int c8 = 0; c8 < 4; ++c8) {
          uint32_t w[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float a = empty ? 0.f : __uint_as_float(o[c8 * 8 + 2 * e]);
            const float b = empty ? 0.f : __uint_as_float(o[c8 * 8 + 2 * e + 1]);
            w[e] = pack_bf16(a, b);
          }
          // 128-byte swizzle of the staging slab: 16-byte chunk index xor (row mod 8)
          const int col = c4 * 32 + c8 * 8;
          const int half = col >> 6, chunk = (col & 63) >> 3;
          uint8_t* dst = stage + half * kHalfBytes + row * 128 + ((chunk ^ (row & 7)) << 4);
          if (PSA_CHECKED(dst >= smem + kOffQ && dst + 16 <= smem + kOffQ + 2u * kSlabBytes &&
                          (reinterpret_cast<uintptr_t>(dst) & 15u) == 0u, 0xD12))
            *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
        }
      }
      tc_fence_before();
      mbar_arrive(bar(kBarOEmpty + qi));
      if (split && use_o1) mbar_arrive(bar(kBarOEmpty + 1));
      if constexpr (kShort) {
        if (out_tok >= 0 && PSA_CHECKED(head >= 0 && head < g.n_heads && out_tok < g.Lt, 0xD18))
          prm.lse[(long long)head * g.Lt + out_tok] = empty ? neg_inf : (m_ref + log2f(l)) * 0.6931471805599453f;
        continue;
      }
      int t0, h0, w0, et, eh, ew, ntok, last;
      const float lse_row = empty ? neg_inf : (m_ref + log2f(l)) * 0.6931471805599453f;
      if (textq) {   // text slab: rows are consecutive text tokens; they follow the L video tokens
        t0 = 0; h0 = 0; w0 = (sub0 + qi) * kSlabTokens; last = 2;
        if (w0 + row < g.n_text && PSA_CHECKED(head >= 0 && head < g.n_heads && w0 >= 0, 0xD10))
          prm.lse[(long long)head * g.Lt + g.L + w0 + row] = lse_row;
      } else if (kBoxes) {
        const long long tok = row_token<kBoxes>(prm, false, qb, sub0 + qi, row);
        if (tok >= 0 && PSA_CHECKED(head >= 0 && head < g.n_heads && tok < g.L, 0xD14)) prm.lse[(long long)head * g.Lt + tok] = lse_row;
        slab_origin(g, qb, 0, t0, h0, w0);
        last = 0;
      } else {
        slab_origin(g, qb, sub0 + qi, t0, h0, w0);
        slab_shape(g, sub0 + qi, et, eh, ew, ntok, last);
        const long long tok = row_token<false>(prm, false, qb, sub0 + qi, row);
        if (tok >= 0 && PSA_CHECKED(head >= 0 && head < g.n_heads && tok < g.L, 0xD11)) prm.lse[(long long)head * g.Lt + tok] = lse_row;
      }
      // Every thread's staged row is made visible to the TMA engine; the warpgroup's first warp
      // waits for all 128 rows (a bounded wait, like every other one) and stores the slab.
      fence_async_smem();
      mbar_arrive(bar(kBarStage + qi));
      if ((warp & 3) == 0) {
        ok = mbar_wait_warp(bar(kBarStage + qi), n_stage & 1u, abort_flag, 0x320 + qi);
        if (!ok) break;
        if (lane == 0) {
          const uint32_t src = sbase + kOffQ + (uint32_t)qi * kSlabBytes;
          if (PSA_CHECKED(w0 >= 0 && h0 >= 0 && t0 >= 0 && head >= 0 && head < g.n_heads && last >= 0 && last <= 2, 0xD13)) {
            auto box = [&](uint32_t row8, int map, int t, int h, int w) {
              tma_store_5d(tms.o + map, src + row8 * 1024u, 0, w, h, t, head);
              tma_store_5d(tms.o + map, src + row8 * 1024u + kHalfBytes, 64, w, h, t, head);
            };
            if (kBoxes && !textq) {
              if constexpr (kBoxes) {
                const EdgeClass& e = prm.cls[block_class(g, qb / g.Sp, qb % g.Sp)];
#pragma unroll 1
                for (int b = e.first_box[sub0 + qi]; b < e.first_box[sub0 + qi + 1]; ++b)
                  if (e.box[b].t != kZeros) box(e.box[b].row8, e.box[b].map, t0 + e.box[b].t, h0 + e.box[b].h, w0 + e.box[b].w);
              }
            } else {
              box(0u, last, t0, h0, w0);
            }
          }
          tma_store_commit();
          tma_store_wait_read();
          mbar_arrive(bar(kBarQEmpty + qi));
        }
        __syncwarp();
      }
      ++n_stage;
    }
    if constexpr (kCluster) {
      if (!met) cluster_sync_all();
    } else {
      if ((warp & 3) == 0 && lane == 0) tma_store_wait_all();
    }
  }

  // ------------------------------------------------------------------------- teardown
  tc_fence_before();
  __syncthreads();
  if constexpr (kCluster) {
    cluster_sync_all();   // every partial result has arrived; no CTA writes into another one any more
    // (not by the first warpgroup, which gave its registers away; nor in a CTA that gave up: its item and the rows' tokens
    // may never have been written to shared memory)
    if (warp >= kFirstSoftmaxWarp && *abort_flag == 0) merge_cluster(prm, smem);
  }
  if (threadIdx.x == 0 && *abort_flag != 0) {
    report_status(prm.ws_header, prm.call_id, PSA_ERR_TIMEOUT, *abort_flag);
  }
  if (warp == kWarpMma) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*tmem_slot), "r"(512) : "memory");
  }
}

// One warp waits, with the kernel's own bounded wait, on a barrier that nothing arrives on.
// The wait must give up after limit_ns, record PSA_ERR_TIMEOUT and return normally.
__global__ void wait_probe_kernel(int* ws_header, int call_id, unsigned long long limit_ns) {
  __shared__ __align__(8) unsigned long long probe_bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    mbar_init(smem_u32(&probe_bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  const bool ok = mbar_wait(smem_u32(&probe_bar), 0, &abort_flag, 0x7e57, limit_ns);
  __syncwarp();
  if (threadIdx.x == 0 && !ok) report_status(ws_header, call_id, PSA_ERR_TIMEOUT, abort_flag);
}

cudaError_t launch_wait_probe(int* ws_header, int call_id, unsigned long long limit_ns, cudaStream_t stream) {
  wait_probe_kernel<<<1, 32, 0, stream>>>(ws_header, call_id, limit_ns);
  return cudaGetLastError();
}

// ----------------------------------------------------------------------------- launchers
size_t plan_smem_bytes(const Geom& g) { return 4 * (size_t)(plan_key_words(g) + g.Tp + g.Sp); }

namespace {
// Launch that may start before its predecessor in the stream has finished (see pdl_wait), in clusters of `cluster`.
struct LaunchConfig {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  LaunchConfig(int grid, int threads, size_t smem, cudaStream_t stream, int cluster) {
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
  }
};
}  // namespace

// Once per device: shared-memory limits, and how many clusters of 2, 4 and 8 CTAs run at a time.
cudaError_t attn_init(int clusters[3]) {
#define PSA_ALL_GRIDS(mode) (const void*)attn_fwd_kernel<mode, kWhole>, (const void*)attn_fwd_kernel<mode, kPadded>, (const void*)attn_fwd_kernel<mode, kCut>
  const void* kernels[] = {PSA_ALL_GRIDS(kTicket), PSA_ALL_GRIDS(kDirect), PSA_ALL_GRIDS(kShared), PSA_ALL_GRIDS(kSharedDirect),
                           (const void*)attn_fwd_kernel<kTicketShort, kWhole>, (const void*)attn_fwd_kernel<kTicketShort, kPadded>};
#undef PSA_ALL_GRIDS
  cudaError_t e = cudaSuccess;
  for (const void* k : kernels)
    if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemAlloc)) != cudaSuccess) return e;
  for (int i = 0; i < 3; ++i) {
    LaunchConfig lc(2 << i, kThreads, kSmemAlloc, nullptr, 2 << i);
    if ((e = cudaOccupancyMaxActiveClusters(&clusters[i], attn_fwd_kernel<kSharedDirect, kCut>, &lc.cfg)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_plan(const PlanParams& hp, const Geom& g, int n_heads_here, int* ws_header,
                        psa_head_params* hp_dev, WorkItem* items, cudaStream_t stream) {
  const size_t smem = plan_smem_bytes(g);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(plan_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  LaunchConfig lc(n_heads_here, kPlanThreads, smem, stream, 1);
  return cudaLaunchKernelEx(&lc.cfg, plan_kernel, hp, g, ws_header, hp_dev, items);
}

template <int kMode>
cudaError_t launch_mode(const LaunchConfig& lc, Grid grid, const TensorMapsCut& tm, const HeadParamsArray& heads, const AttnParamsCut& prm) {
  if constexpr (kMode != kTicketShort) {   // (blocks of one slab are not cut)
    if (grid == kCut) return cudaLaunchKernelEx(&lc.cfg, attn_fwd_kernel<kMode, kCut>, tm, heads, prm);
  }
  TensorMaps plain;
  for (int i = 0; i < 3; ++i) {
    plain.q[i] = tm.q[i];
    plain.k[i] = tm.k[i];
    plain.v[i] = tm.v[i];
    plain.o[i] = tm.o[i];
  }
  const AttnParams& p = prm;
  if (grid == kPadded) return cudaLaunchKernelEx(&lc.cfg, attn_fwd_kernel<kMode, kPadded>, plain, heads, p);
  return cudaLaunchKernelEx(&lc.cfg, attn_fwd_kernel<kMode, kWhole>, plain, heads, p);
}

// heads: read by launches without planning only.  cluster: CTAs per work item, 1: whole items.  direct: all items run
// at once, nothing was planned.  *mode: how the launch hands out its items (empty_slabs: with kTicketEdge for kTicket).
cudaError_t launch_attn(const TensorMapsCut& tm, const HeadParamsArray& heads, const AttnParamsCut& prm, int n_sms, int cluster, Grid grid, bool direct,
                        bool short_items, bool empty_slabs, cudaStream_t stream, Mode* mode) {
  if (prm.n_items <= 0) return cudaSuccess;
  const int ctas = cluster > 1 || direct ? prm.n_items * cluster : (prm.n_items < n_sms ? prm.n_items : n_sms);
  LaunchConfig lc(ctas, kThreads, kSmemAlloc, stream, cluster);
  *mode = cluster > 1 ? (direct ? kSharedDirect : kShared) : (direct ? kDirect : (short_items ? kTicketShort : kTicket));
  const Mode kernel = *mode;
  if (kernel == kTicket && empty_slabs) *mode = kTicketEdge;
  switch (kernel) {
    case kDirect: return launch_mode<kDirect>(lc, grid, tm, heads, prm);
    case kShared: return launch_mode<kShared>(lc, grid, tm, heads, prm);
    case kSharedDirect: return launch_mode<kSharedDirect>(lc, grid, tm, heads, prm);
    case kTicketShort: return launch_mode<kTicketShort>(lc, grid, tm, heads, prm);
    default: return launch_mode<kTicket>(lc, grid, tm, heads, prm);
  }
}

}  // namespace psa

