// Inline-PTX wrappers for sm_100a: mbarrier, TMA tiled loads, tcgen05 (TMEM allocation, UMMA issue,
// commit, TMEM load/store, fences) and the shared-memory / instruction descriptors of tcgen05.mma.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

namespace rehyat {
namespace ptx {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(pred));
  return pred != 0;
}

// ----------------------------------------------------------------------------- dependent launch
// Programmatic dependent launch.  Every kernel of the library is launched as one that may start before its predecessor
// on the stream has ended (launch_kernel in rehyat_tc.cuh).  grid_dep_wait returns when that predecessor is complete and
// its writes are visible; grid_dep_launch lets the next kernel start once all CTAs of this grid have called it or ended.
// The rule that makes early work safe: a CTA calls grid_dep_launch only after its grid_dep_wait, so that a kernel that
// has started may use everything but the results of its direct predecessor, and no kernel ends before its predecessor.
// (Loads of a predecessor's results must not go through pointers the compiler may take for read-only.)
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ----------------------------------------------------------------------------- mbarrier
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// One arrival for the whole warp: every lane has finished (and fenced) its part, the warp synchronises, one lane
// arrives.  The barrier counts warps, not threads: thirty-two arrivals on one address are thirty-two serialised
// shared-memory atomics in front of whoever waits for the barrier.
__device__ __forceinline__ void mbar_arrive_warp(uint32_t bar, int lane) {
  __syncwarp();
  if (lane == 0) mbar_arrive(bar);
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// The same with a suspend-time hint: the thread may stay suspended for up to `hint_ns` before the instruction
// returns false (it still returns at once when the phase completes).  A role that waits long and often then
// leaves the issue slots of its scheduler to the warps that share it.
__device__ __forceinline__ bool mbar_try_wait_hint(uint32_t bar, uint32_t parity, uint32_t hint_ns) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(hint_ns)
      : "memory");
  return ok != 0;
}

// Bounded waits.  Every spin on an mbarrier in the tensor-core kernels goes through mbar_wait: it gives up after
// `limit_ns` of wall time, records `code` in the sticky status word status[0] and publishes the launch's epoch in
// status[1], so that the other CTAs of the same launch stop at their next slow wait instead of each waiting
// out the limit.  `abort_flag` makes the other roles of the CTA stop at once.  A role whose wait returns false
// must not issue anything further (no TMA load, no tcgen05.mma, no barrier arrival it owes): it leaves its loops
// and goes to the common exit of the kernel.  A later launch carries another epoch, so one timeout does not
// poison the launches that follow; the sticky bits stay until the host reads them.
// What a CTA waits for its grid's predecessor does not count: see grid_dep_wait_role.
// The context lives in the CTA's shared memory (set up by one thread before the first __syncthreads) and the
// waits take its shared-memory address, so that it costs the hot loops no registers.
struct WaitCtx {
  int abort_flag;                  // set by whichever thread of the CTA first gives up
  int epoch;                       // of this launch (never 0)
  unsigned long long limit_ns;     // wall-time limit of one wait, as it stands
  int* status;                     // global: [0] sticky error bits, [1] epoch of a launch in which a CTA gave up
  unsigned long long own_limit_ns; // what the host asked for
  unsigned long long start_ns;     // time of wait_ctx_init; 0 once the predecessor is known to have ended
};
// What a kernel receives from the host about waiting (and, for the one test that makes a wait run out, the
// switch that makes the TMA producer withhold every load so that nothing is ever in flight).
struct WaitArgs {
  int* status;
  int epoch;
  unsigned int limit_us;
  int withhold_loads;
};
__device__ __forceinline__ unsigned long long global_timer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void wait_ctx_init(WaitCtx* w, const WaitArgs& a) {
  w->abort_flag = 0;
  w->epoch = a.epoch;
  w->limit_ns = w->own_limit_ns = (unsigned long long)a.limit_us * 1000ull;
  w->start_ns = global_timer_ns();
  w->status = a.status;
}
// grid_dep_wait of a role whose fellows may be waiting on barriers behind it.  How long the predecessor takes says nothing
// about this grid, so the limit of their waits is lifted meanwhile, and is longer afterwards by what the CTA has been
// running: every wait that has begun has the whole of its limit left.  Warps that come together write about the same;
// whoever comes later finds the predecessor ended.
__device__ __forceinline__ void grid_dep_wait_role(uint32_t wctx) {
  constexpr uint32_t o_start = offsetof(WaitCtx, start_ns), o_limit = offsetof(WaitCtx, limit_ns), o_own = offsetof(WaitCtx, own_limit_ns);
  unsigned long long start, own;
  asm volatile("ld.volatile.shared.u64 %0, [%1];" : "=l"(start) : "r"(wctx + o_start));
  if (start != 0ull) asm volatile("st.volatile.shared.u64 [%0], %1;" ::"r"(wctx + o_limit), "l"(~0ull) : "memory");
  grid_dep_wait();
  if (start == 0ull) return;
  asm volatile("ld.volatile.shared.u64 %0, [%1];" : "=l"(own) : "r"(wctx + o_own));
  asm volatile("st.volatile.shared.u64 [%0], %1;" ::"r"(wctx + o_limit), "l"(own + (global_timer_ns() - start)) : "memory");
  asm volatile("st.volatile.shared.u64 [%0], %1;" ::"r"(wctx + o_start), "l"(0ull) : "memory");
}
__device__ __forceinline__ int wait_ctx_aborted(uint32_t wctx) {     // abort_flag is the first word of the context
  int f;
  asm volatile("ld.volatile.shared.b32 %0, [%1];" : "=r"(f) : "r"(wctx));
  return f;
}
// The slow path is on the critical path of the roles that wait often (a try_wait that fails returns within a few
// hundred cycles), so it polls the barrier and the CTA's abort flag only; the global epoch and the timer are
// looked at once per 1024 polls (some tens of microseconds).
__device__ __forceinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, uint32_t wctx, int code, uint32_t hint_ns) {
  const unsigned long long t0 = global_timer_ns();
  for (uint32_t i = 1;; ++i) {
    if (hint_ns ? mbar_try_wait_hint(bar, parity, hint_ns) : mbar_try_wait(bar, parity)) return true;
    if (wait_ctx_aborted(wctx)) return false;
    if ((i & 1023u) == 0u) {
      volatile WaitCtx* w = reinterpret_cast<volatile WaitCtx*>(__cvta_shared_to_generic(wctx));
      if (*reinterpret_cast<volatile int*>(w->status + 1) == w->epoch) { w->abort_flag = 1; return false; }
      if (global_timer_ns() - t0 > w->limit_ns) {
        w->abort_flag = 1;
        atomicOr(w->status, code);
        atomicExch(w->status + 1, w->epoch);
        return false;
      }
      __nanosleep(64);
    }
  }
}
// hint_ns: suspend-time hint of the polls after the first (0: none); the time limit is then looked at once per
// 1024 * hint_ns at most.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint32_t wctx, int code, uint32_t hint_ns = 0) {
  if (mbar_try_wait(bar, parity)) return true;
  return mbar_wait_slow(bar, parity, wctx, code, hint_ns);
}
// Wait of a role for what it has itself put in flight (its TMA loads, its tcgen05.mma through a commit) before
// the CTA may free TMEM and exit.  The abort flag does not cut it short; only the time limit does.
__device__ __forceinline__ bool mbar_wait_drain(uint32_t bar, uint32_t parity, uint32_t wctx) {
  const unsigned long long limit_ns = reinterpret_cast<volatile WaitCtx*>(__cvta_shared_to_generic(wctx))->own_limit_ns;
  const unsigned long long t0 = global_timer_ns();
  for (uint32_t i = 0;; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((i & 63u) == 63u) {
      if (global_timer_ns() - t0 > limit_ns) return false;
      __nanosleep(64);
    }
  }
}

// ----------------------------------------------------------------------------- TMA
__device__ __forceinline__ uint4 ld_global_v4(const void* p) {
  uint4 v;
  asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void prefetch_tensormap(const void* tmap) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(tmap)) : "memory");
}
// 4-D tiled load into this CTA's shared memory, completion counted in bytes on `bar`.
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const void* tmap, uint32_t bar, int x, int y, int z,
                                            int w) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(tmap)), "r"(bar), "r"(x), "r"(y), "r"(z), "r"(w)
      : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const void* tmap, uint32_t bar, int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(tmap)), "r"(bar), "r"(x), "r"(y), "r"(z)
      : "memory");
}
// Makes generic-proxy writes to shared memory visible to the async proxy (UMMA / TMA reads).
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// ----------------------------------------------------------------------------- TMEM
__device__ __forceinline__ void tmem_alloc(uint32_t smem_dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Arrives on `bar` once every tcgen05.mma issued so far by this thread has completed.
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// D[tmem] (+)= A[smem] * B[smem]
__device__ __forceinline__ void umma_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                        uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem]
__device__ __forceinline__ void umma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                        uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// The same for a role that a whole warp runs: all 32 lanes go through it (every decision a vote), the instructions execute in
// the one lane with `leader` set.  Addresses and descriptors then are values of the warp, which is how tcgen05.mma takes
// them: issued by a single thread an MMA costs 45 cycles whatever its size, this way 128 x 64 x 16 takes 32 and 128 x 32 x 16
// takes 16 (A in TMEM, 256 of them back to back).  For MMAs of N = 128, which take 64 either way, the single thread is the
// better form: its waits are shorter (24 heads of 64: window kernel 977 us, in this form 1,018; 320 x 480 layer 312 and 327).
struct Umma {
  uint32_t leader;
  __device__ __forceinline__ Umma() : leader(elect_one()) {}
  // arrives on `bar` once every tcgen05.mma issued so far has completed
  __device__ __forceinline__ void commit(uint32_t bar) const {
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "setp.ne.b32 q, %1, 0;\n\t"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
        ::"r"(bar), "r"(leader) : "memory");
  }
  // D[tmem] (+)= A[smem] * B[smem]
  __device__ __forceinline__ void ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) const {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "setp.ne.b32 q, %5, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(leader) : "memory");
  }
  // D[tmem] (+)= A[tmem] * B[smem]
  __device__ __forceinline__ void ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) const {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "setp.ne.b32 q, %5, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(leader) : "memory");
  }
};

// 32 lanes x 32 consecutive 32-bit columns: thread i of the warp gets lane (base lane + i).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
        "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
        "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
      : "memory");
}

// ----------------------------------------------------------------------------- descriptors
// Shared-memory matrix descriptor of tcgen05.mma (64 bits):
//   [0,14) start address >> 4, [16,30) leading-dimension byte offset >> 4,
//   [32,46) stride-dimension byte offset >> 4, [46,48) version = 1, [61,64) swizzle (2 = 128 B).
// The tiles here are what a TMA load with 128-byte swizzle of a [rows x 64 bf16] box leaves in
// shared memory: row r at r*128 bytes, its eight 16-byte chunks XOR-ed with (r mod 8).
//   K-major operand (the reduction dimension is the contiguous one): SBO = 1024 (8 rows), LBO unused.
//   MN-major operand (M or N contiguous, reduction along rows): SBO = 1024 (8 reduction rows),
//   LBO = distance between consecutive 64-element column blocks.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo_bytes >> 4) << 16) |
         ((uint64_t)(sbo_bytes >> 4) << 32) | (1ull << 46) | (2ull << 61);
}

// The descriptor of the same layout `byte_off` bytes further on (a multiple of 16; the tile stays below the 256 KB
// the address field spans): only the start-address field moves, so one 64-bit add replaces building it again.
// The thread that issues the MMAs is a single thread; what it computes between two MMAs is issue time.
__device__ __forceinline__ uint64_t smem_desc_advance(uint64_t desc, uint32_t byte_off) {
  return desc + (uint64_t)(byte_off >> 4);
}

// Instruction descriptor of tcgen05.mma kind::f16, bf16 x bf16 -> fp32:
//   [4,6) D format (1 = f32), [7,10) A format (1 = bf16), [10,13) B format (1 = bf16),
//   [15] A major (0 = K), [16] B major (0 = K, 1 = MN), [17,23) N >> 3, [24,29) M >> 4.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, int a_mn_major, int b_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn_major << 15) | ((uint32_t)b_mn_major << 16) |
         ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// Writes eight bf16 (one 16-byte chunk) of row `r`, columns [col, col+8) of a [rows x 128] bf16 tile
// kept as two [rows x 64] sub-tiles in the 128-byte-swizzled image described above.  `sub_bytes` is
// the size of one sub-tile (rows * 128).
__device__ __forceinline__ void st_tile_chunk_sw128(uint32_t tile, uint32_t sub_bytes, int r, int col, uint4 v) {
  const uint32_t addr = tile + (uint32_t)(col >> 6) * sub_bytes + (uint32_t)r * 128u +
                        ((((uint32_t)(col & 63) >> 3) ^ ((uint32_t)r & 7u)) << 4);
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

__device__ __forceinline__ uint32_t pack_bf16_relu(float lo, float hi) {   // max(.,0) then round, one instruction
  uint32_t r;
  asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

// ----------------------------------------------------------------------------- packed fp32 pairs
// sm_100 executes add/sub/mul/fma on two fp32 values held in one 64-bit register per instruction.
__device__ __forceinline__ uint64_t pk2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ uint64_t pk2u(uint32_t lo, uint32_t hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
  return r;
}
__device__ __forceinline__ void upk2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ void upk2u(uint64_t v, uint32_t& lo, uint32_t& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "l"(v));
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
__device__ __forceinline__ uint64_t add2_rm(uint64_t a, uint64_t b) {   // rounds towards -infinity
  uint64_t r;
  asm("add.rm.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// 2^x for a pair of values on the FMA pipe instead of the special-function unit: x = n + f with
// n = floor(x) taken by a round-down add of 1.5*2^23 (its low mantissa bits then hold n), 2^f by a
// cubic fitted to the minimax relative error on [0,1) (7.5e-5, below the bf16 rounding the result
// gets), and n added into the exponent field.  Arguments are clamped to >= -126.
__device__ __forceinline__ void ex2_poly2(float x0, float x1, float& y0, float& y1) {
  const uint64_t magic = pk2(12582912.f, 12582912.f);
  const uint64_t x = pk2(fmaxf(x0, -126.f), fmaxf(x1, -126.f));
  const uint64_t r = add2_rm(x, magic);
  const uint64_t f = sub2(x, sub2(r, magic));
  uint64_t p = fma2(pk2(0.078024156f, 0.078024156f), f, pk2(0.22606717f, 0.22606717f));
  p = fma2(p, f, pk2(0.6958338f, 0.6958338f));
  p = fma2(p, f, pk2(0.99992514f, 0.99992514f));
  uint32_t p0, p1, r0, r1;
  upk2u(p, p0, p1);
  upk2u(r, r0, r1);
  y0 = __uint_as_float(p0 + (r0 << 23));
  y1 = __uint_as_float(p1 + (r1 << 23));
}

template <int N>
__device__ __forceinline__ void setmaxnreg_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N>
__device__ __forceinline__ void setmaxnreg_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }

}  // namespace ptx
}  // namespace rehyat
