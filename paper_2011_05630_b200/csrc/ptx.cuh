// Thin wrappers over the sm_100a instructions the tensor-core kernels use: mbarrier, TMA tiled
// loads (no multicast), tcgen05 (tensor memory allocation, UMMA, commit, TMEM loads), and the
// shared-memory / instruction descriptors.  Every wait is bounded: after about a second it
// records where it gave up in a status word and the kernel winds down instead of spinning.
#pragma once
#include <cuda.h>
#include <cuda_fp16.h>
#include <stdint.h>

namespace dlf {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Optional timeline probe (compiled in only with -DDLF_TRACE): CTA 0 stores the global timer at
// a few points after the status word.
#ifdef DLF_TRACE
#define DLF_TRACE_POINT(status, slot) do { if (blockIdx.x == 0) reinterpret_cast<volatile unsigned long long*>(status)[4 + (slot)] = global_ns(); } while (0)
// per-phase cycle sums of CTA 0's thread 0: ACC adds the cycles since the last mark to a slot
#define DLF_TRACE_DECL(acc, mark) long long acc[8] = {0, 0, 0, 0, 0, 0, 0, 0}; long long mark = clock64()
#define DLF_TRACE_ACC(acc, slot, mark) do { const long long now_ = clock64(); acc[slot] += now_ - mark; mark = now_; } while (0)
#define DLF_TRACE_FLUSH(status, acc) do { if (blockIdx.x == 0 && threadIdx.x == 0) for (int i_ = 0; i_ < 8; i_++) reinterpret_cast<volatile long long*>(status)[4 + i_] = acc[i_]; } while (0)
// the same for any one thread of CTA 0, into slots base .. base + 7
#define DLF_TRACE_FLUSH_AT(status, acc, base) do { if (blockIdx.x == 0) for (int i_ = 0; i_ < 8; i_++) reinterpret_cast<volatile long long*>(status)[4 + (base) + i_] = acc[i_]; } while (0)
// ... the first n accounts only (the status block holds 28 slots)
#define DLF_TRACE_FLUSH_N(status, acc, base, n) do { if (blockIdx.x == 0) for (int i_ = 0; i_ < (n); i_++) reinterpret_cast<volatile long long*>(status)[4 + (base) + i_] = acc[i_]; } while (0)
#else
#define DLF_TRACE_POINT(status, slot) do { } while (0)
#define DLF_TRACE_DECL(acc, mark) do { } while (0)
#define DLF_TRACE_ACC(acc, slot, mark) do { } while (0)
#define DLF_TRACE_FLUSH(status, acc) do { } while (0)
#define DLF_TRACE_FLUSH_AT(status, acc, base) do { } while (0)
#define DLF_TRACE_FLUSH_N(status, acc, base, n) do { } while (0)
#endif

// ---- programmatic dependent launch -----------------------------------------------------------------
// A kernel launched with the programmatic-serialization attribute may start while its predecessor
// in the stream still runs: its CTAs are scheduled as SMs free up and run their set-up (barriers,
// TMEM allocation, bias staging); pdl_wait() then blocks until the predecessor grid has completed
// and its memory operations are visible.  Both are no-ops for a normal launch.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Maps and residuals are read with ordinary loads: the kernel before this one may still be writing them when this one's CTAs
// start, while __ldg (and a const __restrict__ argument) promises data that stays as it is for the kernel's whole life, and a
// load that promises that may be moved above pdl_wait().  __ldg is for weights and biases.
template <typename T>
__device__ __forceinline__ T ld_map(const T* p) { return *p; }

// ---- mbarrier ---------------------------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_inval(uint64_t* bar) {
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

constexpr uint64_t kWaitLimitNs = 1000000000ull;  // one second

// Waits for the phase with the given parity.  `abort_flag` is a CTA-shared word: once any wait
// of the CTA has given up, every later wait returns at once so that all roles drain.  On
// giving up, `code` (which wait, which CTA) is stored in the global status word.  HOT marks the waits on
// the critical path between two layers of a fused group: they keep polling much longer before they
// start to sleep.  (try_wait with a suspend-time hint instead of this loop was measured 1-3 % slower.)
// The polling loop is a function of its own (one copy per kernel instead of one per wait site: a kernel has dozens of
// waits, and their inlined loops made up a large part of its code); the first poll, which usually succeeds, stays inline.
template <bool HOT>
__device__ __noinline__ bool mbar_wait_slow(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* status, int code,
                                            uint64_t limit_ns) {
    uint64_t t0 = 0;   // the global timer is read only once a wait has lasted a while
    uint32_t spins = 0;
    while (true) {
        if (mbar_try_wait(bar, parity)) return true;
        // back off: a spinning single-thread role shares its scheduler with the warps doing the work
        if (spins > (HOT ? 2048u : 4u)) __nanosleep(spins > 64 && !HOT ? 128 : 32);
        if ((++spins & 63u) == 0) {
            if (*abort_flag) return false;
            const uint64_t now = global_ns();
            if (t0 == 0) t0 = now;
            if (now - t0 > limit_ns) {
                *abort_flag = 1;
                atomicCAS(status, 0, code);
                return false;
            }
        }
    }
}
template <bool HOT = false>
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                          int* status, int code, uint64_t limit_ns = kWaitLimitNs) {
    if (mbar_try_wait(bar, parity)) return true;
    return mbar_wait_slow<HOT>(bar, parity, abort_flag, status, code, limit_ns);
}

// Warp-wide form: every lane polls (a whole warp stays on the issue path so that the addresses it
// computes are warp-uniform values); the result is voted so that the warp leaves a wait together.
template <bool HOT = false>
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                               int* status, int code, uint64_t limit_ns = kWaitLimitNs) {
    const bool ok = mbar_wait<HOT>(bar, parity, abort_flag, status, code, limit_ns);
    return __all_sync(0xffffffffu, ok);
}

// True in exactly one lane of a converged warp (the same lane every time).
__device__ __forceinline__ bool elect_one() {
    uint32_t pred;
    asm volatile(
        "{\n\t.reg .b32 rx;\n\t.reg .pred px;\n\t"
        "elect.sync rx|px, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, px;\n\t}"
        : "=r"(pred));
    return pred != 0;
}

__device__ __forceinline__ void fence_barrier_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// Makes generic-proxy writes to shared memory visible to the async proxy (TMA, UMMA operand reads).
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// ---- TMA (tiled mode, one CTA, no multicast) ------------------------------------------------------
__device__ __forceinline__ void tma_prefetch_desc(const CUtensorMap* m) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* m, uint64_t* bar, int c0, int c1,
                                            int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}
__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* m, uint64_t* bar, int c0, int c1,
                                            int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2),
        "r"(c3)
        : "memory");
}

__device__ __forceinline__ void tma_load_5d(void* dst, const CUtensorMap* m, uint64_t* bar, int c0, int c1,
                                            int c2, int c3, int c4) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, %7}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2),
        "r"(c3), "r"(c4)
        : "memory");
}

// ---- clusters ----------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// The address of the same shared-memory location in another CTA of the cluster.
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// Hardware barrier of the cluster: every thread arrives and waits once per phase.  (Bounded: what comes before a thread's
// arrival is made of bounded waits.)
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// Arrives on a barrier of any CTA of the cluster (an address from mapa()).  The arrival publishes nothing but itself: what it
// stands for is an accumulator that has been read (tcgen05.wait::ld), and a release at cluster scope would wait for every store
// to shared memory before it (1100 clocks per tile of a CTA pair's epilogue).
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t addr) {
    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
// Loads of a CTA pair: into this CTA's shared memory, completing on a barrier of either CTA (an address from mapa()).
__device__ __forceinline__ void tma_load_3d_pair(void* dst, const CUtensorMap* m, uint32_t bar, int c0, int c1, int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}
__device__ __forceinline__ void tma_load_4d_pair(void* dst, const CUtensorMap* m, uint32_t bar, int c0, int c1, int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}
__device__ __forceinline__ void tma_load_5d_pair(void* dst, const CUtensorMap* m, uint32_t bar, int c0, int c1, int c2, int c3, int c4) {
    asm volatile(
        "cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, %7}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
        : "memory");
}

// ---- tcgen05: tensor memory ---------------------------------------------------------------------
// Allocation is warp-wide; the base address is written to shared memory.
__device__ __forceinline__ void tmem_alloc(uint32_t* smem_dst, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_dst)),
                 "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// The same for a CTA pair (one warp of either CTA; both get the same columns).
__device__ __forceinline__ void tmem_alloc_pair(uint32_t* smem_dst, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_dst)), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before_sync() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after_sync() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Shared-memory matrix descriptor, K-major operand, 128-byte swizzle: rows of 64 fp16 (128 bytes),
// eight rows per 1024-byte swizzle atom, atoms of consecutive row groups 1024 bytes apart.
// The swizzle is a function of the absolute shared-memory address (bits 7..9 select the XOR of
// bits 4..6), so a start address on any 128-byte row of a 1024-byte-aligned buffer is valid with
// base-offset field left at zero.  umma_desc_lo() and kDescHiSw128 below are its two words: start address in 16-byte units and a
// leading offset of 1 (unused); 1024 bytes between row groups, the descriptor version and the swizzle.
// Instruction descriptor: fp16 x fp16 -> fp32, both operands K-major, M = 128, given N.
__host__ __device__ constexpr uint32_t umma_idesc_f16(int n) {
    return (1u << 4) | (static_cast<uint32_t>(n >> 3) << 17) | (static_cast<uint32_t>(128 >> 4) << 24);
}
// A CTA pair's product: M = 256 rows, 128 of them (operand A and accumulator) in either CTA; N columns, half of operand B's
// rows in either CTA; the descriptors' addresses hold in both.
__host__ __device__ constexpr uint32_t umma_idesc_f16_pair(int n) {
    return (1u << 4) | (static_cast<uint32_t>(n >> 3) << 17) | (static_cast<uint32_t>(256 >> 4) << 24);
}
// The barrier at this offset in both CTAs of the pair gets one arrival when every UMMA issued so far has completed.
__device__ __forceinline__ void umma_commit_pair(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(smem_u32(bar)),
                 "h"(static_cast<uint16_t>(3))
                 : "memory");
}
// D[tmem] (+)= A[smem] * B[smem]; issued by one thread.
__device__ __forceinline__ void umma_f16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// Measured on B200 (M = 128, K = 16, fp16): an issue loop run by ONE thread (`if (lane == 0)`) spends
// about 72 cycles per UMMA whatever N is, because every descriptor is a per-thread value that has to
// be moved into uniform registers; the same loop run by the whole warp with warp-uniform descriptors
// and the UMMA group under elect_one() reaches the hardware's rates: 48 cycles at N = 64 (operand
// reads from shared memory), N / 2 cycles from N = 128 up.  Descriptors differ only in the 14-bit
// start-address field, so stepping one is a 64-bit add of (bytes >> 4).
//
// Lean 32-bit form (older issue loops): the descriptors' upper words are constants, only the
// start-address field of the lower word changes from one MMA to the next.
constexpr uint32_t kDescHiSw128 = (1024u >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t umma_desc_lo(uint32_t saddr) { return ((saddr & 0x3FFFFu) >> 4) | (1u << 16); }
// An operand that lies along M instead (rows of 64 consecutive M values of ONE k, eight k to a 1024-byte swizzle atom, atoms of
// further k right behind, further 64 values of M `lbo` bytes away): its low descriptor word, and the instruction descriptor's
// bit that says so of operand A.
constexpr uint32_t kIdescAmn = 1u << 15;
__device__ __forceinline__ uint32_t umma_desc_mn_lo(uint32_t saddr, int lbo) { return ((saddr & 0x3FFFFu) >> 4) | (static_cast<uint32_t>(lbo >> 4) << 16); }
__device__ __forceinline__ void umma_f16_lo(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t idesc,
                                            uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "mov.b64 da, {%1, %2};\n\t"
        "mov.b64 db, {%3, %6};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(idesc), "r"(accumulate), "r"(kDescHiSw128)
        : "memory");
}

// The four K = 16 steps of one 64-channel chunk in a single statement: A and B advance by 32 bytes (2 units) per step, both
// descriptors share the constant high word.  The first step accumulates only if `accumulate` is non-zero.
__device__ __forceinline__ void umma_f16_x4(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t.reg .b32 ta, tb;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "mov.b64 da, {%1, %5};\n\tmov.b64 db, {%2, %5};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n\t"
        "setp.eq.b32 p, %3, %3;\n\t"
        "add.u32 ta, %1, 2;\n\tadd.u32 tb, %2, 2;\n\tmov.b64 da, {ta, %5};\n\tmov.b64 db, {tb, %5};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n\t"
        "add.u32 ta, %1, 4;\n\tadd.u32 tb, %2, 4;\n\tmov.b64 da, {ta, %5};\n\tmov.b64 db, {tb, %5};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n\t"
        "add.u32 ta, %1, 6;\n\tadd.u32 tb, %2, 6;\n\tmov.b64 da, {ta, %5};\n\tmov.b64 db, {tb, %5};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(idesc), "r"(accumulate), "r"(kDescHiSw128)
        : "memory");
}

// KS K = 16 steps (1 to 4) of one 64-channel chunk, and the same for the three taps of a kernel row of a 3x3 layer (A one row
// = 8 units further per tap, B one slab of `w_tap16` units), in a single statement each: statements of their own cost the
// issuing thread about 200 clocks per UMMA in a loop over taps, members of one statement 66 (two 16 -> 16 3x3 layers on one
// 32x32 image: 9.2 -> 7.5 us as one kernel).
#define DLF_UMMA_STEP(CG, AO, KO)                                                                                                    \
    "add.u32 ta, %1, " #AO ";\n\tadd.u32 tb, tc, " #KO ";\n\tmov.b64 da, {ta, %5};\n\tmov.b64 db, {tb, %5};\n\t"                     \
    "tcgen05.mma.cta_group::" #CG ".kind::f16 [%0], da, db, %3, p;\n\t"
#define DLF_UMMA_FIRST(CG)                                                                                                           \
    "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t.reg .b32 ta, tb, tc;\n\tsetp.ne.b32 p, %4, 0;\n\tmov.b32 tc, %2;\n\t"              \
    DLF_UMMA_STEP(CG, 0, 0) "setp.eq.b32 p, %3, %3;\n\t"
#define DLF_UMMA_NEXT_TAP "add.u32 tc, tc, %6;\n\t"
#define DLF_UMMA_OPS                                                                                                                 \
    "}" ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(idesc), "r"(accumulate), "r"(kDescHiSw128), "r"(w_tap16) : "memory"
template <int KS>
__device__ __forceinline__ void umma_f16_row3(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t w_tap16, uint32_t idesc, uint32_t accumulate) {
    if (KS == 1)
        asm volatile(DLF_UMMA_FIRST(1) DLF_UMMA_NEXT_TAP DLF_UMMA_STEP(1, 8, 0) DLF_UMMA_NEXT_TAP DLF_UMMA_STEP(1, 16, 0) DLF_UMMA_OPS);
    if (KS == 2)
        asm volatile(DLF_UMMA_FIRST(1) DLF_UMMA_STEP(1, 2, 2) DLF_UMMA_NEXT_TAP DLF_UMMA_STEP(1, 8, 0) DLF_UMMA_STEP(1, 10, 2) DLF_UMMA_NEXT_TAP
                     DLF_UMMA_STEP(1, 16, 0) DLF_UMMA_STEP(1, 18, 2) DLF_UMMA_OPS);
    if (KS == 3)
        asm volatile(DLF_UMMA_FIRST(1) DLF_UMMA_STEP(1, 2, 2) DLF_UMMA_STEP(1, 4, 4) DLF_UMMA_NEXT_TAP DLF_UMMA_STEP(1, 8, 0) DLF_UMMA_STEP(1, 10, 2)
                     DLF_UMMA_STEP(1, 12, 4) DLF_UMMA_NEXT_TAP DLF_UMMA_STEP(1, 16, 0) DLF_UMMA_STEP(1, 18, 2) DLF_UMMA_STEP(1, 20, 4) DLF_UMMA_OPS);
}
template <int KS, bool PAIR = false>
__device__ __forceinline__ void umma_f16_steps(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, uint32_t accumulate) {
    const uint32_t w_tap16 = 0u;
    if (!PAIR) {
        if (KS == 1) asm volatile(DLF_UMMA_FIRST(1) DLF_UMMA_OPS);
        if (KS == 2) asm volatile(DLF_UMMA_FIRST(1) DLF_UMMA_STEP(1, 2, 2) DLF_UMMA_OPS);
        if (KS == 3) asm volatile(DLF_UMMA_FIRST(1) DLF_UMMA_STEP(1, 2, 2) DLF_UMMA_STEP(1, 4, 4) DLF_UMMA_OPS);
        if (KS == 4) asm volatile(DLF_UMMA_FIRST(1) DLF_UMMA_STEP(1, 2, 2) DLF_UMMA_STEP(1, 4, 4) DLF_UMMA_STEP(1, 6, 6) DLF_UMMA_OPS);
    } else {   // of a CTA pair
        if (KS == 1) asm volatile(DLF_UMMA_FIRST(2) DLF_UMMA_OPS);
        if (KS == 2) asm volatile(DLF_UMMA_FIRST(2) DLF_UMMA_STEP(2, 2, 2) DLF_UMMA_OPS);
        if (KS == 3) asm volatile(DLF_UMMA_FIRST(2) DLF_UMMA_STEP(2, 2, 2) DLF_UMMA_STEP(2, 4, 4) DLF_UMMA_OPS);
        if (KS == 4) asm volatile(DLF_UMMA_FIRST(2) DLF_UMMA_STEP(2, 2, 2) DLF_UMMA_STEP(2, 4, 4) DLF_UMMA_STEP(2, 6, 6) DLF_UMMA_OPS);
    }
}
// ... with operand A along M: 16 k are two 1024-byte atoms, 128 units a step.
template <int KS>
__device__ __forceinline__ void umma_f16_mn_steps(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, uint32_t accumulate) {
    const uint32_t w_tap16 = 0u;
    if (KS == 1) asm volatile(DLF_UMMA_FIRST(1) DLF_UMMA_OPS);
    if (KS == 2) asm volatile(DLF_UMMA_FIRST(1) DLF_UMMA_STEP(1, 128, 2) DLF_UMMA_OPS);
    if (KS == 3) asm volatile(DLF_UMMA_FIRST(1) DLF_UMMA_STEP(1, 128, 2) DLF_UMMA_STEP(1, 256, 4) DLF_UMMA_OPS);
    if (KS == 4) asm volatile(DLF_UMMA_FIRST(1) DLF_UMMA_STEP(1, 128, 2) DLF_UMMA_STEP(1, 256, 4) DLF_UMMA_STEP(1, 384, 6) DLF_UMMA_OPS);
}
#undef DLF_UMMA_STEP
#undef DLF_UMMA_FIRST
#undef DLF_UMMA_NEXT_TAP
#undef DLF_UMMA_OPS

// ---- TMA store (shared -> global, tiled, clipped at the tensor's edges) ---------------------------
__device__ __forceinline__ void tma_store_4d(const CUtensorMap* m, const void* src, int c0, int c1, int c2, int c3) {
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4, %5}], [%1];"
                 ::"l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(src)), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
                 : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// Waits until the committed stores have finished READING shared memory (the buffer may be reused).
__device__ __forceinline__ void tma_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
// ... all but the newest `pending` (0..3) committed stores of this thread have finished reading.
__device__ __forceinline__ void tma_store_wait_read_n(int pending) {
    if (pending <= 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    else if (pending == 1) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
    else if (pending == 2) asm volatile("cp.async.bulk.wait_group.read 2;" ::: "memory");
    else asm volatile("cp.async.bulk.wait_group.read 3;" ::: "memory");
}
__device__ __forceinline__ void tma_store_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// The barrier gets one arrival when every UMMA issued so far by this thread has completed.
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}
// 32 lanes x 16 consecutive fp32 columns: thread t of the warp gets lane (taddr.lane + t).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; i++) v[i] = __uint_as_float(r[i]);
}

// Split form (see tmem_ld32_issue): the load is issued into raw registers and waited for later.
__device__ __forceinline__ void tmem_ld16_issue(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld16_wait(uint32_t (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]) : : "memory");
}

// Two 16-column loads in flight before one wait: 32 consecutive fp32 columns of the thread's lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; i++) v[i] = __uint_as_float(r[i]);
}

// Split form: the load is issued into raw registers and waited for later, so that the next chunk's
// load is in flight while this chunk is being worked on.  The wait names the registers as in/out
// operands: nothing that reads them can be scheduled ahead of it.
__device__ __forceinline__ void tmem_ld32_issue(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld32_wait(uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31]) : : "memory");
}

// acc + x * w with fp16 factors (bit patterns): exact product, one fp32 rounding, no conversions.  (Both factors in registers
// of their own: packed pairs unpacked at every use were measured a fifth slower in the depthwise kernel.)
__device__ __forceinline__ float fma_f32_f16(unsigned short x, unsigned short w, float acc) {
    asm("fma.rn.f32.f16 %0, %1, %2, %0;" : "+f"(acc) : "h"(x), "h"(w));
    return acc;
}
__device__ __forceinline__ void unpack_h2(uint32_t v, unsigned short& lo, unsigned short& hi) {
    asm("mov.b32 {%0, %1}, %2;" : "=h"(lo), "=h"(hi) : "r"(v));
}

__device__ __forceinline__ float apply_act(float v, int act) {
    if (act >= 1) v = fmaxf(v, 0.0f);
    if (act == 2) v = fminf(v, 6.0f);
    return v;
}

// Two values rounded to fp16, then clamped to [lo, hi] as a pair.  Rounding is monotone and the bounds used (0 and 6) are
// fp16 values, so clamping after the rounding gives the same bits as clamping before it - at one instruction per bound and
// PAIR instead of one per bound and value.  An open bound is a NaN: min and max then return their other operand, whatever it
// is.  A NaN stays one without an activation, and is 0 behind ReLU and ReLU6 (max(NaN, 0)), in every kernel (round_act).
__device__ __forceinline__ __half2 act_lo(int act) { return __float2half2_rn(act >= 1 ? 0.0f : __int_as_float(0x7fffffff)); }
__device__ __forceinline__ __half2 act_hi(int act) { return __float2half2_rn(act == 2 ? 6.0f : __int_as_float(0x7fffffff)); }
__device__ __forceinline__ uint32_t pack_half2_clamp(float a, float b, __half2 lo, __half2 hi) {
    const __half2 h = __hmin2(__hmax2(__floats2half2_rn(a, b), lo), hi);
    return *reinterpret_cast<const uint32_t*>(&h);
}
// Epilogue arithmetic in few instructions (it bounds the memory-bound layers): two fp32 additions at once, and a pair rounded
// to fp16 with its activation (none, ReLU, ReLU6).  (The conversion's own ReLU would save the max - ResNet-50 b32 590.7 us instead
// of 594.7, MobileNetV2 b64 543.8 instead of 553.1 - but it keeps a NaN, which ReLU6's min then turns into 6.)
__device__ __forceinline__ float2 add_f2(uint32_t a0, uint32_t a1, uint64_t b) {
    uint64_t r;
    float2 f;
    asm("{\n\t.reg .b64 t;\n\tmov.b64 t, {%1, %2};\n\tadd.rn.f32x2 %0, t, %3;\n\t}" : "=l"(r) : "r"(a0), "r"(a1), "l"(b));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(r));
    return f;
}
template <int ACT>
__device__ __forceinline__ uint32_t round_act(float a, float b) {
    __half2 h = __floats2half2_rn(a, b);
    if (ACT >= 1) h = __hmax2(h, __float2half2_rn(0.0f));
    if (ACT == 2) h = __hmin2(h, __float2half2_rn(6.0f));
    return *reinterpret_cast<const uint32_t*>(&h);
}

// 16 bytes into the shared memory of a CTA of the cluster, counted by a barrier of that CTA (both addresses from mapa()).
__device__ __forceinline__ void st_async_v4(uint32_t addr, float a, float b, float c, float d, uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(addr), "f"(a), "f"(b), "f"(c), "f"(d), "r"(bar) : "memory");
}
// 8 sums, their biases and 8 residual values to 8 rounded outputs.
__device__ __forceinline__ uint4 finish8(const float* v, const float* bias, const uint4& res, __half2 lo, __half2 hi) {
    const float4 c0 = *reinterpret_cast<const float4*>(bias), c1 = *reinterpret_cast<const float4*>(bias + 4);
    const __half2* rh = reinterpret_cast<const __half2*>(&res);
    const float2 f0 = __half22float2(rh[0]), f1 = __half22float2(rh[1]), f2 = __half22float2(rh[2]), f3 = __half22float2(rh[3]);
    uint4 o;
    o.x = pack_half2_clamp(v[0] + c0.x + f0.x, v[1] + c0.y + f0.y, lo, hi);
    o.y = pack_half2_clamp(v[2] + c0.z + f1.x, v[3] + c0.w + f1.y, lo, hi);
    o.z = pack_half2_clamp(v[4] + c1.x + f2.x, v[5] + c1.y + f2.y, lo, hi);
    o.w = pack_half2_clamp(v[6] + c1.z + f3.x, v[7] + c1.w + f3.y, lo, hi);
    return o;
}

}  // namespace dlf
