// sm_100a primitives used by the tensor-core kernels: mbarriers with bounded waits, TMA
// tile loads, tcgen05 (tensor memory, UMMA descriptors, MMA issue, commit, ld/st).
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cuda.h>
#include <stdint.h>

namespace psk {
namespace tc {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Which warp this is, as a value the compiler knows to be the same in all 32 lanes.
__device__ __forceinline__ int warp_index() { return __shfl_sync(0xffffffffu, (int)threadIdx.x / 32, 0); }
// True in one lane of a warp, the same one every time (all 32 have to come here; after a wait on a barrier they need not
// come together, and two groups of lanes that elect one each would issue everything twice: hence the __syncwarp).  Work for a single thread
// that issues MMAs goes behind `warp_index() == w && elect_one()`, not behind a comparison of threadIdx.x: only then
// does the compiler keep an MMA's descriptors in uniform registers.  Measured, one thread issuing 32 in a row with A
// in tensor memory: 48 cycles each up to N = 96 behind a thread index; elected N = 16: 11, 32: 18, 64: 31, 80: 37, 96: 45 (with A in
// shared memory the operand's way bounds them: 40, 40, 47, 52, 55).  Forward of 12 heads x 16 512, r = 32: 179 -> 155 us;
// training, 48 heads x 16 384, r = 64: 5362 -> 4650, 384 heads x 32 768, r = 32: 21 789 -> 20 791.
__device__ __forceinline__ bool elect_one() {
    uint32_t e;
    __syncwarp();
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.b32 %0, 1, 0, p;\n\t}" : "=r"(e));
    return e != 0;
}

// ---------------------------------------------------------------------------
// mbarrier
// ---------------------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// A waiting thread is suspended by the hardware for up to this long per poll instead of spinning:
// spinning warps take issue slots from the warps that do the work.
constexpr uint32_t kSuspendHintNs = 20000;
__device__ __forceinline__ bool mbar_try_wait_addr(uint32_t bar_addr, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar_addr), "r"(parity), "r"(kSuspendHintNs)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    return mbar_try_wait_addr(smem_u32(bar), parity);
}
// Bounded waits.  A wait that is not satisfied at once goes to an out-of-line loop that gives up
// when kWaitLimitNs of wall time (%globaltimer) have passed.  The loser records `code` in *status
// (global), raises the CTA's give-up flag (shared memory) and returns false.  From then on every
// wait of that CTA that is not satisfied at once returns false without waiting, so the CTA runs
// through the rest of its work at full speed: the first lost signal costs one limit, nothing after
// it costs anything.  Kernels therefore never have to leave a loop early because a wait failed --
// which matters wherever a loop contains a barrier that counts its participants.
// Every kernel that waits calls cta_giveup_init() from one thread before its first block-wide
// barrier, may read cta_gave_up() after its last one to skip its global stores, and calls cta_teardown() after that one,
// before it gives tensor memory back.
constexpr uint64_t kWaitLimitNs = 1000000000ull;
__device__ __forceinline__ uint64_t globaltimer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ volatile int* cta_giveup_flag() {
    __shared__ int flag;
    return &flag;
}
__device__ __forceinline__ void cta_giveup_init() { *cta_giveup_flag() = 0; }
__device__ __forceinline__ bool cta_gave_up() { return *cta_giveup_flag() != 0; }
__device__ __forceinline__ bool mbar_test_addr(uint32_t bar_addr, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar_addr), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) { return mbar_test_addr(smem_u32(bar), parity); }
// (the flag of the first to give up also says which barrier it was and which phase)
__device__ __forceinline__ bool wait_failed(int* status, int code, uint32_t bar_addr, uint32_t parity) {
    atomicCAS(const_cast<int*>(cta_giveup_flag()), 0, (int)(bar_addr << 2 | (parity & 1) << 1 | 1));
    if (status != nullptr) atomicCAS(status, 0, code);
    return false;
}
// The bounded loop is one out-of-line copy: waits are everywhere in straight-line kernel code, and
// instruction fetch is what those kernels run out of first.  Nothing precedes the first poll
// (nearly every wait ends inside it, and whatever came before it would delay the waiter's
// wake-up); the flag is read after a poll that came back without the barrier, the clock every
// 1024 such polls.
static __device__ __noinline__ bool mbar_wait_slow(uint32_t bar_addr, uint32_t parity, int* status, int code,
                                                   uint64_t limit_ns) {
    uint64_t t0 = 0;
#pragma unroll 1
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 1024; ++i) {
            if (mbar_try_wait_addr(bar_addr, parity)) return true;
            if (cta_gave_up()) return false;
        }
        const uint64_t now = globaltimer_ns();
        if (t0 == 0) t0 = now;
        else if (now - t0 > limit_ns) break;
    }
    return wait_failed(status, code, bar_addr, parity);
}
// Bounded wait by polling only (no suspension): for a lone issuing thread, whose wake-up latency
// is on the critical path of everything it feeds and whose polling costs no one else issue slots.
// Flag every 64 polls, clock every 4096.
static __device__ __noinline__ bool mbar_spin_slow(uint32_t bar_addr, uint32_t parity, int* status, int code,
                                                   uint64_t limit_ns) {
    uint64_t t0 = 0;
#pragma unroll 1
    for (;;) {
#pragma unroll 1
        for (int g = 0; g < 64; ++g) {
#pragma unroll 1
            for (int i = 0; i < 64; ++i) {
                if (mbar_test_addr(bar_addr, parity)) return true;
            }
            if (cta_gave_up()) return false;
        }
        const uint64_t now = globaltimer_ns();
        if (t0 == 0) t0 = now;
        else if (now - t0 > limit_ns) break;
    }
    return wait_failed(status, code, bar_addr, parity);
}
__device__ __forceinline__ bool mbar_spin(uint64_t* bar, uint32_t parity, int* status, int code) {
    if (mbar_test(bar, parity)) return true;
    return mbar_spin_slow(smem_u32(bar), parity, status, code, kWaitLimitNs);
}
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int* status, int code) {
    if (mbar_test(bar, parity)) return true;       // already complete: no suspension round trip
    return mbar_wait_slow(smem_u32(bar), parity, status, code, kWaitLimitNs);
}

__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// ---------------------------------------------------------------------------
// TMA (tiled bulk tensor copies global -> shared, completion on an mbarrier)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tma_prefetch_desc(const CUtensorMap* m) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
}
// untiled bulk copy global -> shared (16-byte aligned addresses, size a multiple of 16 bytes)
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* m, int c0, int c1, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(bar)), "r"(c0), "r"(c1)
        : "memory");
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* m, int c0, int c1, int c2,
                                            uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}
__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* m, int c0, int c1, int c2, int c3,
                                            uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2),
          "r"(c3)
        : "memory");
}

// Ask for a tile to be brought into L2 (no shared-memory destination, nothing to wait for): the
// later load of the same tile then pays the L2 latency instead of HBM's.
__device__ __forceinline__ void tma_prefetch_4d(const CUtensorMap* m, int c0, int c1, int c2, int c3) {
    asm volatile("cp.async.bulk.prefetch.tensor.4d.L2.global.tile [%0, {%1, %2, %3, %4}];"
                 ::"l"(reinterpret_cast<uint64_t>(m)), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
                 : "memory");
}

// Tiled stores shared -> global (bulk async-group completion).  The issuing thread commits the
// group and waits until the copies have READ their shared-memory source before it is reused.
__device__ __forceinline__ void tma_store_4d(const CUtensorMap* m, const void* src, int c0, int c1, int c2, int c3) {
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];"
                 ::"l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(src)), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
                 : "memory");
}
__device__ __forceinline__ void bulk_store(void* dst, const void* src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

// ---------------------------------------------------------------------------
// Tensor memory
// ---------------------------------------------------------------------------
// One full warp allocates `ncols` (power of two >= 32) columns; the base address lands in *slot.
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)),
                 "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// ---------------------------------------------------------------------------
// UMMA descriptors
// ---------------------------------------------------------------------------
// Instruction descriptor, kind::f16, bf16 x bf16 -> fp32.  a_mn / b_mn: operand is MN-major.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, bool a_mn, bool b_mn) {
    return (1u << 4)                       // D format: fp32
           | (1u << 7)                     // A format: bf16
           | (1u << 10)                    // B format: bf16
           | ((a_mn ? 1u : 0u) << 15)      // A major
           | ((b_mn ? 1u : 0u) << 16)      // B major
           | ((uint32_t)(N >> 3) << 17)    // N / 8
           | ((uint32_t)(M >> 4) << 24);   // M / 16
}
// Shared-memory matrix descriptor.  layout: 0 = no swizzle, 2 = 128-byte swizzle.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes, uint32_t layout) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4)
           | ((uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16)
           | ((uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32)
           | ((uint64_t)1 << 46)                                  // descriptor version (sm_100)
           | ((uint64_t)layout << 61);
}
constexpr uint32_t kSwz128 = 2, kSwzNone = 0;
// The descriptor of the same operand `bytes` further on (bytes a multiple of 16): one 64-bit add,
// so that a loop over K steps does not rebuild descriptors.
__device__ __forceinline__ uint64_t desc_off(uint64_t desc, uint32_t bytes) {
    // The address field (bits 0-13, 16-byte units) never carries: every operand lies inside the
    // CTA's shared memory.  A 32-bit add on the low word is one instruction for the issuing thread,
    // whose instruction count per MMA bounds the tensor pipe's utilisation.
    const uint32_t lo = (uint32_t)desc + (bytes >> 4);
    return (desc & 0xFFFFFFFF00000000ull) | (uint64_t)lo;
}

// D[tmem] (+)= A[smem] * B[smem]; one elected thread issues.
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
// All MMAs issued so far by this thread arrive on `bar` when they complete.
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

// ---------------------------------------------------------------------------
// TMEM <-> registers (32 lanes x 32 bit, N columns per thread; warp w touches lanes 32*(w%4)..)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// The same, naming registers that loads issued a while ago fill: their uses stay behind it.
__device__ __forceinline__ void tmem_ld_wait16(uint32_t (&v)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                   "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15])
                 :: "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld1(uint32_t taddr, uint32_t& v) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(v) : "r"(taddr) : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
          "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
        : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
        ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
          "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]),
          "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]),
          "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
        : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&v)[8]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
        ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
        : "memory");
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// Teardown.  A CTA that has given up a wait must not give its tensor memory back, nor end, with MMAs of its own still running or
// copies into its shared memory still on their way.  Called after the last block-wide barrier, when nobody waits
// any more and the flag is final, by the one warp whose elected lane issues MMAs and which also gives the tensor memory back
// (cta_teardown_warp), or else by all threads (cta_teardown; `issuing`: such a warp, `slot`: which of two).
// Every poll has a limit of its own and takes no notice of the flag:
//  * MMAs: a commit of the lane that issued them, polled;
//  * the barrier that ran out first, polled again: if it waited for a copy, that copy may have come meanwhile;
//  * other copies: a pause.  Those asked for before that wait began have had its second; those after it (nothing is asked for by a
//    thread whose own wait gave up) come within microseconds unless the memory system is lost.  This part is best effort: a copy
//    that has not come within a second has no bound.
constexpr uint64_t kDrainLimitNs = 10000000ull, kDrainPauseNs = 1000000ull;
__device__ __forceinline__ uint64_t* cta_drain_bars() {       // one for each such warp; set up only when needed
    __shared__ uint64_t bars[2];
    return bars;
}
static __device__ __noinline__ bool mbar_drain(uint32_t bar_addr, uint32_t parity) {
    const uint64_t t0 = globaltimer_ns();
#pragma unroll 1
    do {
        if (mbar_test_addr(bar_addr, parity)) return true;
        __nanosleep(1000);
    } while (globaltimer_ns() - t0 < kDrainLimitNs);
    return false;
}
static __device__ __noinline__ void cta_drain_warp(int slot) {
    if (elect_one()) {
        uint64_t* bar = cta_drain_bars() + slot;
        mbar_init(bar, 1);
        mbar_fence_init();
        umma_commit(bar);
        mbar_drain(smem_u32(bar), 0);
        const uint32_t what = (uint32_t)*cta_giveup_flag();
        mbar_drain(what >> 2, what >> 1 & 1);
        const uint64_t t0 = globaltimer_ns();
#pragma unroll 1
        while (globaltimer_ns() - t0 < kDrainPauseNs) __nanosleep(1000);
    }
    __syncwarp();
}
__device__ __forceinline__ void cta_teardown_warp() {
    if (cta_gave_up()) cta_drain_warp(0);
}
__device__ __forceinline__ void cta_teardown(bool issuing, int slot = 0) {
    if (cta_gave_up()) {
        if (issuing) cta_drain_warp(slot);
        __syncthreads();
    }
}

// Byte offset of 16-byte chunk `chunk` (0..7) of row `row` inside a [rows x 128 B] tile held in
// the 128-byte-swizzled layout TMA produces (tile base 1024-byte aligned).
__device__ __forceinline__ uint32_t swz128_offset(uint32_t row, uint32_t chunk) {
    return row * 128u + ((chunk ^ (row & 7u)) << 4);
}

}  // namespace tc
}  // namespace psk
