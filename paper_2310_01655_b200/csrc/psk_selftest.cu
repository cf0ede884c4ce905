// Self-test of the bounded device-side wait (see include/psk.h: psk_selftest_wait_timeout).
#include "psk_internal.cuh"
#include "tc_prims.cuh"

namespace psk {
namespace {

constexpr int kErrSelfTest = 99;

// One CTA of 128 threads waits on an mbarrier that nobody arrives at, through the same bounded
// wait the tensor-core kernels use.  The wait gives up after `limit_ns`, records its code in the
// workspace's status word and raises the CTA's give-up flag; a second wait on the same barrier
// must then come back at once.  Before the waits one lane has asked for a copy and issued an MMA that nobody waits for; after them
// the CTA goes through the kernels' teardown and gives its tensor memory back.
// out[0] = nanoseconds the first wait took (thread 0), out[1] = nanoseconds the second one took, out[2] = threads whose first wait
// returned false, out[3] = threads whose second wait returned false, out[4] = nanoseconds the teardown took, out[5] = 1 if the
// teardown's commit of the MMA had completed after it, out[6] = 1 if the copy had.  Nothing traps, nothing spins without a bound.
__global__ void __launch_bounds__(128) wait_timeout_kernel(int* status, unsigned long long limit_ns,
                                                           unsigned long long* out) {
    __shared__ __align__(1024) uint8_t ops[4096 + 512 + 128];        // A [128 x 16], B [16 x 16] (bf16, zeros), the copy
    __shared__ uint64_t bar, bar_ld;
    __shared__ uint32_t tm_slot;
    __shared__ int failed[2];
    const int tid = threadIdx.x, warp = tc::warp_index();
    for (int e = tid; e < (4096 + 512) / 16; e += 128) reinterpret_cast<uint4*>(ops)[e] = make_uint4(0, 0, 0, 0);
    if (tid == 0) {
        tc::mbar_init(&bar, 1);
        tc::mbar_init(&bar_ld, 1);
        tc::cta_giveup_init();
        tc::mbar_fence_init();
        failed[0] = failed[1] = 0;
    }
    if (warp == 0) { tc::tmem_alloc(&tm_slot, 32); tc::tmem_relinquish(); }
    tc::fence_proxy_async_smem();
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tm = tm_slot;
    if (warp == 0 && tc::elect_one()) {
        tc::mbar_expect_tx(&bar_ld, 128);
        tc::bulk_load(ops + 4096 + 512, out + 8, 128, &bar_ld);
        tc::umma_ss(tm, tc::smem_desc(tc::smem_u32(ops), 2048, 128, tc::kSwzNone), tc::smem_desc(tc::smem_u32(ops) + 4096, 256, 128, tc::kSwzNone),
                    tc::idesc_bf16(128, 16, false, false), 0);
    }
    const uint64_t t0 = tc::globaltimer_ns();
    const bool first = tc::mbar_wait_slow(tc::smem_u32(&bar), 0, status, kErrSelfTest, limit_ns);
    const uint64_t t1 = tc::globaltimer_ns();
    const bool second = tc::mbar_wait_slow(tc::smem_u32(&bar), 0, status, kErrSelfTest, limit_ns);
    const uint64_t t2 = tc::globaltimer_ns();
    if (!first) atomicAdd(&failed[0], 1);
    if (!second) atomicAdd(&failed[1], 1);
    tc::tc_fence_before();
    __syncthreads();
    const uint64_t t3 = tc::globaltimer_ns();
    tc::cta_teardown(warp == 0);
    if (tid == 0) {
        out[0] = t1 - t0; out[1] = t2 - t1;
        out[2] = (unsigned long long)failed[0]; out[3] = (unsigned long long)failed[1];
        out[4] = tc::globaltimer_ns() - t3;
        out[5] = tc::cta_gave_up() && tc::mbar_test(tc::cta_drain_bars(), 0);
        out[6] = tc::mbar_test(&bar_ld, 0);
    }
    if (warp == 0) tc::tmem_dealloc(tm, 32);
}

}  // namespace
}  // namespace psk

extern "C" int psk_selftest_wait_timeout(void* workspace, size_t workspace_bytes, uint64_t limit_ns, void* stream) {
    using namespace psk;
    if (!workspace || workspace_bytes < kStatusBytes || (reinterpret_cast<uintptr_t>(workspace) % kAlign))
        return PSK_ERR_WORKSPACE;
    if (limit_ns == 0 || limit_ns > 100000000ull) return PSK_ERR_INVALID_ARG;      // at most 0.1 s
    cudaStream_t s = (cudaStream_t)stream;
    if (cudaMemsetAsync(workspace, 0, kStatusBytes, s) != cudaSuccess) return PSK_ERR_CUDA;
    // the status word is the first int; the report goes 64 bytes further on, inside the status block
    wait_timeout_kernel<<<1, 128, 0, s>>>(reinterpret_cast<int*>(workspace), limit_ns,
                                          reinterpret_cast<unsigned long long*>(static_cast<char*>(workspace) + 64));
    return cudaGetLastError() == cudaSuccess ? PSK_OK : PSK_ERR_CUDA;
}
