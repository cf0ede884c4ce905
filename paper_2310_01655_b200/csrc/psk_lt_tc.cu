// lt(A B^T) C for given bf16 feature matrices on the tensor cores: Section 3.1's block algorithm,
//   H_l = B_l^T C_l,  Z_l = sum_{j<l} H_j,  rows of block l = lt(A_l B_l^T) C_l + A_l Z_l,
// with fp32 accumulation in tensor memory.  A, B: [batch, n, m] bf16 (m a multiple of 64),
// C: [batch, n, 64] bf16, Out: [batch, n, 64] fp32, blocks of b = 128 or 256 rows.
// Every operand goes to the tensor cores as TMA left it in shared memory: B_l^T C_l contracts over
// the rows (both tiles MN-major), A_l Z_l and A_l B_l^T over the features (A, B K-major, Z MN-major).
#include "tc_common.cuh"

namespace psk {

namespace {

using namespace tc;

// ---------------------------------------------------------------------------
// prefix states, bf16 [batch][t][m][64] (entry l: the sum over the blocks before l; l = 0 unused).
// grid (ceil(m/128), batch): a CTA walks the whole sequence for 128 features, the running sum stays in tensor
// memory and is copied out at every block boundary by the first four warps; the fifth issues the MMAs, the sixth the loads.
// Bound with few CTAs: the latency of a load, with two stages.  (With loads and MMAs issued by one elected lane of a row warp, whose
// other lanes wait for it and read the sum late: batch 1, n 8192, m 64, b 256: 65 us, now 42; batch 24, m 320: 76 and 60; batch 12,
// n 4096, m 1024, b 128: 54 and 44.  Behind a thread index instead of an election: 57, 62, 46.)
// ---------------------------------------------------------------------------
constexpr int kStThreads = 192;
constexpr int kStStage = 32768 + 16384;     // two 64-feature groups of the B tile, the C tile
constexpr int kStSmem = 2 * kStStage + 1024;

__global__ void __launch_bounds__(kStThreads)
lt_tc_state_kernel(const __grid_constant__ CUtensorMap mapB, const __grid_constant__ CUtensorMap mapC, bf16* __restrict__ Z,
                   int m, int t, int tpb, int* status) {
    pdl_sync();
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    __shared__ uint64_t bar_full[2], bar_free[2], bar_acc, bar_read;
    __shared__ uint32_t tm_slot;
    const int tid = threadIdx.x, warp = warp_index();
    const int f0 = blockIdx.x * 128, bt = blockIdx.y;
    const int NT = (t - 1) * tpb;               // the last block's state is never used
    if (tid == 0) {
        cta_giveup_init();
        mbar_init(&bar_full[0], 1); mbar_init(&bar_full[1], 1);
        mbar_init(&bar_free[0], 1); mbar_init(&bar_free[1], 1);
        mbar_init(&bar_acc, 1); mbar_init(&bar_read, 4);
        mbar_fence_init();
    }
    if (warp == 4) { tmem_alloc(&tm_slot, 64); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tm = tm_slot;
    bool ok = true;
    if (warp == 5) {
        if (elect_one()) {
            for (int j = 0; j < NT; ++j) {
                const int s = j & 1;
                if (j >= 2) ok = mbar_spin(&bar_free[s], ((j - 2) >> 1) & 1, status, kErrMma);
                if (!ok) break;
                uint8_t* st = smem + s * kStStage;
                mbar_expect_tx(&bar_full[s], kStStage);
                tma_load_3d(st, &mapB, f0, j * 128, bt, &bar_full[s]);
                tma_load_3d(st + 16384, &mapB, f0 + 64, j * 128, bt, &bar_full[s]);     // beyond m: zeros
                tma_load_3d(st + 32768, &mapC, 0, j * 128, bt, &bar_full[s]);
            }
        }
    } else if (warp == 4) {
        if (elect_one()) {
            constexpr uint32_t idesc = idesc_bf16(128, 64, true, true);
            for (int l = 0; l + 1 < t && ok; ++l) {
                // this block's MMAs add to the accumulator only after everyone has read it
                if (l > 0) ok = mbar_spin(&bar_read, (l - 1) & 1, status, kErrMma);
                for (int tt = 0; tt < tpb && ok; ++tt) {
                    const int j = l * tpb + tt, s = j & 1;
                    ok = mbar_spin(&bar_full[s], (j >> 1) & 1, status, kErrTma);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t base = smem_u32(smem + s * kStStage);
                    const uint64_t ad = smem_desc(base, 16384, 1024, kSwz128);
                    const uint64_t bd = smem_desc(base + 32768, 0, 1024, kSwz128);
#pragma unroll
                    for (int k = 0; k < 8; ++k) umma_ss(tm, desc_off(ad, k * 2048), desc_off(bd, k * 2048), idesc, (j > 0 || k > 0) ? 1u : 0u);
                    umma_commit(&bar_free[s]);
                    if (tt + 1 == tpb) umma_commit(&bar_acc);
                }
            }
        }
    } else {
        const uint32_t lane_tm = tm + ((uint32_t)(warp * 32) << 16);
        for (int l = 0; l + 1 < t; ++l) {
            ok = mbar_wait(&bar_acc, l & 1, status, kErrMma) && ok;
            tc_fence_after();
            if (f0 + tid < m) {                       // (the same for a whole warp, as tensor-memory loads need it; `ok` may not be)
                bf16* dst = Z + (((size_t)bt * t + l + 1) * m + f0 + tid) * 64;
#pragma unroll
                for (int c0 = 0; c0 < 64; c0 += 32) {
                    uint32_t u[32];
                    tmem_ld32(lane_tm + c0, u);
                    tmem_ld_wait();
#pragma unroll
                    for (int j = 0; j < 32; j += 8)
                        if (ok) *reinterpret_cast<uint4*>(dst + c0 + j) =
                            make_uint4(pack_bf16(__uint_as_float(u[j]), __uint_as_float(u[j + 1])), pack_bf16(__uint_as_float(u[j + 2]), __uint_as_float(u[j + 3])),
                                       pack_bf16(__uint_as_float(u[j + 4]), __uint_as_float(u[j + 5])), pack_bf16(__uint_as_float(u[j + 6]), __uint_as_float(u[j + 7])));
                }
            }
            tc_fence_before();
            __syncwarp();
            if (tid % 32 == 0) mbar_arrive(&bar_read);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 4) { cta_teardown_warp(); tmem_dealloc(tm, 64); }
}

// ---------------------------------------------------------------------------
// rows: grid (t, batch), one CTA per block of TPB = b / 128 row tiles.  Warps of the first TPB warpgroups: thread =
// row (masking, epilogue); the last warp: one thread issues every TMA load and every MMA.  The features are
// walked once in chunks of 64: a chunk of the block's A rows multiplies the prefix state's chunk (into
// O) and the same chunk of the block's B rows (into the scores of the tile pairs on and below the diagonal); the
// masked scores then multiply the tiles of C from tensor memory.  Bound: memory; A, B and Z cross it once.
// (With a CTA per row tile B's tiles and Z were read again for the second tile: batch 24, n 8192, m 1024,
// b 256: 234 us.)
// ---------------------------------------------------------------------------
template <int TPB> struct LtRows {
    static constexpr int A = 0, B = TPB * 16384, Z = 2 * B, kStage = Z + 8192, kStages = 2;
    static constexpr int C = kStages * kStage, bytes = C + TPB * 16384 + 1024;
    static constexpr int kThreads = 128 * TPB + 32;
    static constexpr uint32_t kTmem = TPB == 1 ? 256 : 512;            // O 64 TPB, scores 128 per tile pair
    static constexpr uint32_t cS = 128;
};

template <int TPB>
__global__ void __launch_bounds__(LtRows<TPB>::kThreads)
lt_tc_rows_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                  const __grid_constant__ CUtensorMap mapC, const __grid_constant__ CUtensorMap mapZ,
                  float* __restrict__ Out, int n, int m, int t, int* status) {
    using L = LtRows<TPB>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    __shared__ uint64_t bar_full[L::kStages], bar_free[L::kStages], bar_c, bar_s, bar_p[TPB], bar_o[TPB];
    __shared__ uint32_t tm_slot;
    const int tid = threadIdx.x, warp = warp_index();
    const int l = blockIdx.x, bt = blockIdx.y;
    const int row0 = l * TPB * 128, nch = m / 64;
    if (tid == 0) {
        cta_giveup_init();
        for (int i = 0; i < L::kStages; ++i) { mbar_init(&bar_full[i], 1); mbar_init(&bar_free[i], 1); }
        mbar_init(&bar_c, 1); mbar_init(&bar_s, 1);
        for (int w = 0; w < TPB; ++w) { mbar_init(&bar_p[w], 128); mbar_init(&bar_o[w], 1); }
        mbar_fence_init();
    }
    pdl_sync();
    if (warp == 4 * TPB) { tmem_alloc(&tm_slot, L::kTmem); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tm = tm_slot;
    // scores of row tile w against tile tp <= w
    auto scores = [](int w, int tp) { return L::cS + 128u * (w * (w + 1) / 2 + tp); };
    if (warp == 4 * TPB && elect_one()) {
        auto load = [&](int c) {
            const int s = c % L::kStages;
            uint8_t* st = smem + s * L::kStage;
            mbar_expect_tx(&bar_full[s], 2 * TPB * 16384 + (l > 0 ? 8192 : 0));
#pragma unroll
            for (int w = 0; w < TPB; ++w) {
                tma_load_3d(st + L::A + w * 16384, &mapA, c * 64, row0 + w * 128, bt, &bar_full[s]);
                tma_load_3d(st + L::B + w * 16384, &mapB, c * 64, row0 + w * 128, bt, &bar_full[s]);
            }
            if (l > 0) tma_load_3d(st + L::Z, &mapZ, 0, c * 64, bt * t + l, &bar_full[s]);
        };
        for (int c = 0; c < L::kStages && c < nch; ++c) load(c);
        mbar_expect_tx(&bar_c, TPB * 16384);
        for (int w = 0; w < TPB; ++w) tma_load_3d(smem + L::C + w * 16384, &mapC, 0, row0 + w * 128, bt, &bar_c);
        constexpr uint32_t idesc_z = idesc_bf16(128, 64, false, true);
        constexpr uint32_t idesc_s = idesc_bf16(128, 128, false, false);
        bool ok = true;
        for (int c = 0; c < nch && ok; ++c) {
            const int s = c % L::kStages;
            ok = mbar_spin(&bar_full[s], (c / L::kStages) & 1, status, kErrTma);
            if (!ok) break;
            tc_fence_after();
            const uint32_t base = smem_u32(smem + s * L::kStage);
            const uint64_t zd = smem_desc(base + L::Z, 0, 1024, kSwz128);
#pragma unroll
            for (int w = 0; w < TPB; ++w) {
                const uint64_t ad = smem_desc(base + L::A + w * 16384, 0, 1024, kSwz128);
                if (l > 0) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) umma_ss(tm + w * 64, desc_off(ad, k * 32), desc_off(zd, k * 2048), idesc_z, (c > 0 || k > 0) ? 1u : 0u);
                }
#pragma unroll
                for (int tp = 0; tp <= w; ++tp) {
                    const uint64_t bd = smem_desc(base + L::B + tp * 16384, 0, 1024, kSwz128);
#pragma unroll
                    for (int k = 0; k < 4; ++k) umma_ss(tm + scores(w, tp), desc_off(ad, k * 32), desc_off(bd, k * 32), idesc_s, (c > 0 || k > 0) ? 1u : 0u);
                }
            }
            umma_commit(&bar_free[s]);
            if (c + L::kStages < nch) {
                ok = mbar_spin(&bar_free[s], (c / L::kStages) & 1, status, kErrMma);
                if (ok) load(c + L::kStages);
            }
        }
        if (ok) umma_commit(&bar_s);
        ok = ok && mbar_spin(&bar_c, 0, status, kErrTma);
#pragma unroll
        for (int w = 0; w < TPB; ++w) {
            ok = ok && mbar_spin(&bar_p[w], 0, status, kErrMma);
            if (ok) {
                tc_fence_after();
#pragma unroll
                for (int tp = 0; tp <= w; ++tp) {
                    const uint64_t cd = smem_desc(smem_u32(smem + L::C + tp * 16384), 0, 1024, kSwz128);
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        umma_ts(tm + w * 64, tm + scores(w, tp) + k * 8, desc_off(cd, k * 2048), idesc_z, (l > 0 || tp > 0 || k > 0) ? 1u : 0u);
                }
                umma_commit(&bar_o[w]);
            }
        }
    } else if (warp < 4 * TPB) {
        const int w = warp / 4, wt = tid % 128;
        const uint32_t lane_tm = tm + ((uint32_t)((warp % 4) * 32) << 16);
        bool ok = mbar_wait(&bar_s, 0, status, kErrMma);
        tc_fence_after();
        {                                             // (not behind `ok`: all lanes of a warp read and write tensor memory)
            for (int tp = 0; tp <= w; ++tp) {
                const bool diag = tp == w;
                const uint32_t ts = lane_tm + scores(w, tp);
#pragma unroll
                for (int c0 = 0; c0 < 128; c0 += 32) {
                    uint32_t u[32], pk[16];
                    tmem_ld32(ts + c0, u);
                    tmem_ld_wait();
#pragma unroll
                    for (int j = 0; j < 32; j += 2) {
                        const float x = (diag && c0 + j > wt) ? 0.f : __uint_as_float(u[j]);
                        const float y = (diag && c0 + j + 1 > wt) ? 0.f : __uint_as_float(u[j + 1]);
                        pk[j / 2] = pack_bf16(x, y);
                    }
                    // the masked scores as the bf16 A operand of the last GEMM, over the columns just read
                    tmem_st16(ts + c0 / 2, pk);
                }
            }
            tmem_st_wait();
        }
        tc_fence_before();
        mbar_arrive(&bar_p[w]);
        ok = ok && mbar_wait(&bar_o[w], 0, status, kErrMma);
        tc_fence_after();
        {
            float* dst = Out + ((size_t)bt * n + row0 + w * 128 + wt) * 64;
#pragma unroll
            for (int c0 = 0; c0 < 64; c0 += 32) {
                uint32_t u[32];
                tmem_ld32(lane_tm + w * 64 + c0, u);
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 32; j += 4)
                    if (ok) *reinterpret_cast<float4*>(dst + c0 + j) = make_float4(__uint_as_float(u[j]), __uint_as_float(u[j + 1]),
                                                                           __uint_as_float(u[j + 2]), __uint_as_float(u[j + 3]));
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 4 * TPB) { cta_teardown_warp(); tmem_dealloc(tm, L::kTmem); }
}

template <int TPB>
cudaError_t launch_rows(const CUtensorMap& mA, const CUtensorMap& mB, const CUtensorMap& mC, const CUtensorMap& mZ, float* Out, int batch, int n, int m,
                        int t, int* status, cudaStream_t s) {
    using L = LtRows<TPB>;
    PSK_TRY(set_smem(lt_tc_rows_kernel<TPB>, L::bytes));
    prof_begin("lt_tc_rows_kernel", s);
    launch_pdl(lt_tc_rows_kernel<TPB>, dim3(t, batch), L::kThreads, L::bytes, s, mA, mB, mC, mZ, Out, n, m, t, status);
    prof_end(s);
    return cudaGetLastError();
}

bool lt_tc_args_ok(int batch, int n, int m, int k, int b) {
    return batch > 0 && n > 0 && m > 0 && m % 64 == 0 && k == 64 && (b == 128 || b == 256) && n % b == 0 &&
           (int64_t)batch * n < ((int64_t)1 << 31);
}

}  // namespace
}  // namespace psk

using namespace psk;

extern "C" {

size_t psk_lt_multiply_bf16_workspace_bytes(int batch, int n, int m, int k, int b) {
    if (!lt_tc_args_ok(batch, n, m, k, b)) return 0;
    return kStatusBytes + align_up((size_t)batch * (n / b) * m * 64 * sizeof(bf16));
}

int psk_lt_multiply_bf16(int batch, int n, int m, int k, int b, const void* A, const void* B, const void* C, float* Out,
                         void* workspace, size_t workspace_bytes, void* stream) {
    if (!lt_tc_args_ok(batch, n, m, k, b)) return PSK_ERR_SHAPE;
    if (!A || !B || !C || !Out) return PSK_ERR_INVALID_ARG;
    for (const void* p : {A, B, C, (const void*)Out, (const void*)workspace})
        if (reinterpret_cast<uintptr_t>(p) & 15u) return PSK_ERR_ALIGN;
    const size_t need = psk_lt_multiply_bf16_workspace_bytes(batch, n, m, k, b);
    if (!workspace || workspace_bytes < need) return PSK_ERR_WORKSPACE;
    cudaStream_t s = (cudaStream_t)stream;
    int* status = static_cast<int*>(workspace);
    bf16* Z = reinterpret_cast<bf16*>(static_cast<char*>(workspace) + kStatusBytes);
    const int t = n / b, tpb = b / 128;
    if (cudaMemsetAsync(workspace, 0, kStatusBytes, s) != cudaSuccess) return PSK_ERR_CUDA;
    CUtensorMap mA, mB, mC, mZ;
    if (!tc_map_3d(&mA, A, m, n, batch, 64, 128) || !tc_map_3d(&mB, B, m, n, batch, 64, 128) ||
        !tc_map_3d(&mC, C, 64, n, batch, 64, 128) || !tc_map_3d(&mZ, Z, 64, m, (int64_t)batch * t, 64, 64))
        return PSK_ERR_CUDA;
    if (set_smem(lt_tc_state_kernel, kStSmem) != cudaSuccess) return PSK_ERR_CUDA;
    if (t > 1) {
        prof_begin("lt_tc_state_kernel", s);
        launch_pdl(lt_tc_state_kernel, dim3((m + 127) / 128, batch), kStThreads, kStSmem, s, mB, mC, Z, m, t, tpb, status);
        prof_end(s);
    }
    const cudaError_t e = tpb == 1 ? launch_rows<1>(mA, mB, mC, mZ, Out, batch, n, m, t, status, s) : launch_rows<2>(mA, mB, mC, mZ, Out, batch, n, m, t, status, s);
    return e == cudaSuccess ? PSK_OK : PSK_ERR_CUDA;
}

}  // extern "C"
