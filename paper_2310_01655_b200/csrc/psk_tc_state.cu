// Prefix states of the block lower-triangular multiply (Section 3.1) on the tensor cores.
//
// State storage (HBM scratch): S[BH][t][FP][80] bf16, one 160-byte row per feature: the 64
// columns of H_l / Z_l, then the normaliser column (the "| 1" of [V | 1], or the last column of E
// in the backward), then zeros.
//
// Sequence runs (the parallel-prefix remark of Section 3.1): with nseg > 1 a head's blocks are cut
// into nseg runs of (nearly) equal length that are processed by different CTAs.  A first launch takes
// the runs but the last: run 0 writes its prefix states as usual, and each leaves its raw fp32 total in
// scratch; a small kernel turns the totals into running sums; a second launch starts run s >= 1 from
// the sum of the totals before it and writes its prefix states.  Twice the arithmetic (but for the
// first and the last run), nseg - 1 times the parallelism: used when there are too few heads to
// fill the GPU.  The totals alone, followed by a small summing kernel, give the single global
// state of non-causal attention.
#include "tc_common.cuh"

namespace psk {

using namespace tc;

namespace {

// What a launch does with a run of blocks:
constexpr int kModePrefix = 0;         // write the exclusive prefix state at every block boundary
constexpr int kModeTotal = 1;          // write only the raw fp32 total at the end of the run
constexpr int kModeFirst = 2;          // run 0: both; the other runs: the total only

// ---------------------------------------------------------------------------
// Prefix states of one head, sequentially along the sequence (Section 3.1, Z_l = sum_{j<l} H_j):
//   S[l] = sum over blocks before l (after l when `reverse`) of phi(X_blk)^T [Y_blk | y65]
// for feature tiles [T0, T0+TN).  The running sum never leaves tensor memory (fp32); at every
// block boundary it is rounded to bf16 and written out, then the block's own contribution is
// accumulated on top -- the per-block states H_l and the scan over them are fused away.
//   X: tensor that is sketched (K for the forward state, Q for the backward's reverse state)
//   Y: [V] or [dO];  y65: last column (nullptr = all ones);  fscale: per-token d_i, the
//   features of token i are divided by it (nullptr = not) -- phi(q_i)^T [dO_i | y65_i] / d_i is the
//   suffix state's phi(q_i)^T E_i without E ever being formed
//   H, H2: where the tokens' half sketches go as [hi | lo] score operands for the row kernels, which would
//   otherwise sketch every other-side tile again, once per row tile that meets it.  (Rows of 48 heads x 16384,
//   r = 64: forward 1050 -> 554 us, query side 1702 -> 1288, key side 2327 -> 2112; of 384 heads x 32768,
//   r = 32: 4409 -> 3916, 5031 -> 4776, 6249 -> 5867; the walk itself pays 5 to 20 % for it.)
// What bounds a walk of r = 32: the shared-memory path, which the generators' tiles, the stores on their way out and the
// MMAs' operands share (96 heads x 8192, b = 256, before elected issue and unrolled features: 82 % of its cycles on the SMs in
// use, issue slots 51 %, tensor pipe 27 %), and at short blocks the store warpgroup, one body for all tiles with a bulk copy out (144 heads x
// 8192, b = 256: 318 us unrolled and with copies by the lanes, now 234).
// grid (BH, runs, shares).  Warp roles:
//   NWG generator warpgroups  thread = token: read the half sketches, write their feature tiles
//                             (dealt in turn) as MN-major A operands into shared memory; one of them also
//                             puts the half sketches where their rows were;
//   NSW store warpgroups      thread = feature row: at block boundaries reads the accumulators,
//                             centres, rounds and stores them;
//   2 feeder warps            one thread each: every TMA load and sketch GEMM; every state GEMM.
// Stored layout S[blk][FP][80]: one row per feature, 64 state columns, the last column, zeros.
// ---------------------------------------------------------------------------
template <int R, int NWG, int NSW>
struct StateSmem {
    static constexpr uint32_t kG = 2 * R * 128 < 1024 ? 1024 : 2 * R * 128;
    // X: 16 KB slots for the rows to sketch, through which their half sketches leave.  A third one where there is room:
    // with two, a tile's rows can be requested only when the half sketches two tiles earlier have left.
    static constexpr int kXSlots = R < 64 && 3 * 16384 + 49152 + kG + NWG * 32768 + NSW * 128 * 160 + 3072 <= 232448 ? 3 : 2;
    static_assert(R < 64 || kXSlots == 2, "the second half's buffer is single");
    static constexpr uint32_t X = 0;
    static constexpr uint32_t Y = kXSlots * 16384;       // two slots of 16 KB values
    // The operand's columns 64..79 (the last column, zeros) of both slots: 32 of the 128 bytes of a row each, so one chunk of the
    // same layout holds both, slot 1's two 16-byte pieces further on
    static constexpr uint32_t kYSlot = 16384, Ext = Y + 2 * kYSlot;
    static constexpr uint32_t G = Ext + 16384;
    static constexpr uint32_t A0 = G + kG;
    static constexpr uint32_t St = A0 + NWG * 32768;     // a state tile on its way out per store warpgroup: 128 rows x 160 B
    static constexpr uint32_t kSt = NSW * 128 * 160;
    static constexpr bool kStaged = St + kSt + (R == 64 ? 16384 : 0) + 2048 <= 232448;     // where it fits
    // r = 64: the second 64 columns of a tile's [hi | lo] half sketches on their way out (the first, and all of
    // them for r <= 32, leave through the tile's own X buffer)
    static constexpr uint32_t Hl = St + (kStaged ? kSt : 0);
    static constexpr uint32_t total = Hl + (R == 64 ? 16384 : 0);
    static_assert(total + 2048 <= 232448, "shared memory");
};

// Barrier among the 128 threads of a warpgroup.  The generator and store roles never leave a
// loop early: a wait that gave up returns at once from then on (tc_prims.cuh), so they run the
// remaining iterations through, barriers and arrivals included, and nobody is left waiting at a
// barrier that has lost a participant.
__device__ __forceinline__ void wg_barrier(int wg) {
    asm volatile("bar.sync %0, 128;" ::"r"(wg + 1) : "memory");
}

constexpr int kErrState = 3;

// Barriers and centres of a CTA: one object for all the shares that a kernel's code covers.
template <int TN, int NWG>
struct StateShared {
    uint64_t fullx[3], fully[2], yfree[2], ext[2], sk, mread, drain[2], hl[2], hlfree;
    uint64_t aready[NWG], afree[NWG], accfull[TN], accread[TN];
    uint32_t tmem_slot;
    alignas(16) float cm[64];
};

// m as [hi | lo] columns: one tile, or (r = 64) two tiles of 64
template <int R>
__device__ __forceinline__ void store_hl_rows(uint8_t* t0, uint8_t* t1, const float (&m)[R], int row) {
#pragma unroll
    for (int ch = 0; ch < R / 8; ++ch) {
        uint32_t h[4], l[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float a = m[8 * ch + 2 * i], b = m[8 * ch + 2 * i + 1];
            h[i] = pack_bf16(a, b);
            l[i] = pack_bf16(a - __uint_as_float(h[i] << 16), b - __uint_as_float(h[i] & 0xffff0000u));
        }
        *reinterpret_cast<uint4*>(t0 + swz128_offset(row, ch)) = make_uint4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<uint4*>((R == 64 ? t1 : t0) + swz128_offset(row, R == 64 ? ch : R / 8 + ch)) = make_uint4(l[0], l[1], l[2], l[3]);
    }
}

// acc[0..80) of this thread's lane = tot[row * 80 + ...], half a row's loads in flight at a time
static __device__ __noinline__ void state_init_acc(const float* __restrict__ tot, size_t row, uint32_t acc_tmem) {
    const float4* src = reinterpret_cast<const float4*>(tot + row * 80);
#pragma unroll 1
    for (int h = 0; h < 80; h += 40) {
        float4 x[10];
#pragma unroll
        for (int q = 0; q < 10; ++q) x[q] = src[h / 4 + q];
#pragma unroll
        for (int c = 0; c < 40; c += 8) {
            const float4 u = x[c / 4], v = x[c / 4 + 1];
            const uint32_t w[8] = {__float_as_uint(u.x), __float_as_uint(u.y), __float_as_uint(u.z), __float_as_uint(u.w),
                                   __float_as_uint(v.x), __float_as_uint(v.y), __float_as_uint(v.z), __float_as_uint(v.w)};
            tmem_st8(acc_tmem + h + c, w);
        }
    }
}

// SEG = false is the plain walk of a whole head by one CTA (nseg = 1, prefix mode, no start value):
// its run bookkeeping folds away at compile time.
template <int R, int T0, int TN, int NWG, int NSW, bool SEG, typename SH>
__device__ __forceinline__ void
state_walk(SH& sh, const CUtensorMap& mapX, const CUtensorMap& mapY, const CUtensorMap& mapH, const CUtensorMap& mapH2, int want_hl,
           const uint8_t* __restrict__ gimg, int g_heads, int H, int n, int b, int t,
           const float* __restrict__ y65, const float* __restrict__ fscale, const float* __restrict__ cmean,
           int center_mode, int reverse, int nseg_arg, int mode_arg, int run0, int units, float* __restrict__ tot,
           bf16* __restrict__ S, int lin, int* status) {
    using F = Feat<R>;
    using L = StateSmem<R, NWG, NSW>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    const int tid = threadIdx.x, warp = warp_index(), wg = warp / 4, wt = tid % 128;
    const int bh = blockIdx.x;
    const int seg = SEG ? run0 + (int)blockIdx.y : 0, nseg = SEG ? nseg_arg : 1;
    const int mode = !SEG ? kModePrefix : (mode_arg == kModeFirst && seg > 0 ? kModeTotal : mode_arg);
    const int hi = bh % H, bi = bh / H;
    const int g = g_heads == 1 ? 0 : hi;
    const int tpb = b / 128, NJ = n / 128;               // token tiles per block / per head
    // this CTA's run of the sequence: units (blocks; single tiles when there are no blocks to respect)
    // [u0, u1), tiles [j0, j0 + NJs), blocks [p0, p0 + ts)
    const int u0 = (int)((int64_t)units * seg / nseg), u1 = (int)((int64_t)units * (seg + 1) / nseg);
    const int upt = NJ / units;                          // tiles per unit
    const int j0r = SEG ? u0 * upt : 0, NJs = SEG ? (u1 - u0) * upt : NJ;
    const int p0r = SEG ? u0 : 0, ts = SEG ? u1 - u0 : t;
    // [hi | lo] half sketches: written by the CTA with a head's last, smallest share of the tiles, in the pass that visits
    // a run to write its states
    const bool hl = T0 + TN == F::NT && want_hl != 0 && mode != kModeTotal;
    // a later run of a prefix pass starts from the sum of the earlier runs' totals
    const bool init = SEG && mode == kModePrefix && seg > 0;
    constexpr int kThreads = 128 * (NWG + NSW) + 64;

    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sh.fully[i], 1); mbar_init(&sh.yfree[i], 1);
            mbar_init(&sh.ext[i], 1);
        }
        for (int i = 0; i < L::kXSlots; ++i) mbar_init(&sh.fullx[i], 1);
        mbar_init(&sh.hl[0], 1); mbar_init(&sh.hl[1], 1); mbar_init(&sh.hlfree, 1);
        mbar_init(&sh.sk, 1); mbar_init(&sh.mread, NWG); mbar_init(&sh.drain[0], 1); mbar_init(&sh.drain[1], 1);
        for (int i = 0; i < NWG; ++i) { mbar_init(&sh.aready[i], 1); mbar_init(&sh.afree[i], 1); }
        for (int i = 0; i < TN; ++i) { mbar_init(&sh.accread[i], 4); mbar_init(&sh.accfull[i], 1); }
        cta_giveup_init();
        mbar_fence_init();
        tma_prefetch_desc(&mapX); tma_prefetch_desc(&mapY);
    }
    // last-column chunk of both slots: zero, and each slot's column 0 = 1 when the last column is all ones
    for (int e = tid; e < 1024; e += kThreads) reinterpret_cast<uint4*>(smem + L::Ext)[e] = make_uint4(0, 0, 0, 0);
    pdl_sync();            // (before the allocation: a waiting CTA must not hold tensor memory)
    if (warp == 0) { tmem_alloc(&sh.tmem_slot, 512); tmem_relinquish(); }
    if (tid < 64) sh.cm[tid] = cmean != nullptr ? cmean[(size_t)bh * 64 + tid] : 0.f;
    __syncthreads();
    if (y65 == nullptr && tid < 128) {
        *reinterpret_cast<bf16*>(smem + L::Ext + swz128_offset(tid, 0)) = __float2bfloat16_rn(1.f);
        *reinterpret_cast<bf16*>(smem + L::Ext + swz128_offset(tid, 2)) = __float2bfloat16_rn(1.f);
    }
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tm = sh.tmem_slot;
    constexpr uint32_t kAcc = 2 * R;                      // accumulators start after the sketch columns
    // token tile visited at step j of this run (runs and tiles go backwards for suffix sums)
    auto tile_of = [&](int j) { const int gj = j0r + j; return reverse ? (NJ - 1 - gj) : gj; };

    if (wg == NWG + NSW) {
        // =============================== feeders ===============================
        // Two issuing threads in two warps.  The first loads the tiles and issues the sketch
        // GEMMs, the second issues the state GEMMs: between two of its MMAs lies as little as
        // possible (each satisfied wait, commit or TMA issue costs a single thread about a
        // hundred cycles, during which the tensor pipe would idle).
        if (warp == 4 * (NWG + NSW) && elect_one()) {
            bool ok = true;
            constexpr int NX = L::kXSlots;
            auto load_x = [&](int j) {
                // the first tile's barrier also covers the sketch matrices' image
                mbar_expect_tx(&sh.fullx[j % NX], 16384 + (j == 0 ? GImage<R>::bytes : 0u));
                if (j == 0) bulk_load(smem + L::G, gimg + (size_t)g * GImage<R>::bytes, GImage<R>::bytes, &sh.fullx[0]);
                tma_load_4d(smem + L::X + (j % NX) * 16384, &mapX, 0, tile_of(j) * 128, hi, bi, &sh.fullx[j % NX]);
            };
            auto load_y = [&](int j) {
                mbar_expect_tx(&sh.fully[j & 1], 16384);
                tma_load_4d(smem + L::Y + (j & 1) * L::kYSlot, &mapY, 0, tile_of(j) * 128, hi, bi, &sh.fully[j & 1]);
            };
            // the tile's half sketches as [hi | lo] rows, once the generators have put them over its X rows
            auto store_hl = [&](int j) {
                ok = ok && mbar_wait(&sh.hl[j & 1], (j >> 1) & 1, status, kErrState);
                if (!ok) return;
                tma_store_4d(&mapH, smem + L::X + (j % NX) * 16384, 0, tile_of(j) * 128, hi, bi);
                if constexpr (R == 64) tma_store_4d(&mapH2, smem + L::Hl, 0, tile_of(j) * 128, hi, bi);
                bulk_commit();
            };
            load_x(0);
            if (NJs > 1) load_x(1);
            load_y(0);
            ok = mbar_wait(&sh.fullx[0], 0, status, kErrTma);
            tc_fence_after();
            issue_sketch<R>(tm, smem + L::X, smem + L::G);
            umma_commit(&sh.sk);
            for (int j = 0; j + 1 < NJs && ok; ++j) {
                // sketch of the next token tile, as soon as this tile's half sketches are read out
                ok = mbar_wait(&sh.mread, j & 1, status, kErrState);
                ok = ok && mbar_wait(&sh.fullx[(j + 1) % NX], ((j + 1) / NX) & 1, status, kErrTma);
                tc_fence_after();
                issue_sketch<R>(tm, smem + L::X + ((j + 1) % NX) * 16384, smem + L::G);
                umma_commit(&sh.sk);
                // rows of tile j + 2.  Two slots: sketch j has completed (it was read), but its half sketches leave first;
                // three: those of tile j - 1 have left
                if (hl && NX == 3) bulk_wait_read();
                if (ok && (!hl || NX == 3) && j + 2 < NJs) load_x(j + 2);
                // values of the next token tile: their slot held tile j-1
                if (j >= 1) ok = ok && mbar_wait(&sh.yfree[(j + 1) & 1], ((j - 1) >> 1) & 1, status, kErrState);
                if (ok) load_y(j + 1);            // (a wait that gave up: nothing more is asked for or stored)
                if (hl) store_hl(j);
                if (hl && NX == 2) {
                    bulk_wait_read();
                    if constexpr (R == 64) mbar_arrive(&sh.hlfree);
                    if (ok && j + 2 < NJs) load_x(j + 2);
                }
            }
            if (hl) { store_hl(NJs - 1); bulk_wait_read(); }
            // drain: every sketch GEMM has completed before tensor memory is released.  (A barrier
            // of its own: completing sh.sk once more, right behind the last sketch, could flip it
            // twice before a generator thread has looked.)
            umma_commit(&sh.drain[0]);
            mbar_wait(&sh.drain[0], 0, status, kErrMma);
        } else if (warp == 4 * (NWG + NSW) + 1 && elect_one()) {
            constexpr uint32_t idesc_state = idesc_bf16(128, 80, true, true);
            bool ok = true;
            int w = 0;                                    // feature tile number u comes from warpgroup w = u mod NWG, as its
            uint32_t w_par = 0;                           // tile number u / NWG: parity w_par
            const uint64_t ad0 = smem_desc(smem_u32(smem + L::A0), 16384, 1024, kSwz128);
            const uint64_t yd0 = smem_desc(smem_u32(smem + L::Y), L::Ext - L::Y, 1024, kSwz128);
            const uint64_t yd1 = smem_desc(smem_u32(smem + L::Y) + L::kYSlot, L::Ext + 32 - L::Y - L::kYSlot, 1024, kSwz128);
            const int ibase = init ? 0 : 1;               // completions of sh.accread before block 1's
            for (int j = 0; j < NJs && ok; ++j) {
                ok = mbar_spin(&sh.fully[j & 1], (j >> 1) & 1, status, kErrTma);
                if (y65 != nullptr) ok = ok && mbar_spin(&sh.ext[j & 1], (j >> 1) & 1, status, kErrState);
                // block boundary: the store warpgroup has taken (or, for a start from earlier runs,
                // written) the accumulators' values before anything is added to them
                const bool boundary = mode != kModeTotal && (j % tpb == 0) && (j > 0 || init);
                const bool block_end = mode != kModeTotal ? ((j + 1) % tpb == 0) : (j == NJs - 1);
                const uint64_t yd = (j & 1) ? yd1 : yd0;
                const uint32_t acc0 = (j > 0 || init) ? 1u : 0u;
                static_for<0, TN>([&](auto ic) {
                    constexpr int I = decltype(ic)::value;
                    // the store warpgroup has taken this accumulator's values for the boundary
                    if (boundary) ok = ok && mbar_spin(&sh.accread[I], ((j / tpb) - ibase) & 1, status, kErrState);
                    ok = ok && mbar_spin(&sh.aready[w], w_par, status, kErrState);
                    const uint64_t ad = desc_off(ad0, w * 32768);
                    tc_fence_after();
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        umma_ss(tm + kAcc + 80 * I, desc_off(ad, k * 2048), desc_off(yd, k * 2048), idesc_state, k > 0 ? 1u : acc0);
                    umma_commit(&sh.afree[w]);
                    // last token tile of a block: this accumulator is complete, and the store
                    // warpgroup may take it while the remaining tiles are still being issued
                    if (block_end) umma_commit(&sh.accfull[I]);
                    if (++w == NWG) { w = 0; w_par ^= 1; }
                });
                umma_commit(&sh.yfree[j & 1]);
            }
            // drain: every state GEMM has completed before tensor memory is released
            umma_commit(&sh.drain[1]);
            mbar_wait(&sh.drain[1], 0, status, kErrMma);
        }
    } else if (wg >= NWG) {
        // ============================ store warpgroups ============================
        // (the tiles are dealt to them in turn)
        // Tiles leave through shared memory: a warp's 32 rows of 160 B are one contiguous 5 KB
        // piece of the state array, which goes out as one bulk copy.  (Rows stored by their threads directly would be
        // 10 scattered 16-byte stores each: the L1 data path, which the MMA operands and the generators' tiles also
        // go through, is this kernel's busiest unit.)  One body for all tiles: the kernel is short of instruction cache.
        const uint32_t lane_tm = tm + ((uint32_t)((warp % 4) * 32) << 16);
        const int sw = wg - NWG;
        uint8_t* stage = smem + L::St + sw * (128 * 160);
        // totals: the raw fp32 accumulators at the end of the run
        auto dump_totals = [&](uint32_t parity) {
            static_for<0, TN>([&](auto ic) {
                constexpr int I = decltype(ic)::value;
                if (NSW > 1 && I % NSW != sw) return;
                mbar_wait(&sh.accfull[I], parity, status, kErrMma);
                tc_fence_after();
                float4* out = reinterpret_cast<float4*>(tot + ((((size_t)bh * nseg + seg) * F::NT + (T0 + I)) * 128 + wt) * 80);
#pragma unroll
                for (int c0 = 0; c0 < 80; c0 += 16) {
                    uint32_t v[16];
                    tmem_ld16(lane_tm + kAcc + 80 * I + c0, v);
                    tmem_ld_wait();
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        out[c0 / 4 + q] = make_float4(__uint_as_float(v[4 * q]), __uint_as_float(v[4 * q + 1]),
                                                      __uint_as_float(v[4 * q + 2]), __uint_as_float(v[4 * q + 3]));
                }
            });
        };
        if (mode == kModeTotal) dump_totals(0);
        if (init) {
            // a later run starts from the sum of the earlier runs' totals: into the accumulators
            // first, then block 0 of the run is read back like every other block
            for (int I = sw; I < TN; I += NSW)
                state_init_acc(tot, (((size_t)bh * nseg + (seg - 1)) * F::NT + (T0 + I)) * 128 + wt, lane_tm + kAcc + 80 * I);
            tmem_st_wait();
        }
        for (int p = 0; p < ts && mode != kModeTotal; ++p) {
            const int pg = p0r + p;
            const int l = reverse ? (t - 1 - pg) : pg;
#pragma unroll 1
            for (int I = sw; I < TN; I += NSW) {
                if (p > 0) {
                    mbar_wait(&sh.accfull[I], (p - 1) & 1, status, kErrMma);
                    tc_fence_after();
                }
                const bool live = p > 0 || init;          // the accumulator holds values (else: zeros)
                const uint32_t acc = lane_tm + kAcc + 80 * I;
                // this thread's feature row: 80 bf16 = ten 16-byte pieces of the staging tile
                uint4* const grow = reinterpret_cast<uint4*>(S + (((size_t)bh * t + l) * F::FP + (size_t)(T0 + I) * 128 + wt) * 80);
                uint4* dst = L::kStaged ? reinterpret_cast<uint4*>(stage + wt * 160) : grow;
                uint32_t pk[33];                          // the row's 64 columns and the last one, formed before the staging tile is waited for
                if (live && (T0 + I) * 128 + wt / 32 * 32 < F::F) {       // (a warp's rows beyond the last feature: zeros)
                    // centred values, in fp32, without touching the operands (the mode only selects
                    // coefficients):  mode 1: sum phi (y - c)^T = H[:, :64] - H[:, 64] c^T
                    //                 mode 2: last column H[:, 64] - H[:, :64] c
                    // One store warpgroup, staged: all columns in one trip to tensor memory, the accumulator handed back before
                    // they are worked on.  Two (fewer registers), or rows stored directly: 16 columns at a time, the next on their way.
                    constexpr bool kAtOnce = NSW == 1 && L::kStaged;
                    uint32_t v[kAtOnce ? 4 : 2][16], last_raw;
                    tmem_ld1(acc + 64, last_raw);
#pragma unroll
                    for (int h = 0; h < (kAtOnce ? 4 : 1); ++h) tmem_ld16(acc + 16 * h, v[h]);
                    tmem_ld_wait();
                    auto handed_back = [&]() {
                        tc_fence_before();
                        if (wt % 32 == 0) mbar_arrive(&sh.accread[I]);
                    };
                    if (kAtOnce) handed_back();
                    const float last = __uint_as_float(last_raw);
                    const float k1s = center_mode == 1 ? -last : 0.f;
                    const f2 k1 = pack2(k1s, k1s);
                    f2 corr = 0ull;
                    // the row's pair weight (tc_features.cuh) goes into the stored state
                    const float wgt = F::weight((T0 + I) * 128 + wt);
                    const f2 w2 = pack2(wgt, wgt);
                    const bool pad = F::F % 32 != 0 && (T0 + I) * 128 + wt >= F::F;        // (such a row's sums may be anything)
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        if (!kAtOnce && h < 3) tmem_ld16(acc + 16 * (h + 1), v[(h + 1) & 1]);
                        const uint32_t (&u)[16] = v[kAtOnce ? h : h & 1];
#pragma unroll
                        for (int q = 0; q < 16; q += 4) {
                            const ulonglong2 c4 = *reinterpret_cast<const ulonglong2*>(&sh.cm[16 * h + q]);
                            const f2 x0 = fma2(k1, c4.x, pack2(u[q], u[q + 1])), x1 = fma2(k1, c4.y, pack2(u[q + 2], u[q + 3]));
                            if (center_mode == 2) corr = fma2(c4.y, x1, fma2(c4.x, x0, corr));
                            const f2 y0 = mul2(x0, w2), y1 = mul2(x1, w2);
                            pk[8 * h + q / 2] = pad ? 0u : pack_bf16(lo2(y0), hi2(y0));
                            pk[8 * h + q / 2 + 1] = pad ? 0u : pack_bf16(lo2(y1), hi2(y1));
                        }
                        if constexpr (!L::kStaged) {
                            dst[2 * h] = make_uint4(pk[8 * h], pk[8 * h + 1], pk[8 * h + 2], pk[8 * h + 3]);
                            dst[2 * h + 1] = make_uint4(pk[8 * h + 4], pk[8 * h + 5], pk[8 * h + 6], pk[8 * h + 7]);
                        }
                        if (!kAtOnce && h < 3) {
                            tmem_ld_wait16(v[(h + 1) & 1]);
                            if (h == 2) handed_back();        // last read of this accumulator
                        }
                    }
                    pk[32] = pad ? 0u : pack_bf16((last - (lo2(corr) + hi2(corr))) * wgt, 0.f);
                } else {
#pragma unroll
                    for (int q = 0; q < 33; ++q) pk[q] = 0u;
                    if constexpr (!L::kStaged) {
#pragma unroll
                        for (int q = 0; q < 8; ++q) dst[q] = make_uint4(0, 0, 0, 0);
                    }
                    if (live) { __syncwarp(); if (wt % 32 == 0) mbar_arrive(&sh.accread[I]); }
                }
                if constexpr (L::kStaged) {                   // the previous tile has left it
                    if (wt % 32 == 0) bulk_wait_read();
                    __syncwarp();
                }
                if constexpr (L::kStaged) {
#pragma unroll
                    for (int q = 0; q < 8; ++q) dst[q] = make_uint4(pk[4 * q], pk[4 * q + 1], pk[4 * q + 2], pk[4 * q + 3]);
                }
                dst[8] = make_uint4(pk[32], 0, 0, 0);
                dst[9] = make_uint4(0, 0, 0, 0);
                if constexpr (L::kStaged) {
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (wt % 32 == 0) {
                        bulk_store(grow, dst, 32 * 160);
                        bulk_commit();
                    }
                }
            }
        }
        if constexpr (L::kStaged) if (wt % 32 == 0) bulk_wait_read();
        if (SEG && mode == kModeFirst) dump_totals((ts - 1) & 1);
    } else {
        // ============================= generators =============================
        const uint32_t lane_tm = tm + ((uint32_t)((warp % 4) * 32) << 16);
        uint8_t* sA = smem + L::A0 + wg * 32768;
        uint32_t a_uses = 0;                              // times this warpgroup's buffer has been filled
        // last-column entry of this thread's token, requested one token tile ahead of its use
        float y_next = (y65 != nullptr && wg == 0) ? y65[(size_t)bh * n + tile_of(0) * 128 + wt] : 0.f;
        float d_next = fscale != nullptr ? fscale[(size_t)bh * n + tile_of(0) * 128 + wt] : 1.f;
        // Feature tiles are dealt to the warpgroups in turn, on across the token tiles: with TN not a multiple of NWG each has
        // its share over a few token tiles, and one with fewer tiles here starts on the next token tile meanwhile.
        int first = wg;                                   // this warpgroup's first tile of the token tile
        for (int j = 0; j < NJs; ++j, first = (first + (NWG - TN % NWG)) % NWG) {
            mbar_wait(&sh.sk, j & 1, status, kErrMma);
            tc_fence_after();
            FeatGen<R> gen;
            {
                float m[R];
                // features m_a m_b / d: both factors carry 1 / sqrt(d) (d requested a token tile ago)
                const float sc = rsqrtf(d_next);
                if (fscale != nullptr && j + 1 < NJs) d_next = fscale[(size_t)bh * n + tile_of(j + 1) * 128 + wt];
                // (the warpgroup last in turn, with the fewest tiles, also writes the half sketches out, over their dead X rows)
                const bool out = hl && first == NWG - 1;
                read_half_sketch<R>(lane_tm, m, out ? 1.f : sc, lin != 0);
                tc_fence_before();
                wg_barrier(wg);
                if (wt == 0) mbar_arrive(&sh.mread);
                if (out) {
                    // (r = 64: the second tile's single buffer has been stored)
                    if (R == 64 && j > 0) mbar_wait(&sh.hlfree, (j - 1) & 1, status, kErrState);
                    store_hl_rows<R>(smem + L::X + (j % L::kXSlots) * 16384, smem + L::Hl, m, wt);
                    fence_proxy_async_smem();
                    wg_barrier(wg);
                    if (wt == 0) mbar_arrive(&sh.hl[j & 1]);
                    if (fscale != nullptr) {
#pragma unroll
                        for (int c = 0; c < R; ++c) m[c] *= sc;
                    }
                }
                gen.init(m);
            }
            if (y65 != nullptr && wg == 0) {
                // last-column chunk of this token tile; its slot is free once tile j-2's MMAs are done
                if (j >= 2) mbar_wait(&sh.yfree[j & 1], ((j >> 1) - 1) & 1, status, kErrState);
                const float y = y_next;
                if (j + 1 < NJs) y_next = y65[(size_t)bh * n + tile_of(j + 1) * 128 + wt];
                *reinterpret_cast<bf16*>(smem + L::Ext + swz128_offset(wt, 2 * (j & 1))) =
                    __float2bfloat16_rn(y);
                fence_proxy_async_smem();
                wg_barrier(0);
                if (wt == 0) mbar_arrive(&sh.ext[j & 1]);
            }
            // this warpgroup's tiles first, first + NWG, ...
#pragma unroll 1
            for (int I = first; I < TN; I += NWG) {
                if (a_uses > 0) mbar_wait(&sh.afree[wg], (a_uses - 1) & 1, status, kErrMma);
                switch_chunk<0, TN>(I, [&](auto ic) {
                    constexpr int W0 = (T0 + decltype(ic)::value) * 64;           // the tile's first word
                    static_for<0, 16>([&](auto cc) {
                        constexpr int C = decltype(cc)::value;
                        // (rows beyond the last feature keep what an earlier tile left: their sums are never used)
                        if constexpr (2 * (W0 + 4 * C) < F::F) {
                            uint32_t pk[4];
                            gen.template words<W0 + 4 * C>(pk);
                            *reinterpret_cast<uint4*>(sA + (C / 8) * 16384 + swz128_offset(wt, C % 8)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                        }
                    });
                });
                fence_proxy_async_smem();
                wg_barrier(wg);
                if (wt == 0) mbar_arrive(&sh.aready[wg]);
                ++a_uses;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    cta_teardown(warp >= 4 * (NWG + NSW), warp - 4 * (NWG + NSW));
    if (warp == 0) tmem_dealloc(tm, 512);
}


#define PSK_STATE_PARAMS                                                                                            \
    const __grid_constant__ CUtensorMap mapX, const __grid_constant__ CUtensorMap mapY,                                    \
        const __grid_constant__ CUtensorMap mapH, const __grid_constant__ CUtensorMap mapH2, int want_hl, const uint8_t *__restrict__ gimg,  \
        int g_heads, int H, int n, int b, int t, const float *__restrict__ y65, const float *__restrict__ fscale,          \
        const float *__restrict__ cmean, int center_mode, int reverse, int nseg, int mode, int run0, int units,            \
        float *__restrict__ tot, bf16 *__restrict__ S, int lin, int *status
#define PSK_STATE_ARGS                                                                                              \
    mapX, mapY, mapH, mapH2, want_hl, gimg, g_heads, H, n, b, t, y65, fscale, cmean, center_mode, reverse, nseg, mode, run0, units, tot, S, lin, status

// The feature tiles of a head are dealt to SPLIT CTAs, each of which forms the half sketches anew.  blockIdx.z, the
// slowest index: CTAs that run at the same time then run the same specialised code (with the shares of a head side by
// side on neighbouring SMs the kernel took 1.5 times as long, for want of instruction cache).  r = 64 has 17 tiles and tensor memory for four accumulators beside the sketch columns.
// Store warpgroups: the walk stalls at a block boundary until the accumulators have been read, one tile after the other.  Two help
// where a share has two tiles and registers for them (r = 32 in three shares: 48 heads x 16 384, b = 256: 402 us per training step for both
// walks, one warpgroup that reads all columns at once 382, two 374); with five tiles a CTA (one share, 96 heads x 8192) the generators
// bound it (400, 394, 402), r = 16 has 212, 204, 212, and r = 64 no registers (1276, 1237, spills).  (Two shares at r = 32, with
// columns at once and 44 bytes of spill stores: 48 to 72 heads, training, 0.84 to 0.96 of before; the rule is the same for them.)
template <int R, int SPLIT> struct StateSplit {
    static constexpr int NT = Feat<R>::NT, kBase = NT / SPLIT, kMore = NT % SPLIT;
    __host__ __device__ static constexpr int tiles(int z) { return kBase + (z < kMore ? 1 : 0); }
    __host__ __device__ static constexpr int first(int z) { return z * kBase + (z < kMore ? z : kMore); }
    static constexpr int NWG = tiles(0) < 3 ? tiles(0) : 3, NSW = R == 32 && SPLIT == 3 ? 2 : 1, kThreads = 128 * (NWG + NSW) + 64;
};

template <int R, int SPLIT, bool SEG>
__global__ void __launch_bounds__(StateSplit<R, SPLIT>::kThreads) tc_state_kernel(PSK_STATE_PARAMS) {
    using P = StateSplit<R, SPLIT>;
    __shared__ StateShared<P::tiles(0), P::NWG> sh;
    static_for<0, SPLIT>([&](auto zc) {
        constexpr int Z = decltype(zc)::value;
        if (SPLIT == 1 || (int)blockIdx.z == Z) state_walk<R, P::first(Z), P::tiles(Z), P::NWG, P::NSW, SEG>(sh, PSK_STATE_ARGS);
    });
}

// Running sums of a head's run totals, in place: run s becomes the sum over the runs <= s.
__global__ void __launch_bounds__(256)
tc_state_scan_kernel(float4* __restrict__ tot, size_t elems, int nseg) {
    pdl_sync();
    const size_t e = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (e >= elems) return;
    float4* p = tot + (size_t)blockIdx.y * nseg * elems + e;
    float4 run = p[0];
    for (int k0 = 1; k0 < nseg - 1; k0 += 8) {
        float4 v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) if (k0 + q < nseg - 1) v[q] = p[(size_t)(k0 + q) * elems];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            if (k0 + q >= nseg - 1) break;
            run.x += v[q].x; run.y += v[q].y; run.z += v[q].z; run.w += v[q].w;
            p[(size_t)(k0 + q) * elems] = run;
        }
    }
}

// Sum of the run totals of a head, centred, weighted and rounded like a stored state: the single
// global state of non-causal attention, written as the head's only block.  A CTA takes 32 of the state's rows; its threads
// share the 10 KB of a run's total and finish the rows, one lane each, in shared memory.  (A thread per row that read its
// own 320 bytes of every total lived on the L1 cache, of which the row kernels' CTAs, waiting for this kernel on the same SMs
// with up to 227 KB of shared memory each SM, leave next to nothing: 24 heads x 4096, r = 16: 15 us alone and 48 to 85 in front of them.)
constexpr int kSumRows = 32, kSumPitch = 84;              // (floats; 16-byte steps of an odd number: no bank conflicts)
template <int R>
__global__ void __launch_bounds__(128)
tc_state_sum_kernel(const float* __restrict__ tot, int nseg, const float* __restrict__ cmean, int center_mode,
                    bf16* __restrict__ S) {
    pdl_sync();
    using F = Feat<R>;
    __shared__ __align__(16) float rows[kSumRows * kSumPitch];
    __shared__ float cm[64];
    const int row0 = blockIdx.x * kSumRows, bh = blockIdx.y, tid = threadIdx.x;
    constexpr int kVec = kSumRows * 20 / 128;             // 16-byte pieces of the CTA's rows per thread
    if (tid < 64) cm[tid] = cmean != nullptr ? cmean[(size_t)bh * 64 + tid] : 0.f;
    if (row0 < F::F) {                                    // (rows beyond the last feature may hold anything: zeros are stored)
        float4 v[kVec];
#pragma unroll
        for (int q = 0; q < kVec; ++q) v[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4* src = reinterpret_cast<const float4*>(tot + ((size_t)bh * nseg * F::FP + row0) * 80) + tid;
#pragma unroll 2
        for (int s = 0; s < nseg; ++s) {
#pragma unroll
            for (int q = 0; q < kVec; ++q) {
                const float4 x = src[(size_t)s * (F::FP * 20) + 128 * q];
                v[q].x += x.x; v[q].y += x.y; v[q].z += x.z; v[q].w += x.w;
            }
        }
#pragma unroll
        for (int q = 0; q < kVec; ++q) {
            const int e = tid + 128 * q;
            *reinterpret_cast<float4*>(rows + (e / 20) * kSumPitch + 4 * (e % 20)) = v[q];
        }
    }
    __syncthreads();
    if (tid < kSumRows) {
        const int row = row0 + tid;
        float* const mine = rows + tid * kSumPitch;
        uint32_t pk[40];
#pragma unroll
        for (int c = 0; c < 40; ++c) pk[c] = 0u;
        if (row < F::F) {
            const float wgt = F::weight(row), last = mine[64];
            float corr = 0.f;
#pragma unroll
            for (int c = 0; c < 64; c += 4) {
                const float4 u = *reinterpret_cast<const float4*>(mine + c);
                const float x0 = center_mode == 1 ? u.x - last * cm[c] : u.x, x1 = center_mode == 1 ? u.y - last * cm[c + 1] : u.y;
                const float x2 = center_mode == 1 ? u.z - last * cm[c + 2] : u.z, x3 = center_mode == 1 ? u.w - last * cm[c + 3] : u.w;
                if (center_mode == 2) {
                    corr += cm[c] * x0 + cm[c + 1] * x1;
                    corr += cm[c + 2] * x2 + cm[c + 3] * x3;
                }
                pk[c / 2] = pack_bf16(x0 * wgt, x1 * wgt);
                pk[c / 2 + 1] = pack_bf16(x2 * wgt, x3 * wgt);
            }
            pk[32] = pack_bf16((last - corr) * wgt, 0.f);
        }
#pragma unroll
        for (int c = 0; c < 10; ++c) reinterpret_cast<uint4*>(mine)[c] = make_uint4(pk[4 * c], pk[4 * c + 1], pk[4 * c + 2], pk[4 * c + 3]);
    }
    __syncthreads();
    uint4* out = reinterpret_cast<uint4*>(S + ((size_t)bh * F::FP + row0) * 80);
    for (int e = tid; e < kSumRows * 10; e += 128)
        out[e] = *reinterpret_cast<const uint4*>(rows + (e / 10) * kSumPitch + 4 * (e % 10));
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
struct StateArgs {
    const float *y65, *fscale, *cmean;
    int center_mode;
    bool reverse;
    int nseg, mode, run0, runs;        // runs [run0, run0 + runs) of nseg are launched
    float* tot;
    bf16* S;
    CUtensorMap mH[2];                 // where the [hi | lo] half sketches go, if anywhere
    bool want_hl;
};

// units a head's sequence can be cut into: blocks (a run starts at a block boundary), or 128-token
// tiles when there are no blocks to respect
int state_units(const Dims& d) { return d.noncausal ? d.n / 128 : d.t; }

// CTAs per head and run, and runs per head.  Estimated time in nanoseconds: a CTA's walk of its run, times the
// rounds in which the grid fills the SMs.  `step`, `boundary`: measured time of a 128-token tile and of writing
// the states out at a block boundary, for the largest share of a split (12 heads, n = 32 768, b = 256 and 4096; taken before elected
// MMA issue, unrolled features and the second store warpgroup, which made all of them shorter, and not again: none of 270
// sketched shapes tried got slower with the plans they choose);
// `mean`: the average share in percent of the largest.  Where more CTAs than SMs are wanted, the shares of a
// head get in each other's way for r <= 32 (15 % on 96 heads).  A run's start and end cost about 6 us, its start value
// 4 us, the launch between the two passes over the runs 8 us.
struct StatePlan { int split, nseg; };
struct SplitCost { int split, step, boundary, mean; };
constexpr SplitCost kCost16[] = {{1, 1350, 600, 100}, {2, 1140, 200, 100}};
constexpr SplitCost kCost32[] = {{1, 2950, 1300, 100}, {2, 1920, 800, 85}, {3, 1330, 640, 92}, {5, 1220, 220, 100}};
constexpr SplitCost kCost64[] = {{5, 3190, 2700, 85}, {6, 2110, 1840, 94}, {9, 1460, 540, 94}};

StatePlan state_plan(const Dims& d) {
    constexpr long kSMs = 148, kStart = 6000, kInit = 4000, kBetween = 8000;
    const SplitCost* cost = d.r == 16 ? kCost16 : (d.r == 32 ? kCost32 : kCost64);
    const int ncost = d.r == 16 ? 2 : (d.r == 32 ? 4 : 3), units = state_units(d);
    const long upt = d.n / 128 / units;
    auto rounds = [&](long ctas, const SplitCost& c, long walk) {
        return ctas <= kSMs ? walk : ((ctas + kSMs - 1) / kSMs) * walk * c.mean / 100 * (d.r <= 32 && c.split > 1 ? 115 : 100) / 100;
    };
    int lo = 1, hi = units < 64 ? units : 64;
    if (d.seq_segments > 0) lo = hi = (d.seq_segments <= units && units % d.seq_segments == 0) ? d.seq_segments : 1;
    StatePlan p{cost[0].split, 1};
    long best = -1;
    for (int i = 0; i < ncost; ++i)
        for (int s = lo; s <= hi; ++s) {
            const SplitCost& c = cost[i];
            const long run = (units + s - 1) / s, tiles = run * upt, ctas = (long)d.BH() * c.split;
            long t;
            if (d.noncausal) t = rounds(ctas * s, c, tiles * c.step + kStart);
            else if (s == 1) t = rounds(ctas, c, tiles * c.step + run * c.boundary + kStart);
            else t = 2 * rounds(ctas * (s - 1), c, tiles * c.step + run * c.boundary + kStart + kInit / 2) + kBetween;
            if (best < 0 || t < best - best / 20) { best = t; p = StatePlan{c.split, s}; }       // (more CTAs have to pay clearly)
        }
    return p;
}

template <int R, int SPLIT>
cudaError_t launch_split(const Dims& d, const CUtensorMap& mX, const CUtensorMap& mY, const uint8_t* gimg,
                         const StateArgs& a, int* status, cudaStream_t s, int* launches) {
    using P = StateSplit<R, SPLIT>;
    constexpr size_t smem = StateSmem<R, P::NWG, P::NSW>::total + 1024;
    // Programmatic dependence saves a short walk 2 to 6 us (forward of 12 heads x 16 512, two passes over 11 runs: 185 -> 180 us;
    // 12 heads x 1024, training: 88 -> 83).  But CTAs that start early settle on the SMs that happen to be free, shares of a head
    // side by side, and neighbours that run different code are slow (StateSplit): where the shares fill the GPU that costs a
    // training step 3 to 25 % (r = 32, 48 heads x 1024, 2048, 2688: 135, 214, 278 us against 149, 250, 308; r = 64, 16 heads
    // x 2048: 293 against 366; 108 CTAs: 170 against 178; 60 CTAs gain).  Long walks (over 24 tiles; at 64, r = 32, 48 heads: 715
    // against 776) take longer than the launch either way.
    const bool early = d.n / 128 / a.nseg <= 24 && (SPLIT == 1 || (long)d.BH() * a.runs * SPLIT <= 74);
    auto kern = a.nseg > 1 || a.mode != kModePrefix ? tc_state_kernel<R, SPLIT, true> : tc_state_kernel<R, SPLIT, false>;
    PSK_TRY((set_smem(kern, smem)));
    prof_begin(a.mode == kModePrefix ? "tc_state_kernel" : "tc_state_total_kernel", s);
    launch_pdl_if(early, kern, dim3(d.BH(), a.runs, SPLIT), P::kThreads, smem, s, mX, mY, a.mH[0], a.mH[1], a.want_hl ? 1 : 0, gimg, d.g_heads, d.H, d.n, d.b, d.t, a.y65, a.fscale,
                  a.cmean, a.center_mode, a.reverse ? 1 : 0, a.nseg, a.mode, a.run0, state_units(d), a.tot, a.S, d.sketch_linear ? 1 : 0, status);
    prof_end(s);
    ++*launches;
    return cudaGetLastError();
}

template <int R>
cudaError_t launch_states(const Dims& d, const CUtensorMap& mX, const CUtensorMap& mY, const uint8_t* gimg,
                          const StateArgs& a, int* status, cudaStream_t s, int* launches) {
    const int split = state_plan(d).split;
    if constexpr (R == 64) {
        if (split == 9) return launch_split<R, 9>(d, mX, mY, gimg, a, status, s, launches);
        if (split == 6) return launch_split<R, 6>(d, mX, mY, gimg, a, status, s, launches);
        return launch_split<R, 5>(d, mX, mY, gimg, a, status, s, launches);
    } else if constexpr (R == 32) {
        if (split == 5) return launch_split<R, 5>(d, mX, mY, gimg, a, status, s, launches);
        if (split == 3) return launch_split<R, 3>(d, mX, mY, gimg, a, status, s, launches);
        if (split == 2) return launch_split<R, 2>(d, mX, mY, gimg, a, status, s, launches);
        return launch_split<R, 1>(d, mX, mY, gimg, a, status, s, launches);
    } else {
        if (split == 2) return launch_split<R, 2>(d, mX, mY, gimg, a, status, s, launches);
        return launch_split<R, 1>(d, mX, mY, gimg, a, status, s, launches);
    }
}

template <int R>
cudaError_t states_impl(const Dims& d, const CUtensorMap& mX, const CUtensorMap& mY, const uint8_t* gimg, const float* y65,
                        const float* fscale, const float* cmean, int center_mode, bf16* S, bf16* hl, bool reverse, float* tot,
                        int* status, cudaStream_t s, int* launches) {
    const int nseg = tc_state_segments(d);
    StateArgs a{y65, fscale, cmean, center_mode, reverse, nseg, kModePrefix, 0, nseg, tot, S, {mX, mX}, hl != nullptr && !d.noncausal};
    if (a.want_hl && !tc_map_hilo(d, hl, a.mH)) return cudaErrorInvalidValue;
    if (d.noncausal) {
        // one global state per head: totals of every run, then their sum in the stored format
        a.mode = kModeTotal; a.cmean = nullptr; a.center_mode = 0;
        PSK_TRY((launch_states<R>(d, mX, mY, gimg, a, status, s, launches)));
        prof_begin("tc_state_sum_kernel", s);
        launch_pdl(tc_state_sum_kernel<R>, dim3(Feat<R>::FP / kSumRows, d.BH()), 128, 0, s, tot, nseg, cmean, center_mode, S);
        prof_end(s);
        ++*launches;
        return cudaGetLastError();
    }
    if (nseg == 1) return launch_states<R>(d, mX, mY, gimg, a, status, s, launches);
    a.mode = kModeFirst; a.runs = nseg - 1;              // (nothing starts after the last run)
    PSK_TRY((launch_states<R>(d, mX, mY, gimg, a, status, s, launches)));
    if (nseg > 2) {
        const size_t elems = (size_t)Feat<R>::NT * 128 * 20;
        prof_begin("tc_state_scan_kernel", s);
        launch_pdl(tc_state_scan_kernel, dim3((unsigned)((elems + 255) / 256), d.BH()), 256, 0, s, reinterpret_cast<float4*>(tot), elems, nseg);
        prof_end(s);
        ++*launches;
        PSK_TRY(cudaGetLastError());
    }
    a.mode = kModePrefix; a.run0 = 1;
    return launch_states<R>(d, mX, mY, gimg, a, status, s, launches);
}

}  // namespace

int tc_state_segments(const Dims& d) { return state_plan(d).nseg; }

size_t tc_state_total_bytes(const Dims& d) {
    const int nseg = tc_state_segments(d);
    if (nseg <= 1 && !d.noncausal) return 0;
    const size_t nt = d.r == 16 ? Feat<16>::NT : (d.r == 32 ? Feat<32>::NT : Feat<64>::NT);
    return (size_t)d.BH() * nseg * nt * 128 * 80 * sizeof(float);
}

cudaError_t tc_states(const Dims& d, const CUtensorMap& mX, const CUtensorMap& mY, const uint8_t* gimg,
                      const float* y65, const float* fscale, const float* cmean, int center_mode, bf16* S, bf16* hl, bool reverse,
                      float* tot, int* status, cudaStream_t s, int* launches) {
    switch (d.r) {
        case 16: return states_impl<16>(d, mX, mY, gimg, y65, fscale, cmean, center_mode, S, hl, reverse, tot, status, s, launches);
        case 32: return states_impl<32>(d, mX, mY, gimg, y65, fscale, cmean, center_mode, S, hl, reverse, tot, status, s, launches);
        case 64: return states_impl<64>(d, mX, mY, gimg, y65, fscale, cmean, center_mode, S, hl, reverse, tot, status, s, launches);
    }
    return cudaErrorInvalidValue;
}

}  // namespace psk
