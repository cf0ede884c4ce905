// Device helpers shared by the tensor-core kernels (forward and backward translation units).
#pragma once

#include "psk_internal.cuh"
#include "tc_features.cuh"

#include <type_traits>

namespace psk {

typedef __nv_bfloat16 bf16;

// host: tensor maps (defined in psk_tc.cu)
// [B,H,n,64] bf16 rows, box 128 rows x 64 columns, 128-byte swizzle
bool tc_map_rows(CUtensorMap* m, const void* base, int B, int H, int n, int64_t sb, int64_t sh, int64_t sn);
// states S[nblk][80][FP] bf16, box 80 rows x 64 features
bool tc_map_states(CUtensorMap* m, const void* base, int FP, int64_t nblk);
// row-major [rows][cols] bf16 matrix, box box_rows x 64 columns
bool tc_map_2d(CUtensorMap* m, const void* base, int cols, int64_t rows, int box_rows);
// contiguous [outer][rows][cols] bf16, box box_rows x box_cols
bool tc_map_3d(CUtensorMap* m, const void* base, int cols, int64_t rows, int64_t outer, int box_cols, int box_rows);
// per-block states of every head + prefix (reverse = false) or suffix (reverse = true) scan
// center_mode 0: states as they are; 1: values centred by the per-head vector cmean
// (columns < 64 become H[:, c] - cmean[c] H[:, 64]); 2: last column becomes H[:, 64] - H[:, :64] cmean.
// `tot`: scratch of tc_state_total_bytes(d) bytes for the segment totals (may be null when that is 0).
// `hl` (may be null): the half sketches of X's rows as [hi | lo] rows, which the row kernels load as
// the other side's score operand; contiguous [B][H][n][64 HiLoTiles].
// Non-causal (d.noncausal): one state per head, the sum over the whole sequence, stored as block 0.
cudaError_t tc_states(const Dims& d, const CUtensorMap& mX, const CUtensorMap& mY, const uint8_t* gimg,
                      const float* y65, const float* fscale, const float* cmean, int center_mode, bf16* S, bf16* hl, bool reverse,
                      float* tot, int* status, cudaStream_t s, int* launches);
// maps of the 64-column tiles of such an array (the second: r = 64 only, else a copy of the first)
bool tc_map_hilo(const Dims& d, const void* hl, CUtensorMap (&m)[2]);
// runs a head's blocks are cut into by the state kernel (1 = one CTA group walks the whole head)
int tc_state_segments(const Dims& d);
size_t tc_state_total_bytes(const Dims& d);
// the backward's recomputation of the forward rows: writes y65, e65h (see tc_fwd_out_kernel)
// (mK: the keys' [hi | lo] half sketches, with mQraw their second 64 columns for r = 64; the raw key rows with exact
// same-block weights, and then, with a given half sketch, mQraw the raw query rows)
cudaError_t tc_recompute(const Dims& d, const CUtensorMap& mQ, const CUtensorMap& mQraw, const CUtensorMap& mK, const CUtensorMap& mV,
                         const CUtensorMap& mZ, const uint8_t* gimg, const float* cmean, const float* denom,
                         const bf16* dO, float* y65, float* e65h, int* status, cudaStream_t s, int* launches);
// gimg[g] = [G1 | G2]^T of sketch-matrix set g as the shared-memory image of the sketch GEMM's B operand
// (2r rows x 128 B, K-major, 128-byte swizzle): the kernels fetch it with one bulk copy
// (d.sketch_linear: the image of [I | 0] or [I; I | 0] instead, G1 and G2 are not read).
// cmean[bh][c] (unless null) = mean of V[bh][:, c] over up to 1024 evenly spaced rows (deterministic).
// Clears the status word if d.clear_status.
cudaError_t tc_prologue(const Dims& d, const void* G1, const void* G2, uint8_t* gimg, const void* V, float* cmean, int* status,
                        cudaStream_t s, int* launches);

// Scratch layout of the tensor-core path.
struct TcWorkspace { size_t status, vmean, gimg, tot, Z, Sk, Rst, y65, e65h, Oc, Sq, total; };

// the row kernels read the other side's half sketches from an array of the state kernel's (otherwise: the rows
// themselves are given half sketches, or the same-block weights come from the raw rows, or there are no blocks)
inline bool tc_hilo_rows(const Dims& d) { return !d.local && !d.sketch_linear && !d.noncausal; }

template <int R>
inline TcWorkspace tc_ws(const Dims& d, bool backward) {
    TcWorkspace w{};
    const size_t st = (size_t)d.BH() * (d.noncausal ? 1 : d.t) * tc::Feat<R>::FP * 80 * sizeof(bf16);
    const size_t rows = (size_t)d.BH() * d.n;
    size_t off = 0;
    w.status = off; off += kStatusBytes;
    w.vmean = off; off += align_up((size_t)d.BH() * 64 * sizeof(float));
    w.gimg = off; off += align_up((size_t)d.g_heads * 2 * R * 128);
    w.tot = off; off += align_up(tc_state_total_bytes(d));
    w.Z = off; off += align_up(st);
    const size_t hl = tc_hilo_rows(d) ? align_up(rows * (R <= 32 ? 64 : 128) * sizeof(bf16)) : 0;
    w.Sk = off; off += hl;
    if (backward) {
        w.Sq = off; off += hl;
        w.Rst = off; off += align_up(st);
        w.y65 = off; off += align_up(rows * sizeof(float));
        w.e65h = off; off += align_up(rows * sizeof(float));
        if (d.keep_states) { w.Oc = off; off += align_up(rows * 64 * sizeof(bf16)); }   // forward's O - c
    }
    w.total = off;
    return w;
}

#define PSK_TRY(x) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) return e_; } while (0)

template <typename Kern>
inline cudaError_t set_smem(Kern k, size_t bytes) {
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

namespace tc {

constexpr int kErrTma = 1, kErrMma = 2;

// barrier among the 128 row threads (warps 0-3) of a kernel whose fifth warp issues the MMAs;
// only where every row thread is certain to arrive (never inside a loop a failed wait can leave)
__device__ __forceinline__ void consumer_barrier() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

__device__ __forceinline__ uint8_t* align1024(uint8_t* p) {
    return p + ((1024u - (smem_u32(p) & 1023u)) & 1023u);
}

// [G1 | G2]^T as a K-major, 128-byte-swizzled tile: row n (< 2R) holds sketch column n over the 64
// head dimensions.  B operand of the sketch GEMM X [G1 | G2]; built once per call by
// tc_prologue_kernel, then copied into shared memory as it is.
template <int R>
struct GImage { static constexpr uint32_t bytes = 2 * R * 128; };

// Sketch GEMM D[128 tokens x 2R] = X_tile [G1 | G2], 4 K steps of 16 over the head dimension.
template <int R>
__device__ __forceinline__ void issue_sketch(uint32_t d_tmem, const uint8_t* sX, const uint8_t* sG) {
    constexpr uint32_t idesc = idesc_bf16(128, 2 * R, false, false);
#pragma unroll
    for (int k = 0; k < 4; ++k)
        umma_ss(d_tmem, desc_off(smem_desc(smem_u32(sX), 0, 1024, kSwz128), k * 32),
                desc_off(smem_desc(smem_u32(sG), 0, 1024, kSwz128), k * 32), idesc, k > 0);
}

// m[c] = A1[c] A2[c] / sqrt(R) from the sketch accumulator (this thread's lane).
// (`scale`: an extra factor on every entry, folded into the constant)
// `linear`: the half sketch is given, not formed here: the "rows to sketch" are the half sketch
// itself (degree 2: m = x), or its two bf16 terms side by side ([hi | lo]), and the first half of the
// sketch GEMM against an identity-like matrix ([I], [I; I]) just carries it into tensor memory in
// fp32: m[c] = A1[c].
template <int R>
__device__ __forceinline__ void read_half_sketch(uint32_t lane_tmem, float (&m)[R], float scale = 1.f, bool linear = false) {
    const float rs = linear ? scale : rsqrtf((float)R) * scale;
#pragma unroll
    for (int c0 = 0; c0 < R; c0 += 16) {
        uint32_t a1[16], a2[16];
        tmem_ld16(lane_tmem + c0, a1);
        tmem_ld16(lane_tmem + R + c0, a2);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 16; ++j) m[c0 + j] = __uint_as_float(a1[j]) * (linear ? 1.f : __uint_as_float(a2[j])) * rs;
    }
}

// An fp32 half-sketch entry is split into two bf16 terms, m = hi + lo (+ O(2^-17) |m|), and scores s = m(q).m(k) are
// formed as hi.hi + lo.hi + hi.lo: a score is a cancelling sum, so rounding m to a single bf16 would cost several
// percent on rows with few keys.
// The split half sketch as [hi | lo] columns (2R of them) in ceil(2R/64) tiles of
// [128 rows x 128 B], 128-byte-swizzled, zero beyond 2R.  Tile 0 starts with the R `hi` columns,
// so it doubles as the MN-major B operand (N = 64, columns >= R ignored) of the dM GEMMs.
template <int R>
struct HiLoTiles { static constexpr int N = (2 * R + 63) / 64; };
// Tiles of 64 columns that a half sketch takes as a score operand: [hi | lo] of r entries each; one of the rows
// themselves where they are the half sketch (degree 2: r = h, given to the last bit, no lo).
template <int R, bool LIN> struct OthTiles { static constexpr int N = (LIN && R == 64) ? 1 : HiLoTiles<R>::N; };

// (TILES: how many of them are wanted)
template <int R, int TILES = HiLoTiles<R>::N>
__device__ __forceinline__ void store_hilo_tiles(uint8_t* dst, const float (&m)[R], int row) {
    auto chunk = [&](int c) { return reinterpret_cast<uint4*>(dst + (c / 8) * 16384 + swz128_offset(row, c % 8)); };
#pragma unroll
    for (int ch = 0; ch < R / 8; ++ch) {
        uint32_t h[4], l[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float a = m[8 * ch + 2 * i], b = m[8 * ch + 2 * i + 1];
            h[i] = pack_bf16(a, b);
            l[i] = pack_bf16(a - __uint_as_float(h[i] << 16), b - __uint_as_float(h[i] & 0xffff0000u));
        }
        *chunk(ch) = make_uint4(h[0], h[1], h[2], h[3]);
        if (R / 8 + ch < TILES * 8) *chunk(R / 8 + ch) = make_uint4(l[0], l[1], l[2], l[3]);
    }
#pragma unroll
    for (int ch = R / 4; ch < TILES * 8; ++ch) *chunk(ch) = make_uint4(0, 0, 0, 0);
}

}  // namespace tc
}  // namespace psk
