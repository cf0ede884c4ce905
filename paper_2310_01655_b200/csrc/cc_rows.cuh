// Block states and row kernels of the CUDA-core path (fp32 arithmetic), in terms of the 64 x 64
// products of cc_gemm.cuh.
//
// Features.  m (x) m has one distinct entry per unordered pair {a, b}.  The half sketch is cut into
// groups of eight coordinates, and a CHUNK is one pair of groups ab <= bb: 64 features
// f = 8 b' + a' (a = 8 ab + a', b = 8 bb + b').  Chunks with ab < bb stand for both orders and their
// state rows carry the weight 2, the diagonal ones hold both orders themselves: r/8 (r/8 + 1) / 2
// chunks, 640 stored features instead of 1024 for r = 32.  A chunk's features are products of 16
// half-sketch entries that are already in registers or shared memory.
// States in memory: S[BH][t][chunk][64 f][68] fp32: 64 value columns, the normaliser column, padding.
#pragma once

#include "cc_gemm.cuh"

namespace psk {
namespace cc {

struct Slice {              // addressing of one [B,H,n,h] tensor
    int H; int64_t sb, sh, sn;
    __device__ int64_t row(int bh, int i) const {
        return (int64_t)(bh / H) * sb + (int64_t)(bh % H) * sh + (int64_t)i * sn;
    }
};

// Rows [Y | y65]: either 68-column rows of scratch, or the caller's own fp32 values with the last
// column all ones (`ones`).
struct YRows { const float* p; Slice sl; int ones; };

template <int R> constexpr int kChunks = (R / 8) * (R / 8 + 1) / 2;
constexpr int kChunkFloats = 64 * kLd;

template <int R>
__device__ __forceinline__ void chunk_pair(int c, int& ab, int& bb) {
    constexpr int NB = R / 8;
    ab = 0;
    while (c >= NB - ab) { c -= NB - ab; ++ab; }
    bb = ab + c;
}

// 64 rows of [Y | y65] into shared memory [64][kLd] by `nthr` threads (asynchronous; the caller
// commits and waits).  With `ones` the last column is not written here.
__device__ __forceinline__ void load_y_rows(float* dst, const YRows& y, int bh, int i0, int tid, int nthr) {
    const int per = y.ones ? 16 : 17;
    for (int e = tid; e < 64 * per; e += nthr) {
        const int rr = e / per, c = e % per;
        cp16(dst + rr * kLd + 4 * c, y.p + y.sl.row(bh, i0 + rr) + 4 * c);
    }
}

// ---------------------------------------------------------------------------
// Block states (Section 3.1): H_l = phi'(M_l)^T [Y_l | y65], one chunk per 64-thread group, G
// groups (chunks) per CTA share the block's rows in shared memory (two tiles of 64 rows, the
// next one in flight).  Block l's state goes to the slot whose prefix (suffix) sum it enters
// first, l + 1 (l - 1), so that the scan that follows is an inclusive one in place.
// grid (ceil(chunks / G), t - 1, BH).  Bound by the FMA pipe: per token and thread 32 packed FMAs
// beside 4 multiplies, 8 moves and 5 loads.
// ---------------------------------------------------------------------------
template <int R> constexpr int kStateGroups = R == 16 ? 3 : (R == 32 ? 2 : 4);     // divides the chunk count
template <int R> constexpr size_t kStateSmem = 2 * (64 * (R + 4) + kUnit) * sizeof(float);

template <int R>
__global__ void __launch_bounds__(64 * kStateGroups<R>, R == 64 ? 2 : (R == 32 ? 4 : 2))
cc_state_kernel(const float* __restrict__ M, YRows y, int n, int b, int t, int reverse, float* __restrict__ S) {
    pdl_sync();
    extern __shared__ __align__(16) float smem[];
    constexpr int G = kStateGroups<R>, NT = 64 * G, LD = R + 4, kBuf = 64 * LD + kUnit;
    const int tid = threadIdx.x, grp = tid / 64, lane = tid % 64, ry = lane / 8, cx = lane % 8;
    const int l = blockIdx.y + (reverse ? 1 : 0), bh = blockIdx.z;
    const int chunk = blockIdx.x * G + grp;
    const bool live = chunk < kChunks<R>;
    int ab = 0, bb = 0;
    if (live) chunk_pair<R>(chunk, ab, bb);
    auto load = [&](int k) {
        float* dst = smem + (k & 1) * kBuf;
        const float* src = M + ((size_t)bh * n + (size_t)l * b + k * 64) * R;
        for (int e = tid; e < 64 * R / 4; e += NT) cp16(dst + (e / (R / 4)) * LD + 4 * (e % (R / 4)), src + 4 * e);
        load_y_rows(dst + 64 * LD, y, bh, l * b + k * 64, tid, NT);
        cp_commit();
    };
    load(0);
    if (y.ones)
        for (int e = tid; e < 128; e += NT) smem[(e / 64) * kBuf + 64 * LD + (e % 64) * kLd + 64] = 1.f;
    Acc acc;
    acc.zero();
    f2 ext[4] = {0ull, 0ull, 0ull, 0ull};
    const int nk = b / 64;
    for (int k = 0; k < nk; ++k) {
        if (k + 1 < nk) { load(k + 1); cp_wait<1>(); } else { cp_wait<0>(); }
        __syncthreads();
        if (live) {
            const float* sM = smem + (k & 1) * kBuf;
            const float* sY = sM + 64 * LD;
            const float* pa = sM + 8 * ab + ry;
            const float* pb = sM + 8 * bb;
#pragma unroll 4
            for (int j = 0; j < 64; ++j) {
                const float ma = pa[j * LD];
                const f2 ma2 = pack2(ma, ma);
                f2 phi[4];
                load_rows8(phi, pb + j * LD);
#pragma unroll
                for (int i = 0; i < 4; ++i) phi[i] = mul2(phi[i], ma2);
                acc.step(phi, lds22(sY + j * kLd + 4 * cx), lds22(sY + j * kLd + 32 + 4 * cx));
            }
            // the last column: the eight threads of a feature share the tokens
#pragma unroll 2
            for (int j = cx; j < 64; j += 8) {
                const float my = pa[j * LD] * sY[j * kLd + 64];
                const f2 my2 = pack2(my, my);
                f2 mb[4];
                load_rows8(mb, pb + j * LD);
#pragma unroll
                for (int i = 0; i < 4; ++i) ext[i] = fma2(mb[i], my2, ext[i]);
            }
        }
        __syncthreads();
    }
    if (!live) return;
    const float w = ab == bb ? 1.f : 2.f;
    float* out = S + (((size_t)bh * t + (reverse ? l - 1 : l + 1)) * kChunks<R> + chunk) * kChunkFloats;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        float e = (i & 1) ? hi2(ext[i / 2]) : lo2(ext[i / 2]);
        e += __shfl_xor_sync(0xffffffffu, e, 1);
        e += __shfl_xor_sync(0xffffffffu, e, 2);
        e += __shfl_xor_sync(0xffffffffu, e, 4);
        float* row = out + (8 * i + ry) * kLd;
        *reinterpret_cast<float4*>(row + 4 * cx) = make_float4(w * acc.at(i, 0), w * acc.at(i, 1), w * acc.at(i, 2), w * acc.at(i, 3));
        *reinterpret_cast<float4*>(row + 32 + 4 * cx) = make_float4(w * acc.at(i, 4), w * acc.at(i, 5), w * acc.at(i, 6), w * acc.at(i, 7));
        if (cx == 0) *reinterpret_cast<float4*>(row + 64) = make_float4(w * e, 0.f, 0.f, 0.f);
    }
}

// Inclusive prefix over slots 1 .. t-1 (reverse: suffix over slots t-2 .. 0) of each head, in
// place, summed in order.  Eight slots of a thread's four floats are requested at once: the kernel
// is bound by memory, not by the chain of additions.
__global__ void __launch_bounds__(256)
cc_scan_kernel(float4* __restrict__ S, size_t elems, int t, int reverse) {
    pdl_sync();
    const size_t e = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (e >= elems) return;
    float4* p = S + (size_t)blockIdx.y * t * elems + e;
    float4 run = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int k0 = 0; k0 < t - 1; k0 += 8) {
        float4 v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (k0 + q < t - 1) v[q] = p[(size_t)(reverse ? t - 2 - (k0 + q) : k0 + q + 1) * elems];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            if (k0 + q >= t - 1) break;
            run.x += v[q].x; run.y += v[q].y; run.z += v[q].z; run.w += v[q].w;
            p[(size_t)(reverse ? t - 2 - (k0 + q) : k0 + q + 1) * elems] = run;
        }
    }
}

// rows [64][C] of fp32 scratch -> shared memory transposed, dst[c][kLd] (row index contiguous)
template <int C>
__device__ __forceinline__ void load_transposed(float* dst, const float* src, int tid, int nthr) {
#pragma unroll 8
    for (int e = tid; e < 64 * C / 4; e += nthr) {
        const int rr = e % 64, c = (e / 64) * 4;
        const float4 v = *reinterpret_cast<const float4*>(src + (size_t)rr * C + c);
        dst[c * kLd + rr] = v.x; dst[(c + 1) * kLd + rr] = v.y; dst[(c + 2) * kLd + rr] = v.z; dst[(c + 3) * kLd + rr] = v.w;
    }
}
__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 ld4(const __nv_bfloat16* p) {
    const uint2 u = *reinterpret_cast<const uint2*>(p);
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u));
}
__device__ __forceinline__ void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void st4(__nv_bfloat16* p, float4 v) {
    __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), c = __floats2bfloat162_rn(v.z, v.w);
    uint2 u;
    u.x = *reinterpret_cast<unsigned*>(&a); u.y = *reinterpret_cast<unsigned*>(&c);
    *reinterpret_cast<uint2*>(p) = u;
}
// 64 raw rows of a caller's tensor, as they are (dst[row][kLd]) or transposed (dst[c][kLd])
template <typename T, bool TRANSPOSE>
__device__ __forceinline__ void load_raw(float* dst, const T* X, const Slice& sl, int bh, int i0, int tid, int nthr) {
#pragma unroll 8
    for (int e = tid; e < 64 * 16; e += nthr) {
        const int rr = TRANSPOSE ? e % 64 : e / 16, c = 4 * (TRANSPOSE ? e / 64 : e % 16);
        const float4 v = ld4(X + sl.row(bh, i0 + rr) + c);
        if constexpr (TRANSPOSE) {
            dst[c * kLd + rr] = v.x; dst[(c + 1) * kLd + rr] = v.y; dst[(c + 2) * kLd + rr] = v.z; dst[(c + 3) * kLd + rr] = v.w;
        } else {
            *reinterpret_cast<float4*>(dst + rr * kLd + c) = v;
        }
    }
}

// ---------------------------------------------------------------------------
// Rows of lt(W) [Y | y65] for 64 own rows (Section 3.1):
//   sum over chunks of phi'(m_own) S_l  +  sum over the block's other rows of w(own, other) [Y | y65]_other
// with w = (m_own . m_other)^2, LOCAL: (x_own . x_other)^4 from the raw rows (Section 3.2).
//   forward (dv = 0): own = queries, other = keys j <= i, Y = V; writes O = N / d and d = 1 + N[64]
//   backward (dv = 1): own = keys, other = queries i >= j, Y = E, S = suffix states; writes dV
// The work items - state chunks, then 64-row tiles of the block - are dealt to NG groups of 64
// threads (each with shared memory of its own, the next chunk in flight), whose partial sums are
// added at the end: even one head's few rows keep every SM's warps busy.
// grid (b / 64, t, BH).  Bound by the FMA pipe (72 of its clocks per 64 FMAs of a warp's thread).
// ---------------------------------------------------------------------------
template <int R, bool LOCAL, int NG>
struct RowsSmem {
    static constexpr int own = R * kLd + (LOCAL ? kUnit : 0);
    // other side's half sketches (or raw rows), its Y tile, the weights; the two chunk buffers alias
    // them, and the weights alias the raw rows / half sketches where those are as large as a tile
    static constexpr bool kAlias = LOCAL || R == 64;
    static constexpr int oth = kAlias ? kUnit : R * kLd;
    static constexpr int grp = kAlias ? 2 * kUnit : oth + 2 * kUnit;
    static constexpr size_t bytes = (size_t)(own + NG * grp) * sizeof(float);
    static_assert(bytes <= 232448, "shared memory");
};

template <typename T, int R, bool LOCAL, int NG>
__global__ void __launch_bounds__(64 * NG)
cc_rows_kernel(Slice sl, int n, int b, int t, const float* __restrict__ Mown, const float* __restrict__ Moth, YRows y,
               const float* __restrict__ S, const T* __restrict__ Xown, const T* __restrict__ Xoth, int dv,
               T* __restrict__ Out, float* __restrict__ denom) {
    pdl_sync();
    extern __shared__ __align__(16) float smem[];
    using L = RowsSmem<R, LOCAL, NG>;
    constexpr int NT = 64 * NG, NC = kChunks<R>;
    const int tid = threadIdx.x, grp = tid / 64, lane = tid % 64, ry = lane / 8, cx = lane % 8;
    const int tile = blockIdx.x, l = blockIdx.y, bh = blockIdx.z;
    float* sMt = smem;
    float* sXt = smem + R * kLd;
    float* sG = smem + L::own + grp * L::grp;
    const size_t blk0 = (size_t)bh * n + (size_t)l * b;
    const bool states = dv ? l < t - 1 : l > 0;
    const float* Sl = S + ((size_t)bh * t + l) * NC * kChunkFloats;
    auto load_chunk = [&](int c, int buf) {
        const float* src = Sl + (size_t)c * kChunkFloats;
        float* dst = sG + buf * kUnit;
        for (int e = lane; e < kUnit / 4; e += 64) cp16(dst + 4 * e, src + 4 * e);
        cp_commit();
    };
    if (states && grp < NC) load_chunk(grp, 0);
    load_transposed<R>(sMt, Mown + (blk0 + tile * 64) * R, tid, NT);
    if constexpr (LOCAL) load_raw<T, true>(sXt, Xown, sl, bh, l * b + tile * 64, tid, NT);
    __syncthreads();
    Acc acc;
    acc.zero();
    f2 ext[4] = {0ull, 0ull, 0ull, 0ull};
    int item = grp;
    if (states) {
        int buf = 0;
        for (; item < NC; item += NG, buf ^= 1) {
            if (item + NG < NC) { load_chunk(item + NG, buf ^ 1); cp_wait<1>(); } else { cp_wait<0>(); }
            group_sync(grp);
            int ab, bb;
            chunk_pair<R>(item, ab, bb);
            const float* z = sG + buf * kUnit;
            const float* pa = sMt + 8 * ab * kLd + 8 * ry;
            const float* pb = sMt + 8 * bb * kLd + 8 * ry;
#pragma unroll 1
            for (int a = 0; a < 8; ++a) {
                f2 ma[4];
                load_rows8(ma, pa + a * kLd);
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    f2 phi[4];
                    load_rows8(phi, pb + q * kLd);
#pragma unroll
                    for (int i = 0; i < 4; ++i) phi[i] = mul2(phi[i], ma[i]);
                    const float* zr = z + (8 * q + a) * kLd;
                    acc.step(phi, lds22(zr + 4 * cx), lds22(zr + 32 + 4 * cx));
                }
                // the normaliser column: each of a row's eight threads takes one b'
                f2 mb[4];
                load_rows8(mb, pb + cx * kLd);
                const float zl = z[(8 * cx + a) * kLd + 64];
                const f2 zl2 = pack2(zl, zl);
#pragma unroll
                for (int i = 0; i < 4; ++i) ext[i] = fma2(mul2(mb[i], ma[i]), zl2, ext[i]);
            }
            group_sync(grp);
        }
        item -= NC;
    }
    // tiles of the same block
    const int first = dv ? tile : 0, count = dv ? b / 64 - tile : tile + 1;
    float* sO = sG;
    float* sY = sG + L::oth;
    float* sW = L::kAlias ? sG : sY + kUnit;
    for (; item < count; item += NG) {
        const int ot = first + item;
        load_y_rows(sY, y, bh, l * b + ot * 64, lane, 64);
        cp_commit();
        if (y.ones) sY[lane * kLd + 64] = 1.f;
        if constexpr (LOCAL) load_raw<T, true>(sO, Xoth, sl, bh, l * b + ot * 64, lane, 64);
        else load_transposed<R>(sO, Moth + (blk0 + ot * 64) * R, lane, 64);
        cp_wait<0>();
        group_sync(grp);
        Acc sc;
        sc.zero();
        outer_product(sc, LOCAL ? sXt : sMt, sO, LOCAL ? 64 : R, kLd, ry, cx);
        if constexpr (L::kAlias) group_sync(grp);
        const bool diag = ot == tile;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int cj = out_col(cx, j);
            float w[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                float s = sc.at(i, j);
                s *= s;
                if constexpr (LOCAL) s *= s;
                const int ri = out_row(ry, i);
                const bool keep = dv ? cj >= ri : cj <= ri;
                w[i] = (!diag || keep) ? s : 0.f;
            }
            *reinterpret_cast<float4*>(sW + cj * kLd + 8 * ry) = make_float4(w[0], w[1], w[2], w[3]);
            *reinterpret_cast<float4*>(sW + cj * kLd + 8 * ry + 4) = make_float4(w[4], w[5], w[6], w[7]);
        }
        group_sync(grp);
        if (!diag) outer_product(acc, sW, sY, 64, kLd, ry, cx);
        else if (dv) diagonal_product<true>(acc, sW, sY, kLd, ry, cx);
        else diagonal_product<false>(acc, sW, sY, kLd, ry, cx);
        // (the last column is all ones, or nobody reads its sum)
        for (int k = cx; k < 64; k += 8) {
            f2 w[4];
            load_rows8(w, sW + k * kLd + 8 * ry);
            const float yl = sY[k * kLd + 64];
            const f2 yl2 = pack2(yl, yl);
#pragma unroll
            for (int i = 0; i < 4; ++i) ext[i] = fma2(w[i], yl2, ext[i]);
        }
        group_sync(grp);
    }
    // the groups' partial sums, [64][kLd] each
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        float* row = sG + out_row(ry, i) * kLd;
        *reinterpret_cast<float4*>(row + 4 * cx) = make_float4(acc.at(i, 0), acc.at(i, 1), acc.at(i, 2), acc.at(i, 3));
        *reinterpret_cast<float4*>(row + 32 + 4 * cx) = make_float4(acc.at(i, 4), acc.at(i, 5), acc.at(i, 6), acc.at(i, 7));
        float e = (i & 1) ? hi2(ext[i / 2]) : lo2(ext[i / 2]);
        e += __shfl_xor_sync(0xffffffffu, e, 1);
        e += __shfl_xor_sync(0xffffffffu, e, 2);
        e += __shfl_xor_sync(0xffffffffu, e, 4);
        if (cx == 0) row[64] = e;
    }
    __syncthreads();
    for (int e = tid; e < 64 * 16; e += NT) {
        const int rr = e / 16, c = 4 * (e % 16);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        float d = 1.f;
#pragma unroll
        for (int g = 0; g < NG; ++g) {
            const float* row = smem + L::own + g * L::grp + rr * kLd;
            const float4 x = *reinterpret_cast<const float4*>(row + c);
            v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
            d += row[64];
        }
        const int i = l * b + tile * 64 + rr;
        if (!dv) {
            const float inv = 1.f / d;
            v.x *= inv; v.y *= inv; v.z *= inv; v.w *= inv;
            if (c == 0 && denom != nullptr) denom[(size_t)bh * n + i] = d;
        }
        st4(Out + sl.row(bh, i) + c, v);
    }
}

// ---------------------------------------------------------------------------
// Gradient of the own rows' half sketches:
//   dm_own = sum over chunks of the un-tensored d phi' = S_l [Y | y65]_own
//          + sum over the block's other rows of 2 s (Y_own . Y_other) m_other,   s = m_own . m_other
// LOCAL: the same-block part is 4 x^3 (Y_own . Y_other) x_other, a gradient of the raw rows, and
// leaves separately.  Query side (kside = 0): own rows E, other rows [V | 1], others j <= i; key
// side: own rows [V | 1], other rows E, others i >= j.  A stored feature (a, b) with gradient g gives
// dm[a] += g m[b] and dm[b] += g m[a] (its state row carries the pair's weight).
// Work items and groups as in cc_rows_kernel; the products are in dot form, because both the
// states' rows and Y's rows are contiguous along the 65 columns that are summed over.
// ---------------------------------------------------------------------------
template <int R, bool LOCAL, int NG>
struct DphiSmem {
    static constexpr int ldm = R + 4;
    static constexpr int own_m = 0, own_y = 64 * ldm, own_x = own_y + kUnit;
    static constexpr int own = own_x + (LOCAL ? kUnit : 0);
    // per group: two chunk buffers = the other side's half sketches (raw rows) and Y tile / ds;
    // then the gradient accumulator
    static constexpr int dm = 2 * kUnit, grp = dm + 64 * ldm;
    static constexpr size_t bytes = (size_t)(own + NG * grp) * sizeof(float);
    static_assert(bytes <= 232448, "shared memory");
};

template <typename T, int R, bool LOCAL, int NG>
__global__ void __launch_bounds__(64 * NG)
cc_dphi_kernel(Slice sl, int n, int b, int t, const float* __restrict__ Mown, const float* __restrict__ Moth, YRows yown,
               YRows yoth, const float* __restrict__ S, const T* __restrict__ Xown, const T* __restrict__ Xoth, int kside,
               float* __restrict__ dM, float* __restrict__ dXl) {
    pdl_sync();
    extern __shared__ __align__(16) float smem[];
    using L = DphiSmem<R, LOCAL, NG>;
    constexpr int NT = 64 * NG, NC = kChunks<R>, LDM = L::ldm;
    constexpr int LDS_ = LOCAL ? kLd : LDM;             // leading dimension of the rows a score is made of
    constexpr int NCOL = LOCAL ? 8 : R / 8;             // columns of the same-block gradient per thread
    const int tid = threadIdx.x, grp = tid / 64, lane = tid % 64, ry = lane / 8, cx = lane % 8;
    const int tile = blockIdx.x, l = blockIdx.y, bh = blockIdx.z;
    float* sM = smem + L::own_m;
    float* sYo = smem + L::own_y;
    float* sX = smem + L::own_x;
    float* sG = smem + L::own + grp * L::grp;
    float* sD = sG + L::dm;
    const size_t blk0 = (size_t)bh * n + (size_t)l * b;
    const bool states = kside ? l < t - 1 : l > 0;
    const float* Sl = S + ((size_t)bh * t + l) * NC * kChunkFloats;
    auto load_chunk = [&](int c, int buf) {
        const float* src = Sl + (size_t)c * kChunkFloats;
        float* dst = sG + buf * kUnit;
        for (int e = lane; e < kUnit / 4; e += 64) cp16(dst + 4 * e, src + 4 * e);
        cp_commit();
    };
    auto load_m = [&](float* dst, const float* src, int id, int nthr) {
        for (int e = id; e < 64 * R / 4; e += nthr) cp16(dst + (e / (R / 4)) * LDM + 4 * (e % (R / 4)), src + 4 * e);
    };
    load_y_rows(sYo, yown, bh, l * b + tile * 64, tid, NT);
    load_m(sM, Mown + (blk0 + tile * 64) * R, tid, NT);
    cp_commit();
    if (states && grp < NC) load_chunk(grp, 0);
    if (yown.ones && tid < 64) sYo[tid * kLd + 64] = 1.f;
    if constexpr (LOCAL) load_raw<T, false>(sX, Xown, sl, bh, l * b + tile * 64, tid, NT);
    for (int e = lane; e < 64 * LDM; e += 64) sD[e] = 0.f;
    if (states && grp < NC) cp_wait<1>(); else cp_wait<0>();
    __syncthreads();
    int item = grp;
    if (states) {
        int buf = 0;
        for (; item < NC; item += NG, buf ^= 1) {
            if (item + NG < NC) { load_chunk(item + NG, buf ^ 1); cp_wait<1>(); } else { cp_wait<0>(); }
            group_sync(grp);
            int ab, bb;
            chunk_pair<R>(item, ab, bb);
            const float* z = sG + buf * kUnit;
            {
                f2 d[8][8];
                dot_full<kLd, kLd>(d, sYo, z, 16, ry, cx);
                float zl[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) zl[j] = z[(cx + 8 * j) * kLd + 64];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int rr = ry + 8 * i;
                    const float yl = sYo[rr * kLd + 64];
                    const float* mr = sM + rr * LDM;
                    const float ma = mr[8 * ab + cx];
                    float mb[8];
                    *reinterpret_cast<float4*>(mb) = *reinterpret_cast<const float4*>(mr + 8 * bb);
                    *reinterpret_cast<float4*>(mb + 4) = *reinterpret_cast<const float4*>(mr + 8 * bb + 4);
                    float da = 0.f, v[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float g = fmaf(yl, zl[j], sum2(d[i][j]));
                        da = fmaf(g, mb[j], da);
                        v[j] = g * ma;
                    }
                    // entry b' of the second factor's gradient: the sum over the eight a', left with
                    // the thread of the same number
                    float u[4], w[2];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float keep = (cx & 4) ? v[4 + j] : v[j], send = (cx & 4) ? v[j] : v[4 + j];
                        u[j] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
                    }
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const float keep = (cx & 2) ? u[2 + j] : u[j], send = (cx & 2) ? u[j] : u[2 + j];
                        w[j] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
                    }
                    const float keep = (cx & 1) ? w[1] : w[0], send = (cx & 1) ? w[0] : w[1];
                    const float db = keep + __shfl_xor_sync(0xffffffffu, send, 1);
                    // coordinates cx mod 8 of rows ry mod 8: this thread's own
                    float* dr = sD + rr * LDM;
                    dr[8 * ab + cx] += da;
                    dr[8 * bb + cx] += db;
                }
            }
            group_sync(grp);
        }
        item -= NC;
    }
    // tiles of the same block
    f2 gs[4][NCOL / 2], gx[4][NCOL / 2];
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < NCOL / 2; ++q) gs[p][q] = gx[p][q] = 0ull;
    const int first = kside ? tile : 0, count = kside ? b / 64 - tile : tile + 1;
    float* sO = sG;
    float* sY = sG + kUnit;
    for (; item < count; item += NG) {
        const int ot = first + item;
        load_y_rows(sY, yoth, bh, l * b + ot * 64, lane, 64);
        if constexpr (!LOCAL) load_m(sO, Moth + (blk0 + ot * 64) * R, lane, 64);
        cp_commit();
        if (yoth.ones) sY[lane * kLd + 64] = 1.f;
        if constexpr (LOCAL) load_raw<T, false>(sO, Xoth, sl, bh, l * b + ot * 64, lane, 64);
        cp_wait<0>();
        group_sync(grp);
        const bool diag = ot == tile;
        float ds[8][8];
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            if constexpr (LOCAL) {
                // The forward's scores to the last bit.  O and the normaliser carry the error of their score's fourth power, and
                // the derivative x^3 / (1 + x^4)^2 of a row with few keys nearly cancels it, if the error is the same one.  (With
                // the two half sums of dot_half: dQ of the first rows of a head off by 2.4 times as much; same time.)
                float s[4][8];
                dot_half_chain<kLd, kLd>(s, sX, sO, 16, half, ry, cx);
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 8; ++j) ds[4 * half + i][j] = 4.f * s[i][j] * s[i][j] * s[i][j];
            } else {
                f2 s[4][8];
                dot_half<LDM, LDM>(s, sM, sO, R / 4, half, ry, cx);
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 8; ++j) ds[4 * half + i][j] = 2.f * sum2(s[i][j]);
            }
            f2 d[4][8];
            dot_half<kLd, kLd>(d, sYo, sY, 16, half, ry, cx);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float yl = sY[(cx + 8 * j) * kLd + 64];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int rr = ry + 32 * half + 8 * i, cj = cx + 8 * j;
                    const bool keep = kside ? cj >= rr : cj <= rr;
                    const float g = ds[4 * half + i][j] * fmaf(sYo[rr * kLd + 64], yl, sum2(d[i][j]));
                    ds[4 * half + i][j] = (!diag || keep) ? g : 0.f;
                }
            }
        }
        group_sync(grp);
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) sY[(cx + 8 * j) * kLd + ry + 8 * i] = ds[i][j];
        group_sync(grp);
        // same-block gradient += ds (64 own x 64 other) . rows of the other side (64 x 8 NCOL)
        auto columns = [&](int k, f2 (&a)[4], f2 (&c)[NCOL / 2]) {
            load_rows8(a, sY + k * kLd + 8 * ry);
            const float* o = sO + k * LDS_;
            if constexpr (NCOL == 2) {
                c[0] = *reinterpret_cast<const f2*>(o + 2 * cx);
            } else {
                const F22 u = lds22(o + 4 * cx);
                c[0] = u.x; c[1] = u.y;
                if constexpr (NCOL == 8) { const F22 w = lds22(o + 32 + 4 * cx); c[2] = w.x; c[3] = w.y; }
            }
        };
        // (diagonal tile: the pairs that count, see diagonal_step)
        const int k0 = diag && kside ? 8 * ry + 8 : 0, k1 = diag && !kside ? 8 * ry : 64;
#pragma unroll 2
        for (int k = k0; k < k1; ++k) {
            f2 a[4], c[NCOL / 2];
            columns(k, a, c);
#pragma unroll
            for (int q = 0; q < NCOL / 2; ++q) {
                const f2 sw = swap2(c[q]);
#pragma unroll
                for (int p = 0; p < 4; ++p) { gs[p][q] = fma2(a[p], c[q], gs[p][q]); gx[p][q] = fma2(a[p], sw, gx[p][q]); }
            }
        }
        if (diag) {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                f2 a[4], c[NCOL / 2];
                columns(8 * ry + q, a, c);
                if (kside) diagonal_step<true>(gs, gx, a, c, 0, q);
                else diagonal_step<false>(gs, gx, a, c, 0, q);
            }
        }
        group_sync(grp);
    }
    // same-block sums: into the half-sketch gradient, or (LOCAL) a tile of their own
    group_sync(grp);
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < NCOL; ++j) {
            const f2 v = ((i ^ j) & 1) ? gx[i / 2][j / 2] : gs[i / 2][j / 2];
            const float x = (i & 1) ? hi2(v) : lo2(v);
            const int col = NCOL == 8 ? out_col(cx, j) : NCOL * cx + j;
            if constexpr (LOCAL) sG[out_row(ry, i) * kLd + col] = x;
            else sD[out_row(ry, i) * LDM + col] += x;
        }
    __syncthreads();
    const size_t row0 = blk0 + tile * 64;
    for (int e = tid; e < 64 * R / 4; e += NT) {
        const int rr = e / (R / 4), c = 4 * (e % (R / 4));
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int g = 0; g < NG; ++g) {
            const float4 x = *reinterpret_cast<const float4*>(smem + L::own + g * L::grp + L::dm + rr * LDM + c);
            v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
        }
        *reinterpret_cast<float4*>(dM + (row0 + rr) * R + c) = v;
    }
    if constexpr (LOCAL) {
        for (int e = tid; e < 64 * 16; e += NT) {
            const int rr = e / 16, c = 4 * (e % 16);
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int g = 0; g < NG; ++g) {
                const float4 x = *reinterpret_cast<const float4*>(smem + L::own + g * L::grp + rr * kLd + c);
                v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
            }
            *reinterpret_cast<float4*>(dXl + (row0 + rr) * 64 + c) = v;
        }
    }
}

}  // namespace cc
}  // namespace psk
