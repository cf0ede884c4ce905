// Register-tiled fp32 products for the CUDA-core kernels.
//
// A group of 64 threads (two warps) owns a 64 x 64 product; thread `lane` (0..63) = (ry, cx) =
// (lane / 8, lane % 8) owns 8 x 8 of it.  All arithmetic is IEEE fp32 fused multiply-add, issued in
// packed pairs (fma.rn.f32x2: two independent roundings, the same results as two scalar FMAs):
// on B200 scalar and packed FMAs reach the same 128 per clock and SM, but the packed form needs
// half the issue slots, which leaves room for the shared-memory loads.
//
// Two forms, by which index of the operands is contiguous in shared memory:
//   outer: A is [k][64 rows], B is [k][64 columns].  Row pairs are packed; a column pair is used as
//          it is and with its halves swapped, which costs one register move per column instead of
//          the two that duplicating every column value would.
//          rows 8 ry + 0..7, columns 4 cx + 0..3 and 32 + 4 cx + 0..3
//   dot:   A is [64 rows][k], B is [64 columns][k].  Even and odd k are summed in the two halves of
//          a pair and added at the end.  rows ry + 8 i, columns cx + 8 j
// Both maps read shared memory without bank conflicts when the leading dimension is 68 floats
// (or r + 4).
#pragma once

#include "psk_internal.cuh"
#include "packed.cuh"

namespace psk {
namespace cc {

__device__ __forceinline__ f2 swap2(f2 v) { return pack2(hi2(v), lo2(v)); }
struct F22 { f2 x, y; };
__device__ __forceinline__ F22 lds22(const float* p) {       // 16 bytes as two pairs
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
    return F22{v.x, v.y};
}

constexpr int kLd = 68;               // leading dimension of 64- and 65-column tiles in shared memory
constexpr int kUnit = 64 * kLd;       // floats of one such tile

__device__ __forceinline__ void group_sync(int g) { asm volatile("bar.sync %0, 64;" ::"r"(g + 1) : "memory"); }

__device__ __forceinline__ void cp16(float* dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// 8 x 8 accumulator of the outer form.
struct Acc {
    f2 s[4][4], x[4][4];              // straight / swapped column pairs
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int q = 0; q < 4; ++q) s[p][q] = x[p][q] = 0ull;
    }
    // a: four row pairs; b: 4 columns at `b`, 4 at `b + half`
    __device__ __forceinline__ void step(const f2 (&a)[4], const F22& b0, const F22& b1) {
        const f2 c[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const f2 sw = swap2(c[q]);
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                s[p][q] = fma2(a[p], c[q], s[p][q]);
                x[p][q] = fma2(a[p], sw, x[p][q]);
            }
        }
    }
    // value of row i (0..7), column j (0..7; j < 4: 4 cx + j, else 32 + 4 cx + j - 4)
    __device__ __forceinline__ float at(int i, int j) const {
        const f2 v = ((i ^ j) & 1) ? x[i / 2][j / 2] : s[i / 2][j / 2];
        return (i & 1) ? hi2(v) : lo2(v);
    }
};
// row of accumulator row i / column of accumulator column j in the outer form
__device__ __forceinline__ int out_row(int ry, int i) { return 8 * ry + i; }
__device__ __forceinline__ int out_col(int cx, int j) { return (j < 4 ? 0 : 28) + 4 * cx + j; }

__device__ __forceinline__ void load_rows8(f2 (&a)[4], const float* p) {
    const F22 u = lds22(p), v = lds22(p + 4);
    a[0] = u.x; a[1] = u.y; a[2] = v.x; a[3] = v.y;
}

// Token 8 ry + q against the thread's rows 8 ry + 0..7 on the diagonal of a 64 x 64 tile, of which only the pairs
// with token <= row (UPPER: token >= row) count.  Pairs beyond it are left out or multiplied by zeros on both sides: a
// weight of zero alone would let an infinity or a NaN of a row that does not count through.  q is a constant
// after unrolling; c: NQ column pairs, into the accumulators q0, q0 + 1, ...
template <bool UPPER, int NQ, int NA>
__device__ __forceinline__ void diagonal_step(f2 (&s)[4][NA], f2 (&x)[4][NA], const f2 (&a)[4], const f2 (&c)[NQ], int q0, int q) {
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const bool lo = UPPER ? q >= 2 * p : q <= 2 * p, hi = UPPER ? q >= 2 * p + 1 : q <= 2 * p + 1;
        if (!lo && !hi) continue;
#pragma unroll
        for (int j = 0; j < NQ; ++j) {
            const float c0 = lo2(c[j]), c1 = hi2(c[j]);
            s[p][q0 + j] = fma2(a[p], pack2(lo ? c0 : 0.f, hi ? c1 : 0.f), s[p][q0 + j]);
            x[p][q0 + j] = fma2(a[p], pack2(lo ? c1 : 0.f, hi ? c0 : 0.f), x[p][q0 + j]);
        }
    }
}
// acc += At^T B of a diagonal tile, At [64 tokens][kLd] (64 rows), B [64 tokens][ldb] (64 columns); only the
// pairs that count are visited, half as many as in a whole tile
template <bool UPPER>
__device__ __forceinline__ void diagonal_product(Acc& acc, const float* At, const float* B, int ldb, int ry, int cx) {
    const int k1 = UPPER ? 64 : 8 * ry;
#pragma unroll 2
    for (int k = UPPER ? 8 * ry + 8 : 0; k < k1; ++k) {
        f2 a[4];
        load_rows8(a, At + k * kLd + 8 * ry);
        acc.step(a, lds22(B + k * ldb + 4 * cx), lds22(B + k * ldb + 32 + 4 * cx));
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int k = 8 * ry + q;
        f2 a[4];
        load_rows8(a, At + k * kLd + 8 * ry);
        const F22 u = lds22(B + k * ldb + 4 * cx), v = lds22(B + k * ldb + 32 + 4 * cx);
        const f2 c[4] = {u.x, u.y, v.x, v.y};
        diagonal_step<UPPER>(acc.s, acc.x, a, c, 0, q);
    }
}

// acc += At^T B over k < K: At [K][kLd] (64 rows), B [K][ldb] (64 columns)
template <int UNROLL = 4>
__device__ __forceinline__ void outer_product(Acc& acc, const float* At, const float* B, int K, int ldb, int ry, int cx) {
#pragma unroll UNROLL
    for (int k = 0; k < K; ++k) {
        f2 a[4];
        load_rows8(a, At + k * kLd + 8 * ry);
        acc.step(a, lds22(B + k * ldb + 4 * cx), lds22(B + k * ldb + 32 + 4 * cx));
    }
}

// d[i][j] = sum_{k < 4 K4} A[ry + 8 (4 half + i)][k] B[cx + 8 j][k], four of the thread's eight rows
template <int LDA, int LDB>
__device__ __forceinline__ void dot_half(f2 (&d)[4][8], const float* A, const float* B, int K4, int half, int ry, int cx) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) d[i][j] = 0ull;
    const float* a0 = A + (ry + 32 * half) * LDA;
    const float* b0 = B + cx * LDB;
#pragma unroll 2
    for (int k = 0; k < 4 * K4; k += 4) {
        F22 a[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = lds22(a0 + 8 * i * LDA + k);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const F22 b = lds22(b0 + 8 * j * LDB + k);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                d[i][j] = fma2(a[i].x, b.x, d[i][j]);
                d[i][j] = fma2(a[i].y, b.y, d[i][j]);
            }
        }
    }
}
// The same with every sum as one chain over k, in the order of outer_product and so to the last bit the value that it
// forms: for scores whose errors cancel only if the forward and the backward make the same ones.
template <int LDA, int LDB>
__device__ __forceinline__ void dot_half_chain(float (&d)[4][8], const float* A, const float* B, int K4, int half, int ry, int cx) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) d[i][j] = 0.f;
    const float* a0 = A + (ry + 32 * half) * LDA;
    const float* b0 = B + cx * LDB;
#pragma unroll 2
    for (int k = 0; k < 4 * K4; k += 4) {
        float4 a[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4*>(a0 + 8 * i * LDA + k);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float4 b = *reinterpret_cast<const float4*>(b0 + 8 * j * LDB + k);
#pragma unroll
            for (int i = 0; i < 4; ++i) d[i][j] = fmaf(a[i].w, b.w, fmaf(a[i].z, b.z, fmaf(a[i].y, b.y, fmaf(a[i].x, b.x, d[i][j]))));
        }
    }
}
// all eight rows at once: two thirds of the shared-memory loads per product, for 128 accumulator registers
template <int LDA, int LDB>
__device__ __forceinline__ void dot_full(f2 (&d)[8][8], const float* A, const float* B, int K4, int ry, int cx) {
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) d[i][j] = 0ull;
    const float* a0 = A + ry * LDA;
    const float* b0 = B + cx * LDB;
#pragma unroll 1
    for (int k = 0; k < 4 * K4; k += 4) {
        F22 b[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) b[j] = lds22(b0 + 8 * j * LDB + k);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const F22 a = lds22(a0 + 8 * i * LDA + k);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                d[i][j] = fma2(a.x, b[j].x, d[i][j]);
                d[i][j] = fma2(a.y, b[j].y, d[i][j]);
            }
        }
    }
}
__device__ __forceinline__ float sum2(f2 v) { return lo2(v) + hi2(v); }

}  // namespace cc
}  // namespace psk
