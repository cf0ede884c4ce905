// Symmetric feature set of the self-tensored sketch, and its in-register generators.
//
// phi'(x) = m (x) m has r^2 entries but only r(r+1)/2 distinct ones (m_a m_b = m_b m_a), so
// <phi'(q), phi'(k)> = sum over unordered pairs of w_ab (q_a q_b)(k_a k_b) with w_ab = 2 for
// a != b and 1 on the diagonal: the same number the r^2-dimensional product of Algorithm 1 gives.
// The kernels carry one feature per unordered pair.  Every thread generates UNWEIGHTED products
// m_a m_b; the weights are applied once, to the rows of the stored states (Feat::weight), so
// every contraction of fresh features with a state, and every gradient that flows back through a
// state, already carries them.  With weighted gradients d(feature) the half-sketch gradient is
//   dm[a] += d(feature ab) m[b];   dm[b] += d(feature ab) m[a]        for every stored feature,
// the diagonal included (its two updates coincide, which is the factor 2 of d(m_a^2)).
//
// Two feature orders, both in words of two features (f even: the pair (f, f + 1) is one packed bf16x2 product):
//
//  * circulant (r <= 32): feature (s, a) = m[a] m[(a + s) mod r] for shifts s = 0 .. r/2, shift-major,
//    f = s r + a.  Shift r/2 lists every pair {a, a + r/2} twice, so its weight is 1.  A word is an
//    even-aligned pair of entries times an even- or odd-aligned one.
//
//  * blocks (r = 64): pairs of entries p = 0 .. 31, coordinates 2p and 2p + 1.  For every p the word (2p, 2p), (2p, 2p + 1),
//    then for q = p + 1 .. 31 the words (2p, 2q), (2p, 2q + 1) and (2p + 1, 2q), (2p + 1, 2q + 1): one entry times an
//    even-aligned pair.  Last the diagonal entries that are left, (2p + 1, 2p + 1), p = 0 .. 31.
//
// Everything is unrolled: a 64-feature chunk is straight code on registers with fixed indexes, and a kernel's loop over
// chunks enters the chunk's code through switch_chunk().  So only the products are there once per chunk; waits, MMA
// issue and loads are there once.  The products in packed pairs (bf16x2, and fp32 pairs in the backward) are 1 (r = 16), 4 (r = 32)
// and 17 KB (r = 64) of code for the features and 2, 9 and 33 KB for their backward; what a kernel executes has to come
// from an instruction cache of about 32 KB at full rate, at half rate to about 96 KB, at a tenth beyond 128 KB.
// (Before, r <= 32 rotated the half sketch through registers in a loop of two shifts, r = 64 had waits and MMA issue once per chunk and
// scalar FMAs, 130 to 225 KB.  Training, 48 heads x 16 384, r = 64, b = 512: 4647 -> 4030 us; 384 heads x 32 768, r = 32:
// 20 723 -> 20 615; exact blocks, 48 heads x 2688, r = 32: 259 -> 251; degree 8, 96 heads x 8192: 1673 -> 1619.)
#pragma once

#include "packed.cuh"
#include "tc_prims.cuh"

#include <type_traits>

namespace psk {
namespace tc {

template <int I, int N, typename Fn>
__device__ __forceinline__ void static_for(Fn&& f) {
    if constexpr (I < N) {
        f(std::integral_constant<int, I>{});
        static_for<I + 1, N>(f);
    }
}
// f(integral_constant<i>) for a run-time i of [LO, HI), the same for the whole warp: a binary search of branches
template <int LO, int HI, typename Fn>
__device__ __forceinline__ void switch_chunk(int i, Fn&& f) {
    if constexpr (HI - LO == 1) {
        f(std::integral_constant<int, LO>{});
    } else {
        constexpr int MID = (LO + HI) / 2;
        if (i < MID) switch_chunk<LO, MID>(i, f);
        else switch_chunk<MID, HI>(i, f);
    }
}

template <int R>
struct Feat {
    static constexpr bool kCirc = (R <= 32);
    static constexpr int F = kCirc ? (R / 2 + 1) * R : R * (R + 1) / 2;   // stored features
    static constexpr int FK = F;                     // a multiple of the MMA K step
    static constexpr int NC = (F + 63) / 64;         // 64-feature chunks (A staging / state TMA boxes)
    static constexpr int NT = (F + 127) / 128;       // 128-feature tiles (state accumulators)
    static constexpr int FP = NT * 128;              // padded feature extent of stored states
    static_assert(F % 16 == 0, "whole MMA K steps");

    // blocks: first word of pair p (p = r/2: the diagonal entries that are left), and the p of word w
    __host__ __device__ static constexpr int block_base(int p) { return p * (R - p); }
    __host__ __device__ static constexpr int block_of(int w) {
        int p = 0;
        while (p < R / 2 && w >= block_base(p + 1)) ++p;
        return p < R / 2 && w < R * R / 4 ? p : R / 2;
    }
    __host__ __device__ static constexpr int a(int f) {
        if (kCirc) return f % R;
        const int w = f / 2, p = block_of(w);
        if (p == R / 2) return 2 * (f - R * R / 2) + 1;
        const int k = w - block_base(p);              // 0: the diagonal word; then both words of q = p + 1, ...
        return k == 0 ? 2 * p : 2 * p + ((k - 1) & 1);
    }
    __host__ __device__ static constexpr int b(int f) {
        if (kCirc) return (f % R + f / R) % R;
        const int w = f / 2, p = block_of(w);
        if (p == R / 2) return 2 * (f - R * R / 2) + 1;
        const int k = w - block_base(p);
        return 2 * (p + (k + 1) / 2) + (f & 1);
    }
    // weight of stored state row f (0 for padding rows)
    __host__ __device__ static float weight(int f) {
        if (f >= F) return 0.f;
        if (kCirc) return (f < R || f >= F - R) ? 1.f : 2.f;
        if (f >= R * R / 2) return 1.f;
        // block_base(p) = (r/2)^2 - (r/2 - p)^2: a diagonal word leaves a square
        const int left = R * R / 4 - f / 2;
        const int root = (int)(sqrtf((float)left) + 0.5f);
        return ((f & 1) == 0 && root * root == left) ? 1.f : 2.f;
    }
};

// (volatile, here and below: the products depend on nothing that changes in a loop over chunks, and the compiler would
// form all of them before it, and spill them)
__device__ __forceinline__ uint32_t hmul2_bf16(uint32_t x, uint32_t y) {
    uint32_t r;
    asm volatile("mul.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(y));
    return r;
}
// the low (0) or high (1) half of a pair in both halves
template <int HALF>
__device__ __forceinline__ uint32_t twice(uint32_t x) {
    uint32_t r;
    asm volatile("prmt.b32 %0, %1, %1, %2;" : "=r"(r) : "r"(x), "n"(HALF ? 0x3232 : 0x1010));
    return r;
}

// The half sketch of one row as packed bf16 pairs, and the features formed from it:
//   e[k] = (m[2k], m[2k+1]),   circulant order also  o[k] = (m[2k+1], m[(2k+2) mod r]).
// A packed multiply yields two features; the product is rounded to bf16 once more, which the
// tolerance budget covers (relative 2^-9 each, independent across features).
template <int R>
struct FeatGen {
    static constexpr int H = R / 2, HO = Feat<R>::kCirc ? R / 2 : 1;
    uint32_t e[H], o[HO];

    __device__ __forceinline__ void init(const float (&m)[R]) {
#pragma unroll
        for (int k = 0; k < H; ++k) {
            e[k] = pack_bf16(m[2 * k], m[2 * k + 1]);
            if constexpr (Feat<R>::kCirc) o[k] = pack_bf16(m[2 * k + 1], m[(2 * k + 2) % R]);
        }
    }
    // features 2 W, 2 W + 1
    template <int W>
    __device__ __forceinline__ uint32_t word() const {
        if constexpr (2 * W >= Feat<R>::F) {
            return 0u;
        } else if constexpr (Feat<R>::kCirc) {
            constexpr int S = W / H, K = W % H;
            if constexpr (S % 2 == 0) return hmul2_bf16(e[K], e[(K + S / 2) % H]);
            else return hmul2_bf16(e[K], o[(K + S / 2) % H]);
        } else if constexpr (2 * W >= R * R / 2) {
            constexpr int A = Feat<R>::a(2 * W) / 2;                        // (m[2A+1], m[2A+3]) squared
            uint32_t x;
            asm volatile("prmt.b32 %0, %1, %2, 0x7632;" : "=r"(x) : "r"(e[A]), "r"(e[A + 1]));
            return hmul2_bf16(x, x);
        } else {
            constexpr int A = Feat<R>::a(2 * W), Q = Feat<R>::b(2 * W) / 2;
            return hmul2_bf16(twice<A % 2>(e[A / 2]), e[Q]);
        }
    }
    // words W0 .. W0 + N - 1
    template <int W0, int N>
    __device__ __forceinline__ void words(uint32_t (&out)[N]) const {
        static_for<0, N>([&](auto jc) { out[decltype(jc)::value] = word<W0 + decltype(jc)::value>(); });
    }
};

// ---------------------------------------------------------------------------
// Backward of the features: with x the (weighted) gradients of the features, dm[a] += x m[b], dm[b] += x m[a] for every
// stored feature, in packed fp32 pairs (two independent IEEE roundings).  On B200 packed and scalar FMAs
// reach the same rate; the packed ones are half the instructions, and no registers are moved.
// circulant: m and dm as even- and as odd-aligned pairs.  blocks: even-aligned pairs; the sums over a block row's
// second factors stay in two pairs (row 2p, row 2p + 1) while the words of p go by.
// ---------------------------------------------------------------------------
template <int R>
struct Untensor {
    using F = Feat<R>;
    static constexpr int H = R / 2, HO = F::kCirc ? R / 2 : 1;
    f2 me[H], de[H], mo[HO], od[HO];
    f2 row[2];

    __device__ __forceinline__ void init(const float (&m)[R]) {
#pragma unroll
        for (int k = 0; k < H; ++k) {
            me[k] = pack2(m[2 * k], m[2 * k + 1]);
            de[k] = 0ull;
            if constexpr (F::kCirc) { mo[k] = pack2(m[2 * k + 1], m[(2 * k + 2) % R]); od[k] = 0ull; }
        }
        row[0] = row[1] = 0ull;
    }
    // gradients of the features F0 .. F0 + N - 1 (fp32 bit patterns)
    template <int F0, int N>
    __device__ __forceinline__ void add(const uint32_t (&x)[N]) {
        static_for<0, N / 2>([&](auto jc) {
            constexpr int J = decltype(jc)::value, f = F0 + 2 * J;
            if constexpr (f < F::F) {
                const f2 v = pack2(x[2 * J], x[2 * J + 1]);
                if constexpr (F::kCirc) {
                    constexpr int S = f / R, K = f % R / 2, Q = (K + S / 2) % H;
                    if constexpr (S % 2 == 0) {
                        de[K] = fma2(v, me[Q], de[K]);
                        de[Q] = fma2(v, me[K], de[Q]);
                    } else {
                        de[K] = fma2(v, mo[Q], de[K]);
                        od[Q] = fma2(v, me[K], od[Q]);
                    }
                } else if constexpr (f >= R * R / 2) {
                    // (2p + 1, 2p + 1), (2p + 3, 2p + 3): both updates of a diagonal entry coincide
                    constexpr int P = F::a(f) / 2;
                    de[P] = pack2(lo2(de[P]), fmaf(2.f * lo2(v), hi2(me[P]), hi2(de[P])));
                    de[P + 1] = pack2(lo2(de[P + 1]), fmaf(2.f * hi2(v), hi2(me[P + 1]), hi2(de[P + 1])));
                } else {
                    constexpr int A = F::a(f), P = A / 2, Q = F::b(f) / 2;
                    const float ma = A % 2 ? hi2(me[P]) : lo2(me[P]);
                    row[A % 2] = fma2(v, me[Q], row[A % 2]);
                    de[Q] = fma2(v, pack2(ma, ma), de[Q]);
                    if constexpr (f + 2 >= R * R / 2 || F::a(f + 2) / 2 != P) {       // last word of this p
                        de[P] = pack2(lo2(de[P]) + (lo2(row[0]) + hi2(row[0])), hi2(de[P]) + (lo2(row[1]) + hi2(row[1])));
                        row[0] = row[1] = 0ull;
                    }
                }
            }
        });
    }
    __device__ __forceinline__ void finish(float (&dm)[R]) const {
#pragma unroll
        for (int k = 0; k < H; ++k) {
            dm[2 * k] = lo2(de[k]);
            dm[2 * k + 1] = hi2(de[k]);
            if constexpr (F::kCirc) { dm[2 * k] += hi2(od[(k + H - 1) % H]); dm[2 * k + 1] += lo2(od[k]); }
        }
    }
};

}  // namespace tc
}  // namespace psk
