// Learnable sketch (Algorithm 2 of the paper's appendix) with its dense layers on the tensor
// cores: bf16 operands, fp32 accumulation in tensor memory, r = 16 or 32 (8r <= 256), h = 64.
//
//   f(x) = W4^T gelu(W3^T (W2^T LN1(gelu(W1^T LN0(x) + b1)) + b2) + b3) + b4      (two such networks)
//   M    = sqrt(r) tanh(f_1(x) * f_2(x) / sqrt(r))
//
// The wide activations (8r per row) never leave the SM.  With p1, p3 the pre-activations, n0, n1 the
// normalised rows, a2 the narrow activations between the halves and a3 = gelu(p3):
//   ltc_dense_norm_kernel      forward of a 128-row tile in one go, as in attention: groups of 64 columns of p1
//                              (p3) go from tensor memory through the gelu back into tensor memory as the
//                              operand of the next layer.  The normalisation between them needs no second
//                              look at the columns: n1 W2 = rs1 (g W2 - mu1 (1^T W2)).
//                              Kept for the backward: a2 (hi + lo), mu1, rs1 and f, 264 bytes a row (r = 32).
//   ltc_wgrad_kernel           layers 4 and 3 backward: p3 again from a2, then da2 and the weight gradients
//                              a3^T df, dp3^T a2
//   ltc_dense_bwd_norm_kernel  layers 2 and 1 backward: p1 again from n0, then dn0, n1^T da2, dp1^T n0.  The two
//                              row sums of the normalisation's backward are inner products of narrow rows:
//                              sum dn1 = da2 . (1^T W2),  sum dn1 n1 = da2 . (a2 - b2)
// and small kernels around them.  The gains of the normalisations are folded into the following layer's
// weights (z W = n (diag(g) W) + c W), so the normalised activations n are the GEMM operands and their
// gradients come out of the GEMM with the gain already applied.  Weight gradients are sums over ALL rows of
// outer products: every CTA keeps them in tensor memory for all its tiles and adds them to an fp32
// accumulator once; gains, biases and the folded terms are taken from those by a last small kernel.
//
// Bound: the CUDA cores (the gelu and its derivative, the hi/lo splits), with the tensor pipe second: a
// tile of 128 rows and one network is 65 536 gelus forward and twice that with derivatives backward.
// (As sixteen separate layer launches, every activation crossing memory twice, 48 heads x 8192, r = 32,
// forward + backward took 8.4 ms.)
//
// Precision: a half sketch feeds fourth powers of cancelling sums, and single bf16 operands, 2^-9 per entry
// and four layers deep, would leave percents of error on the attention's output.  The forward multiplies
// hi + lo pairs of bf16 terms for both activations and weights, A_hi B_hi + A_lo B_hi + A_hi B_lo: 2^-17.  The
// backward's deltas and weight-gradient operands are single bf16; p1 and p3 are recomputed with the pairs.
#include "cc_gemm.cuh"
#include "tc_common.cuh"

#include <cstdlib>

namespace psk {

namespace {

using namespace tc;

constexpr float kLnEps = 1e-6f;
constexpr size_t kChunkRows = (size_t)1 << 20;        // rows per pass over the networks
constexpr int kMat = 64 * 256;                        // entries of one weight-gradient accumulator [256][64]
// folded vectors of one network: b1' | b2' | b3 | b4 | column sums of diag(g1) W2
constexpr int kVb2 = 256, kVb3 = 320, kVb4 = 576, kVcs = 640, kVec = 704;
constexpr int kSums = 256 + 64 + 256 + 64;            // column sums of one network: dp1 | da2 | dp3 | df

__device__ __forceinline__ float ex2_approx(float x) { float y; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
__device__ __forceinline__ f2 ex2_2(f2 x) { return pack2(ex2_approx(lo2(x)), ex2_approx(hi2(x))); }
__device__ __forceinline__ f2 both(float x) { return pack2(x, x); }

// gelu(x) = x Phi(x) = max(x, 0) - |x| q,  q = Phi(-|x|) = 2^P(|x|), two entries at a time.  P is this
// project's own minimax fit of log2 Phi(-t) on [0, 7] (degree 8, P(0) = -1, weighted so that q and t q are
// off by at most 5e-8; negative leading coefficient, so q goes to 0 beyond).  One special-function
// operation per entry and packed FMAs; written for -|x|: odd coefficients change sign.
__device__ __forceinline__ f2 phi_tail(f2 nax) {
    f2 p = fma2(both(-2.3347236037807306e-06f), nax, both(-3.3734937460394576e-05f));
    p = fma2(p, nax, both(-0.00016127918206620961f));
    p = fma2(p, nax, both(0.00019174156477674842f));
    p = fma2(p, nax, both(0.007126918528228998f));
    p = fma2(p, nax, both(0.052533652633428574f));
    p = fma2(p, nax, both(-0.4591982662677765f));
    p = fma2(p, nax, both(1.1511059999465942f));
    return ex2_2(fma2(p, nax, both(-1.f)));
}
__device__ __forceinline__ f2 neg_abs(f2 x) { return x | 0x8000000080000000ull; }
__device__ __forceinline__ f2 relu2(f2 x) { return pack2(fmaxf(lo2(x), 0.f), fmaxf(hi2(x), 0.f)); }
__device__ __forceinline__ f2 gelu2(f2 x) {
    const f2 nax = neg_abs(x);
    return fma2(nax, phi_tail(nax), relu2(x));
}
// ... and the derivative Phi(x) + x phi(x), phi the normal density 2^(-x^2 log2(e) / 2 - log2(sqrt(2 pi)))
__device__ __forceinline__ f2 gelu2_grad(f2 x, f2& grad) {
    const f2 nax = neg_abs(x);
    const f2 q = phi_tail(nax);
    const f2 h = fma2(q, both(-1.f), both(0.5f));
    const f2 c = (h & 0x7fffffff7fffffffull) | (x & 0x8000000080000000ull);
    const f2 dens = ex2_2(fma2(mul2(x, x), both(-0.72134752044448170f), both(-1.3257480647361593f)));
    grad = fma2(x, dens, fma2(c, both(1.f), both(0.5f)));
    return fma2(nax, q, relu2(x));
}
// v = hi + lo as two packed bf16 words
__device__ __forceinline__ void split2(f2 v, uint32_t& h, uint32_t& l) {
    h = pack_bf16(lo2(v), hi2(v));
    const f2 hf = pack2(__uint_as_float(h << 16), __uint_as_float(h & 0xffff0000u));
    const f2 r = fma2(hf, both(-1.f), v);
    l = pack_bf16(lo2(r), hi2(r));
}
__device__ __forceinline__ f2 unpack2(uint32_t w) { return pack2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u)); }

struct NetLayout {
    int h, r, m;
    int g0, c0, W1, b1, g1, c1, W2, b2, W3, b3, W4, b4, count;
    __host__ __device__ NetLayout(int h_, int r_) : h(h_), r(r_), m(8 * r_) {
        int o = 0;
        g0 = o; o += h; c0 = o; o += h;
        W1 = o; o += h * m; b1 = o; o += m;
        g1 = o; o += m; c1 = o; o += m;
        W2 = o; o += m * r; b2 = o; o += r;
        W3 = o; o += r * m; b3 = o; o += m;
        W4 = o; o += m * r; b4 = o; o += r;
        count = o;
    }
};

// ---------------------------------------------------------------------------
// Weights as shared-memory images (128-byte swizzle), fetched by plain bulk copies.  Groups of 64 columns j
// of the wide side (NG of them):
//   W1h, W1l  [NG][64 k][64 j]   diag(g0) W1 and what rounding it to bf16 left over: MN-major operand of
//                                p1 = n0 W1, K-major operand of dn0 = dp1 W1^T
//   W2c, W4c  [8r j][hi r | lo r]  diag(g1) W2, W4: MN-major operand of a2, f (both terms side by side, so that the hi
//                                term of the activations multiplies them in one instruction), K-major of da3
//   W3h, W3l  [NG][r c][64 j]    MN-major operand of p3, K-major operand of da2
//   W2t       [NG][r c][64 j]    (diag(g1) W2)^T: MN-major operand of dn1
// ---------------------------------------------------------------------------
template <int R> struct Bank {
    static constexpr int M = 8 * R, NG = M / 64, NH = NG / 2;
    static constexpr int kW1 = NG * 8192, kW3 = NG * R * 128, kWc = M * 128;
    static constexpr int W1h = 0, W1l = kW1, W2c = 2 * kW1, W3h = W2c + kWc, W3l = W3h + kW3, W4c = W3l + kW3, W2t = W4c + kWc;
    static constexpr int total = W2t + kW3;
};
constexpr size_t kBankBytes = Bank<32>::total;        // stride between the networks' banks

template <int R>
__global__ void __launch_bounds__(256)
ltc_bank_kernel(const float* __restrict__ params, uint8_t* __restrict__ bank, float* __restrict__ vec) {
    pdl_sync();
    using L = Bank<R>;
    const NetLayout nl(64, R);
    const int net = blockIdx.y, m = L::M;
    const float* P = params + (size_t)net * nl.count;
    uint8_t* B = bank + (size_t)net * kBankBytes;
    constexpr int n1 = 64 * L::M, n2 = R * L::M;       // weights of W1; of each of the others
    constexpr int kBlocks = (n1 + 3 * n2) / 256;
    if ((int)blockIdx.x < kBlocks) {
        int e = blockIdx.x * 256 + threadIdx.x;
        auto put = [&](int off, float v) { *reinterpret_cast<bf16*>(B + off) = __float2bfloat16_rn(v); };
        auto lo_of = [](float v) { return v - __bfloat162float(__float2bfloat16_rn(v)); };
        auto in_tile = [](int row, int col) { return (int)swz128_offset(row, col / 8) + (col % 8) * 2; };
        if (e < n1) {
            const int k = e / m, j = e % m;
            const float v = P[nl.g0 + k] * P[nl.W1 + e];
            const int o = (j / 64) * 8192 + in_tile(k, j % 64);
            put(L::W1h + o, v);
            put(L::W1l + o, lo_of(v));
            return;
        }
        e -= n1;
        const int which = e / n2;
        e -= which * n2;
        if (which == 1) {                              // W3 [c][j]
            const int c = e / m, j = e % m;
            const float v = P[nl.W3 + e];
            const int o = (j / 64) * (R * 128) + in_tile(c, j % 64);
            put(L::W3h + o, v);
            put(L::W3l + o, lo_of(v));
            return;
        }
        const int j = e / R, c = e % R;                // W2, W4 [j][c]
        const float v = which == 0 ? P[nl.g1 + j] * P[nl.W2 + e] : P[nl.W4 + e];
        const int base = which == 0 ? L::W2c : L::W4c;
        put(base + in_tile(j, c), v);
        put(base + in_tile(j, R + c), lo_of(v));
        if (which == 0) put(L::W2t + (j / 64) * (R * 128) + in_tile(c, j % 64), v);
        return;
    }
    // vectors: one warp per entry
    const int v = (blockIdx.x - kBlocks) * 8 + threadIdx.x / 32, lane = threadIdx.x % 32;
    if (v >= kVec) return;
    float s = 0.f, add = 0.f;
    if (v < kVb2) {                                    // b1' = c0 W1 + b1
        if (v < m) {
            add = P[nl.b1 + v];
            for (int k = lane; k < 64; k += 32) s = fmaf(P[nl.c0 + k], P[nl.W1 + k * m + v], s);
        }
    } else if (v < kVb3) {                             // b2' = c1 W2 + b2
        const int c = v - kVb2;
        if (c < R) {
            add = P[nl.b2 + c];
            for (int j = lane; j < m; j += 32) s = fmaf(P[nl.c1 + j], P[nl.W2 + j * R + c], s);
        }
    } else if (v < kVb4) {
        if (v - kVb3 < m) add = P[nl.b3 + v - kVb3];
    } else if (v < kVcs) {
        if (v - kVb4 < R) add = P[nl.b4 + v - kVb4];
    } else {                                           // 1^T diag(g1) W2
        const int c = v - kVcs;
        if (c < R)
            for (int j = lane; j < m; j += 32) s = fmaf(P[nl.g1 + j], P[nl.W2 + j * R + c], s);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) vec[(size_t)net * kVec + v] = s + add;
}

struct Slice {
    int H, n; int64_t sb, sh, sn;
    __device__ int64_t row(size_t R) const {
        const int bh = (int)(R / n), i = (int)(R % n);
        return (int64_t)(bh / H) * sb + (int64_t)(bh % H) * sh + (int64_t)i * sn;
    }
};

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&v)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(taddr) : "memory");
}
// one arrival per warp, after all its lanes
__device__ __forceinline__ void warp_arrive(uint64_t* bar) {
    __syncwarp();
    if (threadIdx.x % 32 == 0) mbar_arrive(bar);
}
// a shared-memory image in pieces of at most 32 KB
__device__ __forceinline__ void load_image(uint8_t* dst, const uint8_t* src, int bytes, uint64_t* bar) {
    for (int o = 0; o < bytes; o += 32768) bulk_load(dst + o, src + o, bytes - o < 32768 ? bytes - o : 32768, bar);
}

// ---------------------------------------------------------------------------
// Forward of one network (blockIdx.y) for tiles of 128 rows.  Persistent; two tiles (slots) in flight per CTA.
// Per slot: two warpgroups (thread = row, one half of every 64-column group each) and one issuing thread.
// Tensor memory of a slot, 256 columns: N 64 (n0, later a2, as hi/lo operand), two 64-column group
// buffers, O 2r.  A group buffer holds p, then in place gelu(p) as an operand, each warpgroup writing over the
// 32 columns it has read: 16 columns of hi pairs, 16 of lo.
// ---------------------------------------------------------------------------
template <int R> constexpr int kFwdSmem = Bank<R>::W2t + 1024;

template <int R>
__global__ void __launch_bounds__(576, 1)
ltc_dense_norm_kernel(Slice sl, const bf16* __restrict__ X, size_t row0, int tiles, const float2* __restrict__ st0,
                      const uint8_t* __restrict__ bank, const float* __restrict__ vec, bf16* __restrict__ a2, size_t a2_net,
                      float2* __restrict__ st1, size_t st1_net, float* __restrict__ f, size_t f_net, int* status) {
    using L = Bank<R>;
    constexpr int NG = L::NG;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* W = align1024(smem_raw);
    __shared__ uint64_t bar_w, bar_n[2], bar_s[2][2], bar_p[2][2], bar_f[2][2], bar_o[2];
    __shared__ uint32_t tm_slot;
    __shared__ __align__(16) float sv[kVec];
    __shared__ float2 s_part[2][2][128];
    const int tid = threadIdx.x, warp = warp_index(), net = blockIdx.y;
    if (tid == 0) {
        cta_giveup_init();
        mbar_init(&bar_w, 1);
        for (int s = 0; s < 2; ++s) {
            mbar_init(&bar_n[s], 8); mbar_init(&bar_o[s], 1);
            for (int b = 0; b < 2; ++b) { mbar_init(&bar_s[s][b], 1); mbar_init(&bar_p[s][b], 8); mbar_init(&bar_f[s][b], 1); }
        }
        mbar_fence_init();
    }
    pdl_sync();
    if (warp == 16) { tmem_alloc(&tm_slot, 512); tmem_relinquish(); }
    for (int e = tid; e < kVec; e += 576) sv[e] = vec[(size_t)net * kVec + e];
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tm = tm_slot;
    constexpr uint32_t cN = 0, cS = 64, cO = 192;
    if (warp >= 16) {
        // ============================ issuing threads ============================
        const int slot = warp - 16;
        if (elect_one()) {
            if (slot == 0) {
                mbar_expect_tx(&bar_w, L::W2t);
                load_image(W, bank + (size_t)net * kBankBytes, L::W2t, &bar_w);
            }
            const uint32_t t0 = tm + slot * 256;
            mbar_spin(&bar_w, 0, status, kErrTma);
            const uint32_t w = smem_u32(W);
            constexpr uint32_t id_s = idesc_bf16(128, 64, false, true), id_o = idesc_bf16(128, 2 * R, false, true),
                               id_l = idesc_bf16(128, R, false, true);
            uint32_t it = 0, pp[2] = {0, 0}, pf[2] = {0, 0};
            for (int tile = blockIdx.x * 2 + slot; tile < tiles; tile += 2 * gridDim.x) {
#pragma unroll
                for (int layer = 0; layer < 2; ++layer, ++it) {
                    mbar_spin(&bar_n[slot], it & 1, status, kErrMma);
                    tc_fence_after();
                    const uint64_t bh = smem_desc(w + (layer ? L::W3h : L::W1h), 0, 1024, kSwz128);
                    const uint64_t bl = smem_desc(w + (layer ? L::W3l : L::W1l), 0, 1024, kSwz128);
                    const uint64_t oc = smem_desc(w + (layer ? L::W4c : L::W2c), 0, 1024, kSwz128);
                    constexpr uint32_t kG1 = 8192, kG3 = R * 128;
                    auto groups = [&](int g) {          // columns 64 g of p1 = n0 W1 or p3 = a2 W3
                        const uint32_t go = g * (layer ? kG3 : kG1);
                        const int ks = layer ? R / 16 : 4;
#pragma unroll
                        for (int part = 0; part < 3; ++part)
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                if (k >= ks) break;
                                // n0: halves of 32 columns, [hi 16 | lo 16]; a2: 16 entries, [hi 8 | lo 8]
                                const uint32_t a = layer ? k * 16 + (part == 1 ? 8 : 0) : (k / 2) * 32 + (k % 2) * 8 + (part == 1 ? 16 : 0);
                                umma_ts(t0 + cS + (g & 1) * 64, t0 + cN + a, desc_off(part == 2 ? bl : bh, go + k * 2048), id_s, (part > 0 || k > 0) ? 1u : 0u);
                            }
                        umma_commit(&bar_s[slot][g & 1]);
                    };
                    groups(0);
                    groups(1);
#pragma unroll
                    for (int g = 0; g < NG; ++g) {
                        const int b = g & 1;
                        mbar_spin(&bar_p[slot][b], pp[b], status, kErrMma);
                        pp[b] ^= 1;
                        tc_fence_after();
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const uint32_t a = t0 + cS + b * 64 + (k / 2) * 32 + (k % 2) * 8;
                            const uint64_t bo = desc_off(oc, g * 8192 + k * 2048);
                            umma_ts(t0 + cO, a, bo, id_o, (g > 0 || k > 0) ? 1u : 0u);
                            umma_ts(t0 + cO, a + 16, bo, id_l, 1u);
                        }
                        if (g + 2 < NG) {
                            umma_commit(&bar_f[slot][b]);
                            mbar_spin(&bar_f[slot][b], pf[b], status, kErrMma);
                            pf[b] ^= 1;
                            groups(g + 2);
                        }
                    }
                    umma_commit(&bar_o[slot]);
                }
            }
        }
    } else {
        // ============================ rows ============================
        const int wg = warp / 4, slot = wg & 1, half = wg >> 1, wt = tid % 128;
        const uint32_t t0 = tm + slot * 256 + ((uint32_t)((warp % 4) * 32) << 16);
        const bool narrow = half < R / 16;              // this half has 16 of the r narrow columns
        const int c16 = half * 16;
        uint32_t ps[2] = {0, 0}, po = 0;
        uint4 xv[4];
        float2 s0 = make_float2(0.f, 0.f);
        auto load_x = [&](int tile) {
            const uint4* src = reinterpret_cast<const uint4*>(X + sl.row(row0 + (size_t)tile * 128 + wt) + 32 * half);
#pragma unroll
            for (int q = 0; q < 4; ++q) xv[q] = src[q];
            s0 = st0[(size_t)tile * 128 + wt];
        };
        int tile = blockIdx.x * 2 + slot;
        if (tile < tiles) load_x(tile);
        for (; tile < tiles; tile += 2 * gridDim.x) {
            const size_t row = (size_t)tile * 128 + wt;
            {
                uint32_t h[16], l[16];
                const f2 mu = both(-s0.x), rs = both(s0.y);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t u[4] = {xv[q].x, xv[q].y, xv[q].z, xv[q].w};
#pragma unroll
                    for (int i = 0; i < 4; ++i) split2(mul2(fma2(unpack2(u[i]), both(1.f), mu), rs), h[4 * q + i], l[4 * q + i]);
                }
                tmem_st16(t0 + cN + 32 * half, h);
                tmem_st16(t0 + cN + 32 * half + 16, l);
                tmem_st_wait();
                tc_fence_before();
                warp_arrive(&bar_n[slot]);
            }
            f2 sum = 0ull, sq = 0ull;
            // p -> gelu(p) of this half of a group, back as an operand
            auto group = [&](int g, const float* bias, bool stats) {
                const int b = g & 1;
                const uint32_t ta = t0 + cS + b * 64 + 32 * half;
                mbar_wait(&bar_s[slot][b], ps[b], status, kErrMma);
                ps[b] ^= 1;
                tc_fence_after();
                uint32_t u[32];
                tmem_ld32(ta, u);
                tmem_ld_wait();
                uint32_t h[16], l[16];
                const float* bp = bias + g * 64 + 32 * half;
#pragma unroll
                for (int i = 0; i < 16; i += 2) {
                    const cc::F22 bb = cc::lds22(bp + 2 * i);
                    const f2 g0 = gelu2(fma2(pack2(__uint_as_float(u[2 * i]), __uint_as_float(u[2 * i + 1])), both(1.f), bb.x));
                    const f2 g1 = gelu2(fma2(pack2(__uint_as_float(u[2 * i + 2]), __uint_as_float(u[2 * i + 3])), both(1.f), bb.y));
                    if (stats) {
                        sum = fma2(g0, both(1.f), sum); sum = fma2(g1, both(1.f), sum);
                        sq = fma2(g0, g0, sq); sq = fma2(g1, g1, sq);
                    }
                    split2(g0, h[i], l[i]);
                    split2(g1, h[i + 1], l[i + 1]);
                }
                tmem_st16(ta, h);
                tmem_st16(ta + 16, l);
                tmem_st_wait();
                tc_fence_before();
                warp_arrive(&bar_p[slot][b]);
            };
#pragma unroll 1
            for (int g = 0; g < NG; g += 2) { group(g, sv, true); group(g + 1, sv, true); }
            s_part[slot][half][wt] = make_float2(lo2(sum) + hi2(sum), lo2(sq) + hi2(sq));
            asm volatile("bar.sync %0, 256;" ::"r"(slot + 1) : "memory");
            const float2 q0 = s_part[slot][0][wt], q1 = s_part[slot][1][wt];
            constexpr float inv = 1.f / (float)L::M;
            const float mu1 = (q0.x + q1.x) * inv;
            const float rs1 = rsqrtf(fmaxf((q0.y + q1.y) * inv - mu1 * mu1, 0.f) + kLnEps);
            if (half == 0 && st1 != nullptr) st1[net * st1_net + row] = make_float2(mu1, rs1);
            // this thread's 16 of the r columns of O: both terms of the weights added up
            auto read_o = [&](float (&o)[16]) {
                mbar_wait(&bar_o[slot], po, status, kErrMma);
                po ^= 1;
                tc_fence_after();
                if (narrow) {
                    uint32_t u[16], v[16];
                    tmem_ld16(t0 + cO + c16, u);
                    tmem_ld16(t0 + cO + R + c16, v);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 16; ++i) o[i] = __uint_as_float(u[i]) + __uint_as_float(v[i]);
                }
            };
            {
                float o[16];
                read_o(o);
                if (narrow) {
                    uint32_t h[8], l[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int c = c16 + 2 * i;
                        const f2 v = pack2(fmaf(rs1, fmaf(-mu1, sv[kVcs + c], o[2 * i]), sv[kVb2 + c]),
                                           fmaf(rs1, fmaf(-mu1, sv[kVcs + c + 1], o[2 * i + 1]), sv[kVb2 + c + 1]));
                        split2(v, h[i], l[i]);
                    }
                    tmem_st8(t0 + cN + 16 * half, h);
                    tmem_st8(t0 + cN + 16 * half + 8, l);
                    tmem_st_wait();
                    if (a2 != nullptr) {                // rows of 64: [hi r | lo r]
                        uint4* dst = reinterpret_cast<uint4*>(a2 + net * a2_net + row * 64 + c16);
                        dst[0] = make_uint4(h[0], h[1], h[2], h[3]);
                        dst[1] = make_uint4(h[4], h[5], h[6], h[7]);
                        dst[R / 8] = make_uint4(l[0], l[1], l[2], l[3]);
                        dst[R / 8 + 1] = make_uint4(l[4], l[5], l[6], l[7]);
                    }
                }
                tc_fence_before();
                warp_arrive(&bar_n[slot]);
            }
#pragma unroll 1
            for (int g = 0; g < NG; g += 2) { group(g, sv + kVb3, false); group(g + 1, sv + kVb3, false); }
            if (tile + 2 * (int)gridDim.x < tiles) load_x(tile + 2 * gridDim.x);      // in flight during the last product
            {
                float o[16];
                read_o(o);
                if (narrow) {
                    float4* dst = reinterpret_cast<float4*>(f + net * f_net + row * R + c16);
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        dst[i] = make_float4(o[4 * i] + sv[kVb4 + c16 + 4 * i], o[4 * i + 1] + sv[kVb4 + c16 + 4 * i + 1],
                                             o[4 * i + 2] + sv[kVb4 + c16 + 4 * i + 2], o[4 * i + 3] + sv[kVb4 + c16 + 4 * i + 3]);
                }
                tc_fence_before();
            }
        }
    }
    // (every MMA has completed: the rows waited for the last product of every tile)
    tc_fence_before();
    __syncthreads();
    cta_teardown(warp >= 16, warp - 16);
    if (warp == 16) tmem_dealloc(tm, 512);
}

// ---------------------------------------------------------------------------
// Layers 4 and 3 backward of one network (blockIdx.y), persistent, one tile of 128 rows at a time:
//   p3 = a2 W3 + b3,  da3 = df W4^T,  dp3 = da3 gelu'(p3),  a3 = gelu(p3)
//   da2 = dp3 W3^T,   dW4 += a3^T df,  dW3 += dp3^T a2      and the column sums of dp3 and df.
// Warps 0-15 (thread = row): warpgroups w and w + 2 take the groups of parity w, a half of 32 columns each; two
// groups are in tensor memory at a time (p3 and da3, 64 columns each).  Their a3 and dp3 go to shared memory
// as bf16 tiles, 128 columns (a step) at a time, the operands of the last three products.  Warp 16: one
// thread loads and issues every MMA; the next step's p3, da3 are formed while the rows work on this one's.
// Warps 17, 18: column sums, from the same tiles.
// ---------------------------------------------------------------------------
constexpr int kBwdThreads = 19 * 32;

// sums of two columns (this lane's) of a [128 x 64] bf16 tile
__device__ __forceinline__ void tile_column_sums(const uint8_t* t, int lane, float& s0, float& s1) {
    const uint8_t* p = t + (lane % 4) * 4;
#pragma unroll 8
    for (int row = 0; row < 128; ++row) {
        const uint32_t w = *reinterpret_cast<const uint32_t*>(p + swz128_offset(row, lane / 4));
        s0 += __uint_as_float(w << 16);
        s1 += __uint_as_float(w & 0xffff0000u);
    }
}
__device__ __forceinline__ void red_add4(float* dst, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dst), "f"(__uint_as_float(a)), "f"(__uint_as_float(b)),
                 "f"(__uint_as_float(c)), "f"(__uint_as_float(d)) : "memory");
}
// 16 accumulator columns of this thread's row into a gradient row
__device__ __forceinline__ void add_columns16(uint32_t taddr, float* dst) {
    uint32_t u[16];
    tmem_ld16(taddr, u);
    tmem_ld_wait();
#pragma unroll
    for (int j = 0; j < 16; j += 4) red_add4(dst + j, u[j], u[j + 1], u[j + 2], u[j + 3]);
}
// 32 columns (16 packed words) of a row into a [128 x 64] tile, half 0 or 1
__device__ __forceinline__ void tile_put32(uint8_t* tile, int row, int half, const uint32_t (&v)[16]) {
#pragma unroll
    for (int j = 0; j < 4; ++j)
        *reinterpret_cast<uint4*>(tile + swz128_offset(row, 4 * half + j)) = make_uint4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
}

template <int R> struct Bwd34 {
    static constexpr int W = Bank<R>::W2t - Bank<R>::W3h;               // W3h | W3l | W4c
    static constexpr int T = W, In = T + 4 * 16384, kIn = 32768;        // a3, dp3 of a step; three (a2, df) inputs
    static constexpr int bytes = In + 3 * kIn + 1024;
};

template <int R>
__global__ void __launch_bounds__(kBwdThreads, 1)
ltc_wgrad_kernel(const __grid_constant__ CUtensorMap mA0, const __grid_constant__ CUtensorMap mA1, const __grid_constant__ CUtensorMap mD0,
                 const __grid_constant__ CUtensorMap mD1, size_t row0, int tiles, const uint8_t* __restrict__ bank,
                 const float* __restrict__ vec, bf16* __restrict__ da2, size_t da2_net, float2* __restrict__ mm, size_t mm_net,
                 float* __restrict__ G, float* __restrict__ sums, int* status) {
    using L = Bank<R>;
    using B = Bwd34<R>;
    constexpr int NH = L::NH;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    __shared__ uint64_t bar_w, bar_ld[3], bar_s[2], bar_rd[2], bar_t, bar_free;
    __shared__ uint32_t tm_slot;
    __shared__ __align__(16) float sb3[256];
    __shared__ float scs[R], sb2[R];
    const int tid = threadIdx.x, warp = warp_index(), lane = tid % 32, net = blockIdx.y;
    const int nt = (tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x, steps = nt * NH;
    const CUtensorMap* mA = net ? &mA1 : &mA0;
    const CUtensorMap* mD = net ? &mD1 : &mD0;
    if (tid == 0) {
        cta_giveup_init();
        mbar_init(&bar_w, 1);
        for (int i = 0; i < 3; ++i) mbar_init(&bar_ld[i], 1);
        for (int b = 0; b < 2; ++b) { mbar_init(&bar_s[b], 1); mbar_init(&bar_rd[b], 8); }
        mbar_init(&bar_t, 16);
        mbar_init(&bar_free, 3);
        mbar_fence_init();
    }
    pdl_sync();
    if (warp == 16) { tmem_alloc(&tm_slot, 512); tmem_relinquish(); }
    for (int e = tid; e < 256; e += kBwdThreads) sb3[e] = vec[(size_t)net * kVec + kVb3 + e];
    if (tid < R) { scs[tid] = vec[(size_t)net * kVec + kVcs + tid]; sb2[tid] = vec[(size_t)net * kVec + kVb2 + tid]; }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tm = tm_slot;
    constexpr uint32_t cDa2 = 256, cW4 = 256 + 32, cW3 = cW4 + 64;
    auto tile_at = [&](int i) { return (int)blockIdx.x + i * (int)gridDim.x; };
    if (warp == 16) {
        if (elect_one()) {
            auto load = [&](int i) {
                uint8_t* dst = smem + B::In + (i % 3) * B::kIn;
                mbar_expect_tx(&bar_ld[i % 3], B::kIn);
                tma_load_2d(dst, mA, 0, (int)row0 + tile_at(i) * 128, &bar_ld[i % 3]);
                tma_load_2d(dst + 16384, mD, 0, tile_at(i) * 128, &bar_ld[i % 3]);
            };
            mbar_expect_tx(&bar_w, B::W);
            load_image(smem, bank + (size_t)net * kBankBytes + L::W3h, B::W, &bar_w);
            load(0);
            if (nt > 1) load(1);
            mbar_spin(&bar_w, 0, status, kErrTma);
            const uint32_t sw = smem_u32(smem);
            constexpr uint32_t w3h = 0, w3l = L::W3l - L::W3h, w4c = L::W4c - L::W3h, kG3 = R * 128;
            constexpr uint32_t id_s = idesc_bf16(128, 64, false, true), id_d = idesc_bf16(128, 64, false, false),
                               id_a = idesc_bf16(128, R, false, false), id_w = idesc_bf16(128, R, true, true);
            auto form = [&](int k) {                   // p3 and da3 of step k
                const int i = k / NH, hf = k % NH;
                if (hf == 0) mbar_spin(&bar_ld[i % 3], (i / 3) & 1, status, kErrTma);
                const uint32_t in = sw + B::In + (i % 3) * B::kIn;
                const uint64_t ad = smem_desc(in, 0, 1024, kSwz128), dd = smem_desc(in + 16384, 0, 1024, kSwz128);
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const int g = 2 * hf + b;
                    if (k > 0) mbar_spin(&bar_rd[b], (k - 1) & 1, status, kErrMma);
                    tc_fence_after();
                    const uint64_t bh = smem_desc(sw + w3h + g * kG3, 0, 1024, kSwz128), bl = smem_desc(sw + w3l + g * kG3, 0, 1024, kSwz128);
                    const uint64_t w4 = smem_desc(sw + w4c + g * 8192, 0, 1024, kSwz128);
#pragma unroll
                    for (int part = 0; part < 3; ++part)
#pragma unroll
                        for (int q = 0; q < R / 16; ++q)
                            umma_ss(tm + b * 128, desc_off(ad, q * 32 + (part == 1 ? 2 * R : 0)), desc_off(part == 2 ? bl : bh, q * 2048), id_s,
                                    (part > 0 || q > 0) ? 1u : 0u);
#pragma unroll
                    for (int q = 0; q < R / 16; ++q)
                        umma_ss(tm + b * 128 + 64, desc_off(dd, q * 32), desc_off(w4, q * 32), id_d, q > 0 ? 1u : 0u);
                    umma_commit(&bar_s[b]);
                }
            };
            form(0);
            for (int k = 0; k < steps; ++k) {
                const int i = k / NH, hf = k % NH;
                if (k + 1 < steps) form(k + 1);
                if (!mbar_spin(&bar_t, k & 1, status, kErrMma)) break;       // (gave up: no more copies are asked for)
                tc_fence_after();
                // tile i - 1 is done with (its last products have completed, its da2 has been read): its input buffer
                // takes tile i + 2
                if (hf == 0 && i + 2 < nt) load(i + 2);
                const uint32_t in = sw + B::In + (i % 3) * B::kIn, t3 = sw + B::T, td = t3 + 32768;
                const uint64_t dk = smem_desc(td, 0, 1024, kSwz128);
                const uint64_t am = smem_desc(t3, 16384, 1024, kSwz128), dm = smem_desc(td, 16384, 1024, kSwz128);
                const uint64_t a2b = smem_desc(in, 0, 1024, kSwz128), dfb = smem_desc(in + 16384, 0, 1024, kSwz128);
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    umma_ss(tm + cDa2, desc_off(dk, (q / 4) * 16384 + (q % 4) * 32),
                            desc_off(smem_desc(sw + w3h + (2 * hf + q / 4) * kG3, 0, 1024, kSwz128), (q % 4) * 32), id_a, (hf > 0 || q > 0) ? 1u : 0u);
#pragma unroll
                for (int q = 0; q < 8; ++q) umma_ss(tm + cW4 + hf * R, desc_off(am, q * 2048), desc_off(dfb, q * 2048), id_w, (i > 0 || q > 0) ? 1u : 0u);
#pragma unroll
                for (int q = 0; q < 8; ++q) umma_ss(tm + cW3 + hf * R, desc_off(dm, q * 2048), desc_off(a2b, q * 2048), id_w, (i > 0 || q > 0) ? 1u : 0u);
                umma_commit(&bar_free);
            }
            if (steps > 0) mbar_spin(&bar_free, (steps - 1) & 1, status, kErrMma);
        }
    } else if (warp > 16) {
        const int j = warp - 17;                       // atom j of dp3; warp 17 also df
        float s[2][2] = {{0.f, 0.f}, {0.f, 0.f}}, d0 = 0.f, d1 = 0.f;
        for (int k = 0; k < steps; ++k) {
            const int i = k / NH, hf = k % NH;
            mbar_wait(&bar_t, k & 1, status, kErrMma);
            if (NH > 1 && hf == 1) tile_column_sums(smem + B::T + 32768 + j * 16384, lane, s[1][0], s[1][1]);
            else tile_column_sums(smem + B::T + 32768 + j * 16384, lane, s[0][0], s[0][1]);
            if (j == 0 && hf == 0) {
                mbar_wait(&bar_ld[i % 3], (i / 3) & 1, status, kErrTma);
                tile_column_sums(smem + B::In + (i % 3) * B::kIn + 16384, lane, d0, d1);
            }
            warp_arrive(&bar_free);
        }
        float* s_dp3 = sums + (size_t)net * kSums + 320;
#pragma unroll
        for (int hf = 0; hf < NH; ++hf) {
            atomicAdd(s_dp3 + hf * 128 + j * 64 + 2 * lane, s[hf][0]);
            atomicAdd(s_dp3 + hf * 128 + j * 64 + 2 * lane + 1, s[hf][1]);
        }
        if (j == 0 && 2 * lane < R) {
            atomicAdd(sums + (size_t)net * kSums + 576 + 2 * lane, d0);
            atomicAdd(sums + (size_t)net * kSums + 576 + 2 * lane + 1, d1);
        }
    } else {
        const int wg = warp / 4, p = wg & 1, half = wg >> 1, wt = tid % 128;
        const uint32_t lane_tm = tm + ((uint32_t)((warp % 4) * 32) << 16);
        // da2 of tile i, 16 columns per warpgroup: stored, and this part of the two row sums of the normalisation's
        // backward, da2 . (1^T W2) and da2 . (a2 - b2), over 8r
        auto finish_tile = [&](int i) {
            if (wg >= R / 16) return;
            const int c0 = 16 * wg;
            const size_t row = (size_t)tile_at(i) * 128 + wt;
            uint32_t u[16];
            tmem_ld16(lane_tm + cDa2 + c0, u);
            tmem_ld_wait();
            const uint8_t* ta = smem + B::In + (i % 3) * B::kIn;
            mbar_wait(&bar_ld[i % 3], (i / 3) & 1, status, kErrTma);
            float m1 = 0.f, m2 = 0.f;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const uint4 h = *reinterpret_cast<const uint4*>(ta + swz128_offset(wt, c0 / 8 + q));
                const uint4 l = *reinterpret_cast<const uint4*>(ta + swz128_offset(wt, (R + c0) / 8 + q));
                const uint32_t hw[4] = {h.x, h.y, h.z, h.w}, lw[4] = {l.x, l.y, l.z, l.w};
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int c = c0 + 8 * q + e;
                    const float v = __uint_as_float(u[8 * q + e]);
                    const float a = __uint_as_float((e & 1) ? (hw[e / 2] & 0xffff0000u) : (hw[e / 2] << 16)) +
                                    __uint_as_float((e & 1) ? (lw[e / 2] & 0xffff0000u) : (lw[e / 2] << 16));
                    m1 = fmaf(v, scs[c], m1);
                    m2 = fmaf(v, a - sb2[c], m2);
                }
            }
            uint32_t pk[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) pk[e] = pack_bf16(__uint_as_float(u[2 * e]), __uint_as_float(u[2 * e + 1]));
            uint4* dst = reinterpret_cast<uint4*>(da2 + net * da2_net + row * 64 + c0);
            dst[0] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            dst[1] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
            constexpr float inv = 1.f / (float)L::M;
            mm[net * mm_net + row * 2 + wg] = make_float2(m1 * inv, m2 * inv);
        };
        for (int k = 0; k < steps; ++k) {
            const int i = k / NH, hf = k % NH;
            const uint32_t ta = lane_tm + p * 128 + 32 * half;
            const float* bp = sb3 + (2 * hf + p) * 64 + 32 * half;
            mbar_wait(&bar_s[p], k & 1, status, kErrMma);
            tc_fence_after();
            uint32_t a3[16], dp[16];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                uint32_t u[16], v[16];
                tmem_ld16(ta + 16 * q, u);
                tmem_ld16(ta + 64 + 16 * q, v);
                tmem_ld_wait();
                if (q == 1) { tc_fence_before(); warp_arrive(&bar_rd[p]); }
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const f2 bb = *reinterpret_cast<const f2*>(bp + 16 * q + 2 * e);
                    f2 gr;
                    const f2 g = gelu2_grad(fma2(pack2(__uint_as_float(u[2 * e]), __uint_as_float(u[2 * e + 1])), both(1.f), bb), gr);
                    const f2 d = mul2(pack2(__uint_as_float(v[2 * e]), __uint_as_float(v[2 * e + 1])), gr);
                    a3[8 * q + e] = pack_bf16(lo2(g), hi2(g));
                    dp[8 * q + e] = pack_bf16(lo2(d), hi2(d));
                }
            }
            if (k > 0) mbar_wait(&bar_free, (k - 1) & 1, status, kErrMma);
            tc_fence_after();
            if (hf == 0 && i > 0) finish_tile(i - 1);
            tile_put32(smem + B::T + p * 16384, wt, half, a3);
            tile_put32(smem + B::T + 32768 + p * 16384, wt, half, dp);
            fence_proxy_async_smem();
            tc_fence_before();
            warp_arrive(&bar_t);
        }
        if (steps > 0) {
            mbar_wait(&bar_free, (steps - 1) & 1, status, kErrMma);
            tc_fence_after();
            finish_tile(nt - 1);
            if (wg < 2 * NH) {                         // one of the gradient accumulators each
                const int hf = wg % NH, which = wg / NH;
                float* dst = G + ((size_t)net * 4 + (which ? 2 : 3)) * kMat + (size_t)(hf * 128 + wt) * 64;
#pragma unroll
                for (int c = 0; c < R; c += 16) add_columns16(lane_tm + (which ? cW3 : cW4) + hf * R + c, dst + c);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 16) { cta_teardown_warp(); tmem_dealloc(tm, 512); }
}

// ---------------------------------------------------------------------------
// Layers 2 and 1 backward of one network, in the manner of ltc_wgrad_kernel:
//   p1 = n0 W1 + b1',  n1 = rs1 (gelu(p1) - mu1),  dn1 = da2 (diag(g1) W2)^T,
//   dp1 = rs1 (dn1 - m1 - n1 m2) gelu'(p1),   m1, m2 the mean of dn1 and of dn1 n1 (from ltc_wgrad_kernel)
//   dn0 = dp1 W1^T,   dW2 += n1^T da2,   dW1 += dp1^T n0      and the column sums of dp1 and da2.
// Inputs by TMA: da2 and the hi terms of n0 in two buffers, the lo terms (needed only for p1) in one.
// ---------------------------------------------------------------------------
template <int R> struct Bwd12 {
    static constexpr int W1 = 0, W2t = 2 * Bank<R>::kW1, T = W2t + Bank<R>::kW3;       // T: n1, dp1 of a step
    static constexpr int In = T + 4 * 16384, kIn = 32768, Lo = In + 2 * kIn;
    static constexpr int bytes = Lo + 16384 + 1024;
};

template <int R>
__global__ void __launch_bounds__(kBwdThreads, 1)
ltc_dense_bwd_norm_kernel(const __grid_constant__ CUtensorMap mN, const __grid_constant__ CUtensorMap mNlo,
                          const __grid_constant__ CUtensorMap mD0, const __grid_constant__ CUtensorMap mD1, size_t row0, int tiles,
                          const uint8_t* __restrict__ bank, const float* __restrict__ vec, const float2* __restrict__ st1, size_t st1_net,
                          const float2* __restrict__ mm, size_t mm_net, float* __restrict__ dn0, size_t dn0_net,
                          float* __restrict__ G, float* __restrict__ sums, int* status) {
    using L = Bank<R>;
    using B = Bwd12<R>;
    constexpr int NH = L::NH;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    __shared__ uint64_t bar_w, bar_ld[2], bar_lo, bar_s[2], bar_rd[2], bar_t, bar_free;
    __shared__ uint32_t tm_slot;
    __shared__ __align__(16) float sb1[256];
    const int tid = threadIdx.x, warp = warp_index(), lane = tid % 32, net = blockIdx.y;
    const int nt = (tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x, steps = nt * NH;
    const CUtensorMap* mD = net ? &mD1 : &mD0;
    if (tid == 0) {
        cta_giveup_init();
        mbar_init(&bar_w, 1); mbar_init(&bar_lo, 1);
        for (int b = 0; b < 2; ++b) { mbar_init(&bar_ld[b], 1); mbar_init(&bar_s[b], 1); mbar_init(&bar_rd[b], 8); }
        mbar_init(&bar_t, 16);
        mbar_init(&bar_free, 3);
        mbar_fence_init();
    }
    pdl_sync();
    if (warp == 16) { tmem_alloc(&tm_slot, 512); tmem_relinquish(); }
    for (int e = tid; e < 256; e += kBwdThreads) sb1[e] = vec[(size_t)net * kVec + e];
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tm = tm_slot;
    constexpr uint32_t cN0 = 256, cW2 = cN0 + 64, cW1 = cW2 + 64;
    auto tile_at = [&](int i) { return (int)blockIdx.x + i * (int)gridDim.x; };
    if (warp == 16) {
        if (elect_one()) {
            auto load = [&](int i) {
                uint8_t* dst = smem + B::In + (i & 1) * B::kIn;
                mbar_expect_tx(&bar_ld[i & 1], B::kIn);
                tma_load_2d(dst, mD, 0, tile_at(i) * 128, &bar_ld[i & 1]);
                tma_load_2d(dst + 16384, &mN, 0, tile_at(i) * 128, &bar_ld[i & 1]);
            };
            auto load_lo = [&](int i) {
                mbar_expect_tx(&bar_lo, 16384);
                tma_load_2d(smem + B::Lo, &mNlo, 0, tile_at(i) * 128, &bar_lo);
            };
            mbar_expect_tx(&bar_w, B::T);
            load_image(smem, bank + (size_t)net * kBankBytes + L::W1h, 2 * L::kW1, &bar_w);
            load_image(smem + B::W2t, bank + (size_t)net * kBankBytes + L::W2t, L::kW3, &bar_w);
            load(0);
            load_lo(0);
            mbar_spin(&bar_w, 0, status, kErrTma);
            const uint32_t sw = smem_u32(smem);
            constexpr uint32_t w1l = L::kW1, kG3 = R * 128;
            constexpr uint32_t id_s = idesc_bf16(128, 64, false, true), id_n = idesc_bf16(128, 64, false, false),
                               id_w2 = idesc_bf16(128, R, true, true), id_w1 = idesc_bf16(128, 64, true, true);
            const uint64_t nl = smem_desc(sw + B::Lo, 0, 1024, kSwz128);
            auto form = [&](int k) {                   // p1 and dn1 of step k
                const int i = k / NH, hf = k % NH;
                // (a wait in front of a copy that gave up: no more copies are asked for)
                if (k > 0 && (!mbar_spin(&bar_rd[0], (k - 1) & 1, status, kErrMma) || !mbar_spin(&bar_rd[1], (k - 1) & 1, status, kErrMma))) return false;
                if (hf == 0) {
                    if (i > 0) load_lo(i);             // (the last products that read it have completed: they were read out)
                    mbar_spin(&bar_ld[i & 1], (i >> 1) & 1, status, kErrTma);
                    mbar_spin(&bar_lo, i & 1, status, kErrTma);
                }
                tc_fence_after();
                const uint32_t in = sw + B::In + (i & 1) * B::kIn;
                const uint64_t dd = smem_desc(in, 0, 1024, kSwz128), nh = smem_desc(in + 16384, 0, 1024, kSwz128);
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const int g = 2 * hf + b;
                    const uint64_t bh = smem_desc(sw + g * 8192, 0, 1024, kSwz128), bl = smem_desc(sw + w1l + g * 8192, 0, 1024, kSwz128);
                    const uint64_t w2 = smem_desc(sw + B::W2t + g * kG3, 0, 1024, kSwz128);
#pragma unroll
                    for (int part = 0; part < 3; ++part)
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            umma_ss(tm + b * 128, desc_off(part == 1 ? nl : nh, q * 32), desc_off(part == 2 ? bl : bh, q * 2048), id_s,
                                    (part > 0 || q > 0) ? 1u : 0u);
#pragma unroll
                    for (int q = 0; q < R / 16; ++q)
                        umma_ss(tm + b * 128 + 64, desc_off(dd, q * 32), desc_off(w2, q * 2048), id_s, q > 0 ? 1u : 0u);
                    umma_commit(&bar_s[b]);
                }
                return true;
            };
            form(0);
            for (int k = 0; k < steps; ++k) {
                const int i = k / NH, hf = k % NH;
                if (hf == 0 && i + 1 < nt) {           // the other input buffer: tile i - 1 is done with
                    if (k > 0 && !mbar_spin(&bar_free, (k - 1) & 1, status, kErrMma)) break;
                    load(i + 1);
                }
                if (k + 1 < steps && !form(k + 1)) break;
                mbar_spin(&bar_t, k & 1, status, kErrMma);
                tc_fence_after();
                const uint32_t in = sw + B::In + (i & 1) * B::kIn, t1 = sw + B::T, td = t1 + 32768;
                const uint64_t dk = smem_desc(td, 0, 1024, kSwz128);
                const uint64_t nm = smem_desc(t1, 16384, 1024, kSwz128), dm = smem_desc(td, 16384, 1024, kSwz128);
                const uint64_t dab = smem_desc(in, 0, 1024, kSwz128), n0b = smem_desc(in + 16384, 0, 1024, kSwz128);
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    umma_ss(tm + cN0, desc_off(dk, (q / 4) * 16384 + (q % 4) * 32),
                            desc_off(smem_desc(sw + (2 * hf + q / 4) * 8192, 0, 1024, kSwz128), (q % 4) * 32), id_n, (hf > 0 || q > 0) ? 1u : 0u);
#pragma unroll
                for (int q = 0; q < 8; ++q) umma_ss(tm + cW2 + hf * R, desc_off(nm, q * 2048), desc_off(dab, q * 2048), id_w2, (i > 0 || q > 0) ? 1u : 0u);
#pragma unroll
                for (int q = 0; q < 8; ++q) umma_ss(tm + cW1 + hf * 64, desc_off(dm, q * 2048), desc_off(n0b, q * 2048), id_w1, (i > 0 || q > 0) ? 1u : 0u);
                umma_commit(&bar_free);
            }
            if (steps > 0) mbar_spin(&bar_free, (steps - 1) & 1, status, kErrMma);
        }
    } else if (warp > 16) {
        const int j = warp - 17;                       // atom j of dp1; warp 17 also da2
        float s[2][2] = {{0.f, 0.f}, {0.f, 0.f}}, d0 = 0.f, d1 = 0.f;
        for (int k = 0; k < steps; ++k) {
            const int i = k / NH, hf = k % NH;
            mbar_wait(&bar_t, k & 1, status, kErrMma);
            if (NH > 1 && hf == 1) tile_column_sums(smem + B::T + 32768 + j * 16384, lane, s[1][0], s[1][1]);
            else tile_column_sums(smem + B::T + 32768 + j * 16384, lane, s[0][0], s[0][1]);
            if (j == 0 && hf == 0) {
                mbar_wait(&bar_ld[i & 1], (i >> 1) & 1, status, kErrTma);
                tile_column_sums(smem + B::In + (i & 1) * B::kIn, lane, d0, d1);
            }
            warp_arrive(&bar_free);
        }
        float* s_dp1 = sums + (size_t)net * kSums;
#pragma unroll
        for (int hf = 0; hf < NH; ++hf) {
            atomicAdd(s_dp1 + hf * 128 + j * 64 + 2 * lane, s[hf][0]);
            atomicAdd(s_dp1 + hf * 128 + j * 64 + 2 * lane + 1, s[hf][1]);
        }
        if (j == 0 && 2 * lane < R) {
            atomicAdd(sums + (size_t)net * kSums + 256 + 2 * lane, d0);
            atomicAdd(sums + (size_t)net * kSums + 256 + 2 * lane + 1, d1);
        }
    } else {
        const int wg = warp / 4, p = wg & 1, half = wg >> 1, wt = tid % 128;
        const uint32_t lane_tm = tm + ((uint32_t)((warp % 4) * 32) << 16);
        auto finish_tile = [&](int i) {                // dn0, 16 columns per warpgroup
            uint32_t u[16];
            tmem_ld16(lane_tm + cN0 + 16 * wg, u);
            tmem_ld_wait();
            uint4* dst = reinterpret_cast<uint4*>(dn0 + net * dn0_net + ((size_t)tile_at(i) * 128 + wt) * 64 + 16 * wg);
#pragma unroll
            for (int q = 0; q < 4; ++q) dst[q] = make_uint4(u[4 * q], u[4 * q + 1], u[4 * q + 2], u[4 * q + 3]);
        };
        // mu1, rs1, m1, m2 of this thread's row, requested a tile ahead
        float2 nst = make_float2(0.f, 0.f), nm0 = nst, nm1 = nst;
        auto load_row = [&](int i) {
            const size_t row = (size_t)tile_at(i) * 128 + wt;
            nst = st1[net * st1_net + row0 + row];
            nm0 = mm[net * mm_net + row * 2];
            if constexpr (R > 16) nm1 = mm[net * mm_net + row * 2 + 1];
        };
        if (nt > 0) load_row(0);
        float mu1 = 0.f, rs1 = 0.f, m1 = 0.f, m2 = 0.f;
        for (int k = 0; k < steps; ++k) {
            const int i = k / NH, hf = k % NH;
            if (hf == 0) {
                mu1 = nst.x; rs1 = nst.y; m1 = nm0.x + nm1.x; m2 = nm0.y + nm1.y;
                if (i + 1 < nt) load_row(i + 1);
            }
            const f2 nmu = both(-mu1 * rs1), rs = both(rs1), nm1r = both(-m1 * rs1), nm2r = both(-m2 * rs1);
            const uint32_t ta = lane_tm + p * 128 + 32 * half;
            const float* bp = sb1 + (2 * hf + p) * 64 + 32 * half;
            mbar_wait(&bar_s[p], k & 1, status, kErrMma);
            tc_fence_after();
            uint32_t n1[16], dp[16];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                uint32_t u[16], v[16];
                tmem_ld16(ta + 16 * q, u);
                tmem_ld16(ta + 64 + 16 * q, v);
                tmem_ld_wait();
                if (q == 1) { tc_fence_before(); warp_arrive(&bar_rd[p]); }
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const f2 bb = *reinterpret_cast<const f2*>(bp + 16 * q + 2 * e);
                    f2 gr;
                    const f2 g = gelu2_grad(fma2(pack2(__uint_as_float(u[2 * e]), __uint_as_float(u[2 * e + 1])), both(1.f), bb), gr);
                    const f2 n = fma2(g, rs, nmu);
                    // rs1 (dn1 - m1 - n1 m2)
                    const f2 d = fma2(n, nm2r, fma2(pack2(__uint_as_float(v[2 * e]), __uint_as_float(v[2 * e + 1])), rs, nm1r));
                    const f2 o = mul2(d, gr);
                    n1[8 * q + e] = pack_bf16(lo2(n), hi2(n));
                    dp[8 * q + e] = pack_bf16(lo2(o), hi2(o));
                }
            }
            if (k > 0) mbar_wait(&bar_free, (k - 1) & 1, status, kErrMma);
            tc_fence_after();
            if (hf == 0 && i > 0) finish_tile(i - 1);
            tile_put32(smem + B::T + p * 16384, wt, half, n1);
            tile_put32(smem + B::T + 32768 + p * 16384, wt, half, dp);
            fence_proxy_async_smem();
            tc_fence_before();
            warp_arrive(&bar_t);
        }
        if (steps > 0) {
            mbar_wait(&bar_free, (steps - 1) & 1, status, kErrMma);
            tc_fence_after();
            finish_tile(nt - 1);
            const int hf = wg % 2, which = wg / 2;     // dW2, dW1; first and second 128 rows
            if (hf < NH) {
                float* dst = G + ((size_t)net * 4 + (which ? 0 : 1)) * kMat + (size_t)(hf * 128 + wt) * 64;
#pragma unroll
                for (int c = 0; c < 64; c += 16)
                    if (which || c < R) add_columns16(lane_tm + (which ? cW1 + hf * 64 : cW2 + hf * R) + c, dst + c);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 16) { cta_teardown_warp(); tmem_dealloc(tm, 512); }
}

// ---------------------------------------------------------------------------
// CUDA-core helpers
// ---------------------------------------------------------------------------
// Mean and 1 / sigma of every row (st0), and (n0 != nullptr: the backward) n0 = (x - mean) / sigma as hi + lo
// rows.  Eight lanes per row, eight columns each, two rows' loads in flight per lane: six shuffles serve four rows.
// (A whole warp per row took 67 us for 393 216 rows, ten shuffles each; now 26.)
constexpr int kLnRows = 64;                            // rows per CTA
__device__ __forceinline__ void unpack8(const uint4& q, float (&v)[8]) {
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) { v[2 * i] = __uint_as_float(w[i] << 16); v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u); }
}
__device__ __forceinline__ float sum8(float s) {       // over the eight lanes of a row
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    return s + __shfl_xor_sync(0xffffffffu, s, 4);
}
__global__ void __launch_bounds__(256)
ltc_ln0_kernel(Slice sl, const bf16* __restrict__ X, size_t row0, bf16* __restrict__ n0, bf16* __restrict__ n0_lo, float2* __restrict__ st0) {
    pdl_sync();
    const int ch = threadIdx.x % 8, r = threadIdx.x / 8;
    uint4 x[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) x[q] = *reinterpret_cast<const uint4*>(X + sl.row(row0 + blockIdx.x * kLnRows + r + 32 * q) + 8 * ch);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const size_t i = (size_t)blockIdx.x * kLnRows + r + 32 * q;
        float v[8], s = 0.f, t = 0.f;
        unpack8(x[q], v);
#pragma unroll
        for (int c = 0; c < 8; ++c) s += v[c];
        const float mu = sum8(s) * (1.f / 64.f);
#pragma unroll
        for (int c = 0; c < 8; ++c) { v[c] -= mu; t = fmaf(v[c], v[c], t); }
        const float rs = rsqrtf(sum8(t) * (1.f / 64.f) + kLnEps);
        if (ch == 0) st0[i] = make_float2(mu, rs);
        if (n0 != nullptr) {
            uint32_t h[4], l[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) split2(pack2(v[2 * c] * rs, v[2 * c + 1] * rs), h[c], l[c]);
            *reinterpret_cast<uint4*>(n0 + i * 64 + 8 * ch) = make_uint4(h[0], h[1], h[2], h[3]);
            *reinterpret_cast<uint4*>(n0_lo + i * 64 + 8 * ch) = make_uint4(l[0], l[1], l[2], l[3]);
        }
    }
}

// dX = back through the first normalisation of the two networks' gradients of n0 (+ add).  Lanes and rows as above.
__global__ void __launch_bounds__(256)
ltc_ln0_bwd_kernel(Slice sl, size_t row0, const float* __restrict__ dn0, size_t dn0_net, const bf16* __restrict__ n0,
                   const float2* __restrict__ st0, const bf16* __restrict__ add, bf16* __restrict__ dX) {
    pdl_sync();
    const int ch = threadIdx.x % 8, r = threadIdx.x / 8;
    float4 g[2][4];
    uint4 nq[2], aq[2];
    float rs[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const size_t i = (size_t)blockIdx.x * kLnRows + r + 32 * q, o = i * 64 + 8 * ch;
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            g[q][2 * t] = *reinterpret_cast<const float4*>(dn0 + t * dn0_net + o);
            g[q][2 * t + 1] = *reinterpret_cast<const float4*>(dn0 + t * dn0_net + o + 4);
        }
        nq[q] = *reinterpret_cast<const uint4*>(n0 + o);
        aq[q] = add != nullptr ? *reinterpret_cast<const uint4*>(add + row0 * 64 + o) : make_uint4(0, 0, 0, 0);
        rs[q] = st0[i].y;
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const float d[8] = {g[q][0].x + g[q][2].x, g[q][0].y + g[q][2].y, g[q][0].z + g[q][2].z, g[q][0].w + g[q][2].w,
                            g[q][1].x + g[q][3].x, g[q][1].y + g[q][3].y, g[q][1].z + g[q][3].z, g[q][1].w + g[q][3].w};
        float n[8], a[8], s1 = 0.f, s2 = 0.f;
        unpack8(nq[q], n);
        unpack8(aq[q], a);
#pragma unroll
        for (int c = 0; c < 8; ++c) { s1 += d[c]; s2 = fmaf(d[c], n[c], s2); }
        const float m1 = sum8(s1) * (1.f / 64.f), m2 = sum8(s2) * (1.f / 64.f);
        uint32_t pk[4];
#pragma unroll
        for (int c = 0; c < 4; ++c)
            pk[c] = pack_bf16(fmaf(rs[q], d[2 * c] - m1 - n[2 * c] * m2, a[2 * c]), fmaf(rs[q], d[2 * c + 1] - m1 - n[2 * c + 1] * m2, a[2 * c + 1]));
        *reinterpret_cast<uint4*>(dX + sl.row(row0 + (size_t)blockIdx.x * kLnRows + r + 32 * q) + 8 * ch) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
    }
}

// M = sqrt(r) tanh(f1 f2 / sqrt(r)), written as the [hi | lo] rows (64 bf16 columns, zero beyond 2r) the
// attention kernels read in their linear sketch mode; one thread = 8 entries of a row
__device__ __forceinline__ void load8f(const float* p, float (&v)[8]) {
    const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
template <int R>
__global__ void __launch_bounds__(256)
ltc_combine_kernel(const float* __restrict__ f1, const float* __restrict__ f2p, size_t rows, bf16* __restrict__ S) {
    pdl_sync();
    const size_t e = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (e >= rows * (R / 8)) return;
    const size_t row = e / (R / 8);
    const int c0 = (int)(e % (R / 8)) * 8;
    const float sr = sqrtf((float)R), isr = rsqrtf((float)R);
    float a[8], b[8];
    load8f(f1 + row * R + c0, a);
    load8f(f2p + row * R + c0, b);
    uint32_t h[4], l[4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
        split2(pack2(sr * tanhf(a[2 * j] * b[2 * j] * isr), sr * tanhf(a[2 * j + 1] * b[2 * j + 1] * isr)), h[j], l[j]);
    bf16* dst = S + row * 64 + c0;
    *reinterpret_cast<uint4*>(dst) = make_uint4(h[0], h[1], h[2], h[3]);
    *reinterpret_cast<uint4*>(dst + R) = make_uint4(l[0], l[1], l[2], l[3]);
#pragma unroll
    for (int z = 2 * R; z < 64; z += R) *reinterpret_cast<uint4*>(dst + z) = make_uint4(0, 0, 0, 0);
}

// df1 = dM (1 - t^2) f2, df2 = dM (1 - t^2) f1 as bf16 rows (r of 64 columns); dM = the first r columns of dS, the
// gradient of the [hi | lo] rows (M = hi + lo)
template <int R>
__global__ void __launch_bounds__(256)
ltc_combine_bwd_kernel(const float* __restrict__ f1, const float* __restrict__ f2p, const bf16* __restrict__ dS, size_t rows,
                       bf16* __restrict__ df1, bf16* __restrict__ df2) {
    pdl_sync();
    const size_t e = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (e >= rows * (R / 8)) return;
    const size_t row = e / (R / 8);
    const int c0 = (int)(e % (R / 8)) * 8;
    const float isr = rsqrtf((float)R);
    float a[8], b[8];
    load8f(f1 + row * R + c0, a);
    load8f(f2p + row * R + c0, b);
    const uint4 d4 = *reinterpret_cast<const uint4*>(dS + row * 64 + c0);
    const uint32_t dw[4] = {d4.x, d4.y, d4.z, d4.w};
    uint32_t o1[4], o2[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float t0 = tanhf(a[2 * j] * b[2 * j] * isr), t1 = tanhf(a[2 * j + 1] * b[2 * j + 1] * isr);
        const float u0 = __uint_as_float(dw[j] << 16) * (1.f - t0 * t0), u1 = __uint_as_float(dw[j] & 0xffff0000u) * (1.f - t1 * t1);
        o1[j] = pack_bf16(u0 * b[2 * j], u1 * b[2 * j + 1]);
        o2[j] = pack_bf16(u0 * a[2 * j], u1 * a[2 * j + 1]);
    }
    *reinterpret_cast<uint4*>(df1 + row * 64 + c0) = make_uint4(o1[0], o1[1], o1[2], o1[3]);
    *reinterpret_cast<uint4*>(df2 + row * 64 + c0) = make_uint4(o2[0], o2[1], o2[2], o2[3]);
}

// parameter gradients of one network from the four accumulators and the column sums
//   G1t = dp1^T n0, G2 = n1^T da2, G3t = dp3^T a2, G4 = a3^T df   (each [256][64])
// Entries that are sums over 8r or r products take a warp each, the others a thread.
__global__ void __launch_bounds__(256)
ltc_finish_kernel(int h, int r, const float* __restrict__ params, const float* __restrict__ G, const float* __restrict__ sums,
                  float* __restrict__ dparams) {
    pdl_sync();
    const NetLayout nl(h, r);
    const int net = blockIdx.y, m = nl.m;
    const float* P = params + (size_t)net * nl.count;
    float* dP = dparams + (size_t)net * nl.count;
    const float* G1t = G + (size_t)net * 4 * kMat;
    const float* G2 = G1t + kMat;
    const float* G3t = G2 + kMat;
    const float* G4 = G3t + kMat;
    const float* s_dp1 = sums + (size_t)net * kSums;
    const float* s_da2 = s_dp1 + 256;
    const float* s_dp3 = s_da2 + 64;
    const float* s_df = s_dp3 + 256;
    const int nsum = 2 * h + 2 * m, sum_blocks = (nsum + 7) / 8;
    if ((int)blockIdx.x < sum_blocks) {
        const int w = blockIdx.x * 8 + threadIdx.x / 32, lane = threadIdx.x % 32;
        if (w >= nsum) return;
        float g = 0.f;
        int e;
        if (w < h) {                                           // dg0[k] = sum_j W1[k][j] G1t[j][k]
            e = nl.g0 + w;
            for (int j = lane; j < m; j += 32) g = fmaf(P[nl.W1 + w * m + j], G1t[j * 64 + w], g);
        } else if (w < 2 * h) {                                // dc0[k] = sum_j W1[k][j] s_dp1[j]
            const int k = w - h;
            e = nl.c0 + k;
            for (int j = lane; j < m; j += 32) g = fmaf(P[nl.W1 + k * m + j], s_dp1[j], g);
        } else if (w < 2 * h + m) {                            // dg1[j] = sum_c W2[j][c] G2[j][c]
            const int j = w - 2 * h;
            e = nl.g1 + j;
            for (int c = lane; c < r; c += 32) g = fmaf(P[nl.W2 + j * r + c], G2[j * 64 + c], g);
        } else {                                               // dc1[j] = sum_c W2[j][c] s_da2[c]
            const int j = w - 2 * h - m;
            e = nl.c1 + j;
            for (int c = lane; c < r; c += 32) g = fmaf(P[nl.W2 + j * r + c], s_da2[c], g);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
        if (lane == 0) dP[e] += g;
        return;
    }
    const int e = (blockIdx.x - sum_blocks) * 256 + threadIdx.x;
    if (e >= nl.count || e < nl.W1 || (e >= nl.g1 && e < nl.W2)) return;
    float g = 0.f;
    if (e < nl.b1) {                                           // dW1[k][j] = g0[k] G1t[j][k] + c0[k] s_dp1[j]
        const int k = (e - nl.W1) / m, j = (e - nl.W1) % m;
        g = P[nl.g0 + k] * G1t[j * 64 + k] + P[nl.c0 + k] * s_dp1[j];
    } else if (e < nl.g1) {
        g = s_dp1[e - nl.b1];
    } else if (e < nl.b2) {                                    // dW2[j][c] = g1[j] G2[j][c] + c1[j] s_da2[c]
        const int j = (e - nl.W2) / r, c = (e - nl.W2) % r;
        g = P[nl.g1 + j] * G2[j * 64 + c] + P[nl.c1 + j] * s_da2[c];
    } else if (e < nl.W3) {
        g = s_da2[e - nl.b2];
    } else if (e < nl.b3) {                                    // dW3[c][j] = G3t[j][c]
        const int c = (e - nl.W3) / m, j = (e - nl.W3) % m;
        g = G3t[j * 64 + c];
    } else if (e < nl.W4) {
        g = s_dp3[e - nl.b3];
    } else if (e < nl.b4) {                                    // dW4[j][c] = G4[j][c]
        const int j = (e - nl.W4) / r, c = (e - nl.W4) % r;
        g = G4[j * 64 + c];
    } else {
        g = s_df[e - nl.b4];
    }
    dP[e] += g;
}

// ---------------------------------------------------------------------------
// host
// ---------------------------------------------------------------------------
struct LtcWs {
    size_t bank, vec, st0, f, a2, st1, G, sums, n0, n0_lo, df, da2, mm, dn0, total;
    size_t C, rows;             // rows per pass; rows of one tensor
    bool full;                  // a2, st1 and f of every row of both tensors are kept (else: f of one pass)
};

// Rows per pass.  PSK_LEARNED_CHUNK_ROWS in the environment overrides the default (a multiple of
// 128; read at every call, so that workspace queries and calls of one process agree as long as
// it is not changed between them): for tests of the chunk loop on small inputs, and for tuning.
size_t chunk_rows() {
    const char* e = std::getenv("PSK_LEARNED_CHUNK_ROWS");
    if (e != nullptr) {
        const long long v = std::atoll(e);
        if (v >= 128 && v % 128 == 0) return (size_t)v;
    }
    return kChunkRows;
}

// `full`: the backward's layout, which a forward call that keeps its states writes into
LtcWs ltc_ws(const Dims& d, bool full) {
    LtcWs w{};
    const size_t rows = (size_t)d.BH() * d.n, chunk = chunk_rows();
    const size_t C = w.C = rows < chunk ? rows : chunk;
    w.rows = rows;
    w.full = full;
    size_t off = 0;
    auto take = [&](size_t bytes) { const size_t o = off; off += align_up(bytes); return o; };
    w.bank = take(2 * kBankBytes);
    w.vec = take((size_t)2 * kVec * sizeof(float));
    w.st0 = take(C * sizeof(float2));
    w.f = take((full ? 4 * rows : 2 * C) * d.r * sizeof(float));         // [tensor][net][rows][r]
    if (full) {
        w.a2 = take(4 * rows * 64 * sizeof(bf16));                       // [tensor][net][rows][64]
        w.st1 = take(4 * rows * sizeof(float2));
        w.G = take((size_t)2 * 4 * kMat * sizeof(float));                // G and sums are zeroed together
        w.sums = take((size_t)2 * kSums * sizeof(float));
        w.n0 = take(C * 64 * sizeof(bf16));
        w.n0_lo = take(C * 64 * sizeof(bf16));
        w.df = take(2 * C * 64 * sizeof(bf16));
        w.da2 = take(2 * C * 64 * sizeof(bf16));
        w.mm = take(4 * C * sizeof(float2));
        w.dn0 = take(2 * C * 64 * sizeof(float));
    }
    w.total = off;
    return w;
}

// CTAs per network: both networks run side by side, one CTA per SM
inline int net_ctas(int tiles_of_work) { return tiles_of_work < 74 ? tiles_of_work : 74; }

cudaError_t row_stats(const Dims& d, const LtcWs& w, const void* X, size_t row0, int c, bool n0, char* ws, cudaStream_t s, int* launches) {
    prof_begin("ltc_ln0_kernel", s);
    launch_pdl(ltc_ln0_kernel, c / kLnRows, 256, 0, s, Slice{d.H, d.n, d.sb, d.sh, d.sn}, (const bf16*)X, row0,
               n0 ? (bf16*)(ws + w.n0) : nullptr, n0 ? (bf16*)(ws + w.n0_lo) : nullptr, (float2*)(ws + w.st0));
    prof_end(s);
    ++*launches;
    return cudaGetLastError();
}

// S = the [hi | lo] rows of the half sketch of X, tensor 0 or 1 (contiguous [rows][64] bf16)
template <int R>
cudaError_t sketch_t(const Dims& d, const LtcWs& w, int tensor, const void* X, void* S, char* ws, int* status, cudaStream_t s, int* launches) {
    const Slice sl{d.H, d.n, d.sb, d.sh, d.sn};
    PSK_TRY(set_smem(ltc_dense_norm_kernel<R>, kFwdSmem<R>));
    for (size_t row0 = 0; row0 < w.rows; row0 += w.C) {
        const int c = (int)(w.rows - row0 < w.C ? w.rows - row0 : w.C), tiles = c / 128;
        PSK_TRY(row_stats(d, w, X, row0, c, false, ws, s, launches));
        // strides between the networks' arrays, and where this pass's rows begin in them
        const size_t net_rows = w.full ? w.rows : w.C, first = w.full ? tensor * 2 * w.rows + row0 : 0;
        float* f = (float*)(ws + w.f) + first * R;
        prof_begin("ltc_dense_norm_kernel", s);
        launch_pdl(ltc_dense_norm_kernel<R>, dim3(net_ctas((tiles + 1) / 2), 2), 576, kFwdSmem<R>, s, sl, (const bf16*)X, row0, tiles,
                   (const float2*)(ws + w.st0), (const uint8_t*)(ws + w.bank), (const float*)(ws + w.vec),
                   w.full ? (bf16*)(ws + w.a2) + first * 64 : nullptr, net_rows * 64, w.full ? (float2*)(ws + w.st1) + first : nullptr, net_rows, f,
                   net_rows * R, status);
        prof_end(s);
        ++*launches;
        PSK_TRY(cudaGetLastError());
        prof_begin("ltc_combine_kernel", s);
        launch_pdl(ltc_combine_kernel<R>, (unsigned)(((size_t)c * (R / 8) + 255) / 256), 256, 0, s, (const float*)f, (const float*)(f + net_rows * R), (size_t)c,
                   (bf16*)S + row0 * 64);
        prof_end(s);
        ++*launches;
        PSK_TRY(cudaGetLastError());
    }
    return cudaSuccess;
}

template <int R>
cudaError_t sketch_bwd_t(const Dims& d, const LtcWs& w, int tensor, const void* X, const void* dS, const void* add, void* dX, char* ws,
                         int* status, cudaStream_t s, int* launches) {
    const Slice sl{d.H, d.n, d.sb, d.sh, d.sn};
    const size_t C = w.C;
    bf16* df = (bf16*)(ws + w.df);
    bf16* da2 = (bf16*)(ws + w.da2);
    const bf16* a2 = (const bf16*)(ws + w.a2) + (size_t)tensor * 2 * w.rows * 64;
    const float2* st1 = (const float2*)(ws + w.st1) + (size_t)tensor * 2 * w.rows;
    const uint8_t* bank = (const uint8_t*)(ws + w.bank);
    const float* vec = (const float*)(ws + w.vec);
    float* G = (float*)(ws + w.G);
    float* sums = (float*)(ws + w.sums);
    CUtensorMap mA[2], mDf[2], mDa[2], mN, mNlo;
    bool ok = tc_map_2d(&mN, ws + w.n0, 64, C, 128) && tc_map_2d(&mNlo, ws + w.n0_lo, 64, C, 128);
    for (int t = 0; t < 2; ++t)
        ok = ok && tc_map_2d(&mA[t], a2 + t * w.rows * 64, 64, w.rows, 128) && tc_map_2d(&mDf[t], df + t * C * 64, 64, C, 128) &&
             tc_map_2d(&mDa[t], da2 + t * C * 64, 64, C, 128);
    if (!ok) return cudaErrorInvalidValue;
    PSK_TRY(set_smem(ltc_wgrad_kernel<R>, Bwd34<R>::bytes));
    PSK_TRY(set_smem(ltc_dense_bwd_norm_kernel<R>, Bwd12<R>::bytes));
    for (size_t row0 = 0; row0 < w.rows; row0 += C) {
        const int c = (int)(w.rows - row0 < C ? w.rows - row0 : C), tiles = c / 128;
        const float* f = (const float*)(ws + w.f) + (tensor * 2 * w.rows + row0) * R;
        PSK_TRY(row_stats(d, w, X, row0, c, true, ws, s, launches));
        prof_begin("ltc_combine_bwd_kernel", s);
        launch_pdl(ltc_combine_bwd_kernel<R>, (unsigned)(((size_t)c * (R / 8) + 255) / 256), 256, 0, s, f, f + w.rows * R, (const bf16*)dS + row0 * 64,
                   (size_t)c, df, df + C * 64);
        prof_end(s);
        const dim3 grid(net_ctas(tiles), 2);
        prof_begin("ltc_wgrad_kernel", s);
        launch_pdl(ltc_wgrad_kernel<R>, grid, kBwdThreads, Bwd34<R>::bytes, s, mA[0], mA[1], mDf[0], mDf[1], row0, tiles, bank, vec, da2, C * 64,
                   (float2*)(ws + w.mm), 2 * C, G, sums, status);
        prof_end(s);
        prof_begin("ltc_dense_bwd_norm_kernel", s);
        launch_pdl(ltc_dense_bwd_norm_kernel<R>, grid, kBwdThreads, Bwd12<R>::bytes, s, mN, mNlo, mDa[0], mDa[1], row0, tiles, bank, vec, st1, w.rows,
                   (const float2*)(ws + w.mm), 2 * C, (float*)(ws + w.dn0), C * 64, G, sums, status);
        prof_end(s);
        prof_begin("ltc_ln0_bwd_kernel", s);
        launch_pdl(ltc_ln0_bwd_kernel, c / kLnRows, 256, 0, s, sl, row0, (const float*)(ws + w.dn0), C * 64,
                   (const bf16*)(ws + w.n0), (const float2*)(ws + w.st0), (const bf16*)add, (bf16*)dX);
        prof_end(s);
        *launches += 4;
        PSK_TRY(cudaGetLastError());
    }
    return cudaSuccess;
}

}  // namespace

bool learned_tc_supported(const Dims& d) { return d.bf16 && d.learned && d.h == 64 && (d.r == 16 || d.r == 32); }

size_t learned_tc_workspace_bytes(const Dims& d, bool full) { return ltc_ws(d, full).total; }

// operand bank of both networks; backward: also clears the gradient accumulators
cudaError_t learned_tc_prepare(const Dims& d, bool full, bool backward, char* ws, cudaStream_t s, int* launches) {
    const LtcWs w = ltc_ws(d, full);
    const int blocks = (64 * 8 * d.r + 3 * 8 * d.r * d.r) / 256 + (kVec + 7) / 8;
    prof_begin("ltc_bank_kernel", s);
    if (d.r == 16) launch_pdl(ltc_bank_kernel<16>, dim3(blocks, 2), 256, 0, s, d.lparams, (uint8_t*)(ws + w.bank), (float*)(ws + w.vec));
    else launch_pdl(ltc_bank_kernel<32>, dim3(blocks, 2), 256, 0, s, d.lparams, (uint8_t*)(ws + w.bank), (float*)(ws + w.vec));
    prof_end(s);
    ++*launches;
    PSK_TRY(cudaGetLastError());
    if (backward) PSK_TRY(cudaMemsetAsync(ws + w.G, 0, (w.sums - w.G) + (size_t)2 * kSums * sizeof(float), s));
    return cudaSuccess;
}

// S = the [hi | lo] rows of the half sketch of X, tensor 0 (Q) or 1 (K); `full`: what the backward reads again
// (a2, the row statistics, f) stays in the workspace
cudaError_t learned_tc_sketch(const Dims& d, bool full, int tensor, const void* X, void* S, char* ws, int* status, cudaStream_t s, int* launches) {
    const LtcWs w = ltc_ws(d, full);
    return d.r == 16 ? sketch_t<16>(d, w, tensor, X, S, ws, status, s, launches) : sketch_t<32>(d, w, tensor, X, S, ws, status, s, launches);
}

// dX = chain rule through both networks of the gradient dS of the [hi | lo] rows (+ add, a contiguous [rows][64] bf16 array
// or null: the part of the gradient that reached X directly); the weight-gradient
// accumulators in the workspace grow by this tensor's share (learned_tc_finish turns them into
// parameter gradients)
cudaError_t learned_tc_sketch_bwd(const Dims& d, int tensor, const void* X, const void* dS, const void* add, void* dX, char* ws,
                                  int* status, cudaStream_t s, int* launches) {
    const LtcWs w = ltc_ws(d, true);
    return d.r == 16 ? sketch_bwd_t<16>(d, w, tensor, X, dS, add, dX, ws, status, s, launches)
                     : sketch_bwd_t<32>(d, w, tensor, X, dS, add, dX, ws, status, s, launches);
}

// parameter gradients (added to d.dlparams) from everything learned_tc_sketch_bwd accumulated
cudaError_t learned_tc_finish(const Dims& d, char* ws, cudaStream_t s, int* launches) {
    const LtcWs w = ltc_ws(d, true);
    const NetLayout nl(d.h, d.r);
    prof_begin("ltc_finish_kernel", s);
    launch_pdl(ltc_finish_kernel, dim3((2 * nl.h + 2 * nl.m + 7) / 8 + (nl.count + 255) / 256, 2), 256, 0, s, d.h, d.r, d.lparams, (const float*)(ws + w.G),
               (const float*)(ws + w.sums), d.dlparams);
    prof_end(s);
    ++*launches;
    return cudaGetLastError();
}

}  // namespace psk
