// CUDA-core path: causal Polysketch attention in fp32 arithmetic, the steps of
// Section 3.1 as separate kernels (half sketch -> per-block states H_l -> prefix scan
// Z_l -> output rows P_l + phi'(Q_l) Z_l -> division by D~).  Serves fp32 storage (the
// tensor cores' tf32 rounding cannot hold 1e-4 through a degree-4 polynomial) and
// cross-checks the tensor-core path on bf16 storage.
#include "cc_rows.cuh"

namespace psk {

// The forward's arrays come first and lie the same in both layouts: with PSK_FLAG_KEEP_STATES the
// backward finds the half sketches and the prefix states where the forward left them.
CcWorkspace cc_workspace(const Dims& d, bool backward) {
    CcWorkspace w{};
    const size_t rows = (size_t)d.BH() * d.n;
    const size_t chunks = (size_t)(d.r / 8) * (d.r / 8 + 1) / 2;
    const size_t st = (size_t)d.BH() * d.t * chunks * cc::kChunkFloats * sizeof(float);
        size_t off = 0;
    w.status = off; off += kStatusBytes;
    w.Mq = off;  off += align_up(rows * d.r * sizeof(float));
    w.Mk = off;  off += align_up(rows * d.r * sizeof(float));
    w.Zst = off; off += align_up(st);
    if (d.bf16) { w.Vt = off; off += align_up(rows * 64 * sizeof(float)); }      // fp32 values are read where the caller has them
    if (backward) {
        w.E = off;   off += align_up(rows * cc::kLd * sizeof(float));
        w.Rst = off; off += align_up(st);
        w.dMq = off; off += align_up(rows * d.r * sizeof(float));
        w.dMk = off; off += align_up(rows * d.r * sizeof(float));
        if (d.local) {     // gradients that reach Q and K directly, through the exact same-block weights
            w.dXq = off; off += align_up(rows * 64 * sizeof(float));
            w.dXk = off; off += align_up(rows * 64 * sizeof(float));
        }
    }
    // The size reported is what full r^2 x 65 states per block take, as it has always been; the
    // distinct features need less of it.
    const size_t full = align_up((size_t)d.BH() * d.t * d.r * d.r * 65 * sizeof(float)), row65 = align_up(rows * 65 * sizeof(float));
    const size_t m = align_up(rows * d.r * sizeof(float));
    size_t reported = kStatusBytes + 2 * m + row65 + full;
    if (backward) reported += row65 + full + 2 * m + (d.local ? 2 * align_up(rows * 64 * sizeof(float)) : 0);
    w.total = off > reported ? off : reported;
    return w;
}

namespace {

constexpr int H64 = 64;     // head dimension (only value supported)
using cc::Slice;

// ---------------------------------------------------------------------------
// Half sketch m(x) = (x G1)*(x G2)/sqrt(r)  (Algorithm 1, degree-2 level): 64 rows per 64-thread
// group, two groups per CTA, one or two tensors (Q and K) per launch.  A thread holds eight rows of
// the same few columns of x G1 and of x G2 (16 columns in two passes for r = 64), so their product is
// formed in registers.
// ---------------------------------------------------------------------------
template <int R> struct SkTile {
    static constexpr int kPasses = R == 64 ? 2 : 1, kCols = R / 8 / kPasses, NP = kCols / 2;
};

// a1, a2: rows 8 ry + i, columns base + kCols cx + j of X G1 and X G2 (Xt [64][kLd], G [64][R])
template <int R>
__device__ __forceinline__ void sketch_products(float (&a1)[8][SkTile<R>::kCols], float (&a2)[8][SkTile<R>::kCols],
                                                const float* Xt, const float* G1, const float* G2, int base, int ry, int cx) {
    using namespace cc;
    constexpr int NP = SkTile<R>::NP, KC = SkTile<R>::kCols;
    f2 s[2][4][NP], x[2][4][NP];
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int q = 0; q < NP; ++q) s[m][p][q] = x[m][p][q] = 0ull;
#pragma unroll 4
    for (int k = 0; k < 64; ++k) {
        f2 a[4];
        load_rows8(a, Xt + k * kLd + 8 * ry);
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            const float* g = (m ? G2 : G1) + k * R + base + KC * cx;
            f2 c[NP];
            if constexpr (NP == 1) c[0] = *reinterpret_cast<const f2*>(g);
            else { const F22 u = lds22(g); c[0] = u.x; c[1] = u.y; }
#pragma unroll
            for (int q = 0; q < NP; ++q) {
                const f2 sw = swap2(c[q]);
#pragma unroll
                for (int p = 0; p < 4; ++p) { s[m][p][q] = fma2(a[p], c[q], s[m][p][q]); x[m][p][q] = fma2(a[p], sw, x[m][p][q]); }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < KC; ++j) {
            const f2 v1 = ((i ^ j) & 1) ? x[0][i / 2][j / 2] : s[0][i / 2][j / 2];
            const f2 v2 = ((i ^ j) & 1) ? x[1][i / 2][j / 2] : s[1][i / 2][j / 2];
            a1[i][j] = (i & 1) ? hi2(v1) : lo2(v1);
            a2[i][j] = (i & 1) ? hi2(v2) : lo2(v2);
        }
}

template <int R> constexpr size_t kSketchSmem = (2 * H64 * R + 2 * cc::kUnit) * sizeof(float);

template <typename T, int R>
__global__ void __launch_bounds__(128)
sketch_kernel(Slice sl, const T* __restrict__ X0, const T* __restrict__ X1, const T* __restrict__ G1, const T* __restrict__ G2,
              int g_heads, int n, float* __restrict__ M0, float* __restrict__ M1, float* __restrict__ Phi_out) {
    extern __shared__ __align__(16) float smem[];
    using namespace cc;
    constexpr int KC = SkTile<R>::kCols;
    float* sG1 = smem;                  // [64][R]
    float* sG2 = sG1 + H64 * R;         // [64][R]
    const int tid = threadIdx.x, grp = tid / 64, lane = tid % 64, ry = lane / 8, cx = lane % 8;
    float* sXt = sG2 + H64 * R + grp * kUnit;
    const int bh = blockIdx.y, i0 = blockIdx.x * 128 + grp * 64;
    const T* X = blockIdx.z ? X1 : X0;
    float* M = (blockIdx.z ? M1 : M0) + ((size_t)bh * n + i0) * R;
    const int g = (g_heads == 1) ? 0 : (bh % sl.H);
    for (int e = tid; e < H64 * R / 4; e += 128) {
        *reinterpret_cast<float4*>(sG1 + 4 * e) = ld4(G1 + (size_t)g * H64 * R + 4 * e);
        *reinterpret_cast<float4*>(sG2 + 4 * e) = ld4(G2 + (size_t)g * H64 * R + 4 * e);
    }
    load_raw<T, true>(sXt, X, sl, bh, i0, lane, 64);
    __syncthreads();
    const float rs = rsqrtf((float)R);
#pragma unroll 1
    for (int base = 0; base < R; base += 8 * KC) {
        float a1[8][KC], a2[8][KC];
        sketch_products<R>(a1, a2, sXt, sG1, sG2, base, ry, cx);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            float* dst = M + (size_t)(8 * ry + i) * R + base + KC * cx;
            if constexpr (KC == 2) *reinterpret_cast<float2*>(dst) = make_float2(a1[i][0] * a2[i][0] * rs, a1[i][1] * a2[i][1] * rs);
            else *reinterpret_cast<float4*>(dst) = make_float4(a1[i][0] * a2[i][0] * rs, a1[i][1] * a2[i][1] * rs,
                                                               a1[i][2] * a2[i][2] * rs, a1[i][3] * a2[i][3] * rs);
        }
    }
    if (Phi_out != nullptr) {           // phi'(x)[a*R+b] = m_a m_b (Section 1.2 ordering)
        __syncthreads();                // (this CTA's rows of M, written above, are visible to all of it)
        float* phi = Phi_out + ((size_t)bh * n + i0) * R * R;
        for (int e = lane; e < 64 * R * R / 4; e += 64) {
            const int rr = e / (R * R / 4), f = 4 * (e % (R * R / 4));
            const float ma = M[rr * R + f / R];
            const float4 mb = *reinterpret_cast<const float4*>(M + rr * R + f % R);
            *reinterpret_cast<float4*>(phi + (size_t)rr * R * R + f) = make_float4(ma * mb.x, ma * mb.y, ma * mb.z, ma * mb.w);
        }
    }
}

// ---------------------------------------------------------------------------
// Degree p = 2 (Algorithm 1 with p/2 = 1): the "half sketch" is the row itself, M = X, and
// phi'(x) = x (x) x has h^2 entries: exact degree-2 polynomial attention, no Gaussians.
// Forward copy M = X (optionally Phi = X (x) X); backward dX = dM (+ add).  One warp per row.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256)
identity_sketch_kernel(Slice sl, int n, int total_rows, const T* __restrict__ X, float* __restrict__ M,
                       float* __restrict__ Phi) {
    const int row = blockIdx.x * 8 + threadIdx.x / 32, lane = threadIdx.x % 32;
    if (row >= total_rows) return;
    const int64_t base = sl.row(row / n, row % n);
    const float x0 = ldf(X + base + lane), x1 = ldf(X + base + lane + 32);
    M[(size_t)row * 64 + lane] = x0;
    M[(size_t)row * 64 + lane + 32] = x1;
    if (Phi != nullptr) {
        for (int a = 0; a < 64; ++a) {
            const float xa = __shfl_sync(0xffffffffu, a < 32 ? x0 : x1, a % 32);
            Phi[((size_t)row * 64 + a) * 64 + lane] = xa * x0;
            Phi[((size_t)row * 64 + a) * 64 + lane + 32] = xa * x1;
        }
    }
}

template <typename T>
__global__ void __launch_bounds__(256)
identity_sketch_bwd_kernel(Slice sl, int n, int total_rows, const float* __restrict__ dM,
                           const float* __restrict__ add, T* __restrict__ dX) {
    const int row = blockIdx.x * 8 + threadIdx.x / 32, lane = threadIdx.x % 32;
    if (row >= total_rows) return;
    const int64_t base = sl.row(row / n, row % n);
#pragma unroll
    for (int c = lane; c < 64; c += 32) {
        float v = dM[(size_t)row * 64 + c];
        if (add != nullptr) v += add[(size_t)row * 64 + c];
        stf(dX + base + c, v);
    }
}

// ---------------------------------------------------------------------------
// Degree p = 8: one more level of Algorithm 1's recursion.  Two independent degree-2 sketches
//   M1 = (X Ga1)*(X Ga2)/sqrt(r),  M2 = (X Gb1)*(X Gb2)/sqrt(r)
// are combined through r x r Gaussians,  M = (M1 Gc1)*(M2 Gc2)/sqrt(r); phi' = M (x) M as before.
// G1 holds [Ga1; Gb1; Gc1] and G2 holds [Ga2; Gb2; Gc2], each (2h + r) x r row-major per head.
// 32 rows per CTA; the Gaussians are read from global memory (they stay in cache).
// ---------------------------------------------------------------------------
template <int R> struct Sk8 {
    static constexpr int kRows = 32, kLd = R + 1;
    static constexpr int kGRows = 2 * H64 + R;             // rows of one packed Gaussian set
    static constexpr int X = 0;                            // [32][65]
    static constexpr int A1 = X + kRows * 65, A2 = A1 + kRows * kLd, B1 = A2 + kRows * kLd, B2 = B1 + kRows * kLd;
    static constexpr int M1 = B2 + kRows * kLd, M2 = M1 + kRows * kLd, C1 = M2 + kRows * kLd, C2 = C1 + kRows * kLd;
    static constexpr int total = C2 + kRows * kLd;
    static constexpr size_t bytes = (size_t)total * sizeof(float);
};

// shared by the forward and the backward: X tile -> A1, A2, B1, B2, M1, M2, C1 = M1 Gc1, C2 = M2 Gc2
template <typename T, int R>
__device__ __forceinline__ void sketch8_forward_tile(float* smem, Slice sl, const T* __restrict__ X,
                                                     const T* __restrict__ g1, const T* __restrict__ g2,
                                                     int bh, int i0, int tid) {
    using L = Sk8<R>;
    for (int e = tid; e < L::kRows * H64; e += 256) {
        const int rr = e / H64, c = e % H64;
        smem[L::X + rr * 65 + c] = ldf(X + sl.row(bh, i0 + rr) + c);
    }
    __syncthreads();
    const float rs = rsqrtf((float)R);
    for (int e = tid; e < L::kRows * R; e += 256) {
        const int rr = e / R, c = e % R;
        float a1 = 0.f, a2 = 0.f, b1 = 0.f, b2 = 0.f;
        for (int t = 0; t < H64; ++t) {
            const float x = smem[L::X + rr * 65 + t];
            a1 = fmaf(x, ldf(g1 + t * R + c), a1);
            a2 = fmaf(x, ldf(g2 + t * R + c), a2);
            b1 = fmaf(x, ldf(g1 + (H64 + t) * R + c), b1);
            b2 = fmaf(x, ldf(g2 + (H64 + t) * R + c), b2);
        }
        const int o = rr * L::kLd + c;
        smem[L::A1 + o] = a1; smem[L::A2 + o] = a2; smem[L::B1 + o] = b1; smem[L::B2 + o] = b2;
        smem[L::M1 + o] = a1 * a2 * rs;
        smem[L::M2 + o] = b1 * b2 * rs;
    }
    __syncthreads();
    for (int e = tid; e < L::kRows * R; e += 256) {
        const int rr = e / R, c = e % R;
        float c1 = 0.f, c2 = 0.f;
        for (int k = 0; k < R; ++k) {
            c1 = fmaf(smem[L::M1 + rr * L::kLd + k], ldf(g1 + (2 * H64 + k) * R + c), c1);
            c2 = fmaf(smem[L::M2 + rr * L::kLd + k], ldf(g2 + (2 * H64 + k) * R + c), c2);
        }
        smem[L::C1 + rr * L::kLd + c] = c1;
        smem[L::C2 + rr * L::kLd + c] = c2;
    }
    __syncthreads();
}

template <typename T, int R>
__global__ void __launch_bounds__(256)
sketch8_kernel(Slice sl, const T* __restrict__ X, const T* __restrict__ G1, const T* __restrict__ G2,
               int g_heads, int n, float* __restrict__ M_out, float* __restrict__ Phi_out) {
    extern __shared__ float smem[];
    using L = Sk8<R>;
    const int bh = blockIdx.y, i0 = blockIdx.x * L::kRows, tid = threadIdx.x;
    const int g = (g_heads == 1) ? 0 : (bh % sl.H);
    const T* g1 = G1 + (size_t)g * L::kGRows * R;
    const T* g2 = G2 + (size_t)g * L::kGRows * R;
    sketch8_forward_tile<T, R>(smem, sl, X, g1, g2, bh, i0, tid);
    const float rs = rsqrtf((float)R);
    for (int e = tid; e < L::kRows * R; e += 256) {
        const int rr = e / R, c = e % R;
        const float m = smem[L::C1 + rr * L::kLd + c] * smem[L::C2 + rr * L::kLd + c] * rs;
        smem[L::M1 + rr * L::kLd + c] = m;                 // (M1 is dead: keep M for Phi)
        M_out[((size_t)bh * n + i0 + rr) * R + c] = m;
    }
    if (Phi_out != nullptr) {
        __syncthreads();
        for (int e = tid; e < L::kRows * R * R; e += 256) {
            const int rr = e / (R * R), f = e % (R * R);
            Phi_out[((size_t)bh * n + i0 + rr) * R * R + f] =
                smem[L::M1 + rr * L::kLd + f / R] * smem[L::M1 + rr * L::kLd + f % R];
        }
    }
}

// Chain rule through the degree-8 half sketch (forward values recomputed):
//   dC1 = dM*C2/sqrt(r), dC2 = dM*C1/sqrt(r);  dM1 = dC1 Gc1^T, dM2 = dC2 Gc2^T;
//   dA1 = dM1*A2/sqrt(r), dA2 = dM1*A1/sqrt(r), dB1 = dM2*B2/sqrt(r), dB2 = dM2*B1/sqrt(r);
//   dX = dA1 Ga1^T + dA2 Ga2^T + dB1 Gb1^T + dB2 Gb2^T.
template <typename T, int R>
__global__ void __launch_bounds__(256)
sketch8_bwd_kernel(Slice sl, const T* __restrict__ X, const T* __restrict__ G1, const T* __restrict__ G2,
                   int g_heads, int n, const float* __restrict__ dM, T* __restrict__ dX) {
    extern __shared__ float smem[];
    using L = Sk8<R>;
    const int bh = blockIdx.y, i0 = blockIdx.x * L::kRows, tid = threadIdx.x;
    const int g = (g_heads == 1) ? 0 : (bh % sl.H);
    const T* g1 = G1 + (size_t)g * L::kGRows * R;
    const T* g2 = G2 + (size_t)g * L::kGRows * R;
    sketch8_forward_tile<T, R>(smem, sl, X, g1, g2, bh, i0, tid);
    const float rs = rsqrtf((float)R);
    // dC1, dC2 over C1, C2 (each entry is read and written by one thread)
    for (int e = tid; e < L::kRows * R; e += 256) {
        const int rr = e / R, c = e % R, o = rr * L::kLd + c;
        const float gm = dM[((size_t)bh * n + i0 + rr) * R + c] * rs;
        const float c1 = smem[L::C1 + o], c2 = smem[L::C2 + o];
        smem[L::C1 + o] = gm * c2;
        smem[L::C2 + o] = gm * c1;
    }
    __syncthreads();
    // dM1, dM2 over M1, M2 (M1, M2 themselves are no longer needed)
    for (int e = tid; e < L::kRows * R; e += 256) {
        const int rr = e / R, k = e % R;
        float d1 = 0.f, d2 = 0.f;
        for (int c = 0; c < R; ++c) {
            d1 = fmaf(smem[L::C1 + rr * L::kLd + c], ldf(g1 + (2 * H64 + k) * R + c), d1);
            d2 = fmaf(smem[L::C2 + rr * L::kLd + c], ldf(g2 + (2 * H64 + k) * R + c), d2);
        }
        smem[L::M1 + rr * L::kLd + k] = d1;
        smem[L::M2 + rr * L::kLd + k] = d2;
    }
    __syncthreads();
    // dA1, dA2, dB1, dB2 over A1, A2, B1, B2
    for (int e = tid; e < L::kRows * R; e += 256) {
        const int rr = e / R, c = e % R, o = rr * L::kLd + c;
        const float d1 = smem[L::M1 + o] * rs, d2 = smem[L::M2 + o] * rs;
        const float a1 = smem[L::A1 + o], a2 = smem[L::A2 + o], b1 = smem[L::B1 + o], b2 = smem[L::B2 + o];
        smem[L::A1 + o] = d1 * a2; smem[L::A2 + o] = d1 * a1;
        smem[L::B1 + o] = d2 * b2; smem[L::B2 + o] = d2 * b1;
    }
    __syncthreads();
    for (int e = tid; e < L::kRows * H64; e += 256) {
        const int rr = e / H64, t = e % H64;
        float dx = 0.f;
        for (int c = 0; c < R; ++c) {
            const int o = rr * L::kLd + c;
            dx = fmaf(smem[L::A1 + o], ldf(g1 + t * R + c), dx);
            dx = fmaf(smem[L::A2 + o], ldf(g2 + t * R + c), dx);
            dx = fmaf(smem[L::B1 + o], ldf(g1 + (H64 + t) * R + c), dx);
            dx = fmaf(smem[L::B2 + o], ldf(g2 + (H64 + t) * R + c), dx);
        }
        stf(dX + sl.row(bh, i0 + rr) + t, dx);
    }
}

// ---------------------------------------------------------------------------
// Row preparation: mode 0 writes V in fp32 (bf16 storage; rows of 64); mode 1 writes
// E = [dO/d | -(dO.O)/d] (rows of kLd).  16 lanes per row.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256)
rows_prep_kernel(Slice sl, int n, int total_rows, int mode, const T* __restrict__ V,
                 const T* __restrict__ O, const float* __restrict__ denom,
                 const T* __restrict__ dO, float* __restrict__ out) {
    const int row = blockIdx.x * 16 + threadIdx.x / 16, lane = threadIdx.x % 16;
    if (row >= total_rows) return;      // (total_rows is a multiple of 128: whole warps)
    const int64_t base = sl.row(row / n, row % n) + 4 * lane;
    if (mode == 0) {
        *reinterpret_cast<float4*>(out + (size_t)row * 64 + 4 * lane) = cc::ld4(V + base);
        return;
    }
    float* o = out + (size_t)row * cc::kLd;
    float4 v = cc::ld4(dO + base);
    const float4 u = cc::ld4(O + base);
    float dot = (v.x * u.x + v.y * u.y) + (v.z * u.z + v.w * u.w);
#pragma unroll
    for (int s = 8; s > 0; s >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, s);
    const float inv = 1.f / denom[row];
    v.x *= inv; v.y *= inv; v.z *= inv; v.w *= inv;
    *reinterpret_cast<float4*>(o + 4 * lane) = v;
    if (lane == 0) *reinterpret_cast<float4*>(o + 64) = make_float4(-dot * inv, 0.f, 0.f, 0.f);
}

// ---------------------------------------------------------------------------
// Chain rule through the half sketch: dX = ((dM*A2) G1^T + (dM*A1) G2^T)/sqrt(r),
// A1 = X G1, A2 = X G2 recomputed.  Groups, rows and tensors as in sketch_kernel.  `add` (optional,
// [rows][64]): gradient that reached X without passing through the sketch, added before the
// result is rounded.
// ---------------------------------------------------------------------------
template <int R> struct SkBwdSmem {
    static constexpr int G = 2 * H64 * R, Gt = 2 * R * cc::kLd;
    static constexpr int U = 2 * R * cc::kLd;          // U1, U2 transposed
    static constexpr size_t bytes = (size_t)(G + Gt + 2 * (cc::kUnit + U)) * sizeof(float);
};

template <typename T, int R>
__global__ void __launch_bounds__(128)
sketch_bwd_kernel(Slice sl, const T* __restrict__ X0, const T* __restrict__ X1, const T* __restrict__ G1, const T* __restrict__ G2,
                  int g_heads, int n, const float* __restrict__ dM0, const float* __restrict__ dM1,
                  const float* __restrict__ add0, const float* __restrict__ add1, T* __restrict__ dX0, T* __restrict__ dX1) {
    extern __shared__ __align__(16) float smem[];
    using namespace cc;
    using L = SkBwdSmem<R>;
    constexpr int KC = SkTile<R>::kCols;
    float* sG1 = smem;                      // [64][R]
    float* sG2 = sG1 + H64 * R;             // [64][R]
    float* sGt = sG2 + H64 * R;             // [2R][kLd]: rows of G1^T, then of G2^T
    const int tid = threadIdx.x, grp = tid / 64, lane = tid % 64, ry = lane / 8, cx = lane % 8;
    float* sXt = sGt + L::Gt + grp * (kUnit + L::U);
    float* sU = sXt + kUnit;                // [2R][kLd]: rows of (dM*A2)^T, then of (dM*A1)^T
    const int bh = blockIdx.y, i0 = blockIdx.x * 128 + grp * 64;
    const T* X = blockIdx.z ? X1 : X0;
    const float* dM = (blockIdx.z ? dM1 : dM0) + ((size_t)bh * n + i0) * R;
    const float* add = blockIdx.z ? add1 : add0;
    T* dX = blockIdx.z ? dX1 : dX0;
    const int g = (g_heads == 1) ? 0 : (bh % sl.H);
    for (int e = tid; e < H64 * R / 4; e += 128) {
        const int k = e / (R / 4), c = 4 * (e % (R / 4));
        const float4 u = ld4(G1 + (size_t)g * H64 * R + 4 * e), v = ld4(G2 + (size_t)g * H64 * R + 4 * e);
        *reinterpret_cast<float4*>(sG1 + 4 * e) = u;
        *reinterpret_cast<float4*>(sG2 + 4 * e) = v;
        float* t1 = sGt + c * kLd + k;
        float* t2 = sGt + (R + c) * kLd + k;
        t1[0] = u.x; t1[kLd] = u.y; t1[2 * kLd] = u.z; t1[3 * kLd] = u.w;
        t2[0] = v.x; t2[kLd] = v.y; t2[2 * kLd] = v.z; t2[3 * kLd] = v.w;
    }
    load_raw<T, true>(sXt, X, sl, bh, i0, lane, 64);
    __syncthreads();
    const float rs = rsqrtf((float)R);
#pragma unroll 1
    for (int base = 0; base < R; base += 8 * KC) {
        float a1[8][KC], a2[8][KC];
        sketch_products<R>(a1, a2, sXt, sG1, sG2, base, ry, cx);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            float gm[KC];
            const float* src = dM + (size_t)(8 * ry + i) * R + base + KC * cx;
            if constexpr (KC == 2) { const float2 v = *reinterpret_cast<const float2*>(src); gm[0] = v.x; gm[1] = v.y; }
            else *reinterpret_cast<float4*>(gm) = *reinterpret_cast<const float4*>(src);
#pragma unroll
            for (int j = 0; j < KC; ++j) {
                const float m = gm[j] * rs;
                a2[i][j] *= m;
                a1[i][j] *= m;
            }
        }
#pragma unroll
        for (int j = 0; j < KC; ++j) {
            float* u1 = sU + (base + KC * cx + j) * kLd + 8 * ry;
            float* u2 = u1 + R * kLd;
            *reinterpret_cast<float4*>(u1) = make_float4(a2[0][j], a2[1][j], a2[2][j], a2[3][j]);
            *reinterpret_cast<float4*>(u1 + 4) = make_float4(a2[4][j], a2[5][j], a2[6][j], a2[7][j]);
            *reinterpret_cast<float4*>(u2) = make_float4(a1[0][j], a1[1][j], a1[2][j], a1[3][j]);
            *reinterpret_cast<float4*>(u2 + 4) = make_float4(a1[4][j], a1[5][j], a1[6][j], a1[7][j]);
        }
    }
    group_sync(grp);
    Acc acc;
    acc.zero();
    outer_product(acc, sU, sGt, 2 * R, kLd, ry, cx);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int rr = i0 + 8 * ry + i;
        T* dst = dX + sl.row(bh, rr);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = 32 * h + 4 * cx;
            float4 v = make_float4(acc.at(i, 4 * h), acc.at(i, 4 * h + 1), acc.at(i, 4 * h + 2), acc.at(i, 4 * h + 3));
            if (add != nullptr) {
                const float4 a = *reinterpret_cast<const float4*>(add + ((size_t)bh * n + rr) * 64 + c);
                v.x += a.x; v.y += a.y; v.z += a.z; v.w += a.w;
            }
            st4(dst + c, v);
        }
    }
}

// ---------------------------------------------------------------------------
// host-side launch helpers
// ---------------------------------------------------------------------------
#define PSK_TRY(x) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) return e_; } while (0)

template <typename K>
cudaError_t allow_smem(K kernel, size_t bytes) {
    if (bytes <= 48 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// Half sketches of one tensor, or (X1 != nullptr) of two tensors of the same layout.
template <typename T, int R>
cudaError_t launch_sketch(const Dims& d, const T* X0, const T* X1, const T* G1, const T* G2, float* M0, float* M1, float* Phi,
                          cudaStream_t s, int* launches) {
    Slice sl{d.H, d.sb, d.sh, d.sn};
    if (!d.learned && d.p == 4) {
        PSK_TRY((allow_smem(sketch_kernel<T, R>, kSketchSmem<R>)));
        prof_begin("sketch_kernel", s);
        sketch_kernel<T, R><<<dim3(d.n / 128, d.BH(), X1 != nullptr ? 2 : 1), 128, kSketchSmem<R>, s>>>(
            sl, X0, X1, G1, G2, d.g_heads, d.n, M0, M1, Phi);
        prof_end(s);
        ++*launches;
        return cudaGetLastError();
    }
    for (int i = 0; i < (X1 != nullptr ? 2 : 1); ++i) {
        const T* X = i ? X1 : X0;
        float* M = i ? M1 : M0;
        if (d.learned) {          // Algorithm 2: two dense networks
            PSK_TRY(learned_sketch(d, X, M, Phi, s, launches));
            continue;
        }
        if (d.p == 2) {           // M = X (R = 64 = h)
            const int rows = d.BH() * d.n;
            prof_begin("identity_sketch_kernel", s);
            identity_sketch_kernel<T><<<(rows + 7) / 8, 256, 0, s>>>(sl, d.n, rows, X, M, Phi);
        } else {                  // p = 8, one more recursion level: packed Gaussians [Ga; Gb; Gc]
            PSK_TRY((allow_smem(sketch8_kernel<T, R>, Sk8<R>::bytes)));
            prof_begin("sketch8_kernel", s);
            sketch8_kernel<T, R><<<dim3(d.n / Sk8<R>::kRows, d.BH()), 256, Sk8<R>::bytes, s>>>(sl, X, G1, G2, d.g_heads, d.n, M, Phi);
        }
        prof_end(s);
        ++*launches;
        PSK_TRY(cudaGetLastError());
    }
    return cudaSuccess;
}

// Prefix (suffix) states of every block: block states, then the scan over them.
template <int R>
cudaError_t launch_states(const Dims& d, const float* M, const cc::YRows& y, float* S, bool reverse,
                          cudaStream_t s, int* launches) {
    if (d.t == 1) return cudaSuccess;
    constexpr int G = cc::kStateGroups<R>, NC = cc::kChunks<R>;
    PSK_TRY((allow_smem(cc::cc_state_kernel<R>, cc::kStateSmem<R>)));
    prof_begin("state_kernel", s);
    cc::cc_state_kernel<R><<<dim3((NC + G - 1) / G, d.t - 1, d.BH()), 64 * G, cc::kStateSmem<R>, s>>>(M, y, d.n, d.b, d.t, reverse ? 1 : 0, S);
    prof_end(s);
    ++*launches;
    PSK_TRY(cudaGetLastError());
    if (d.t == 2) return cudaSuccess;            // the only state there is needs no sum
    const size_t elems = (size_t)NC * cc::kChunkFloats / 4;
    prof_begin("scan_kernel", s);
    cc::cc_scan_kernel<<<dim3((unsigned)((elems + 255) / 256), d.BH()), 256, 0, s>>>(reinterpret_cast<float4*>(S), elems, d.t, reverse ? 1 : 0);
    prof_end(s);
    ++*launches;
    return cudaGetLastError();
}

template <typename T, int R>
cudaError_t launch_rows(const Dims& d, const float* Mown, const float* Moth, const cc::YRows& y, const float* S, const T* Xown,
                        const T* Xoth, bool dv, T* Out, float* denom, cudaStream_t s, int* launches) {
    const dim3 grid(d.b / 64, d.t, d.BH());
    Slice sl{d.H, d.sb, d.sh, d.sn};
    prof_begin(dv ? "bwd_v_kernel" : "fwd_out_kernel", s);
    if (d.local) {
        using L = cc::RowsSmem<R, true>;
        PSK_TRY((allow_smem(cc::cc_rows_kernel<T, R, true>, L::bytes)));
        cc::cc_rows_kernel<T, R, true><<<grid, 64 * L::NG, L::bytes, s>>>(sl, d.n, d.b, d.t, Mown, Moth, y, S, Xown, Xoth, dv ? 1 : 0, Out, denom);
    } else {
        using L = cc::RowsSmem<R, false>;
        PSK_TRY((allow_smem(cc::cc_rows_kernel<T, R, false>, L::bytes)));
        cc::cc_rows_kernel<T, R, false><<<grid, 64 * L::NG, L::bytes, s>>>(sl, d.n, d.b, d.t, Mown, Moth, y, S, Xown, Xoth, dv ? 1 : 0, Out, denom);
    }
    prof_end(s);
    ++*launches;
    return cudaGetLastError();
}

template <typename T, int R>
cudaError_t launch_dphi(const Dims& d, const float* Mown, const float* Moth, const cc::YRows& yown, const cc::YRows& yoth, const float* S,
                        const T* Xown, const T* Xoth, bool kside, float* dM, float* dXl, cudaStream_t s, int* launches) {
    const dim3 grid(d.b / 64, d.t, d.BH());
    Slice sl{d.H, d.sb, d.sh, d.sn};
    prof_begin(kside ? "bwd_k_kernel" : "bwd_q_kernel", s);
    if (d.local) {
        using L = cc::DphiSmem<R, true>;
        PSK_TRY((allow_smem(cc::cc_dphi_kernel<T, R, true>, L::bytes)));
        cc::cc_dphi_kernel<T, R, true><<<grid, 64 * L::NG, L::bytes, s>>>(sl, d.n, d.b, d.t, Mown, Moth, yown, yoth, S, Xown, Xoth, kside ? 1 : 0, dM, dXl);
    } else {
        using L = cc::DphiSmem<R, false>;
        PSK_TRY((allow_smem(cc::cc_dphi_kernel<T, R, false>, L::bytes)));
        cc::cc_dphi_kernel<T, R, false><<<grid, 64 * L::NG, L::bytes, s>>>(sl, d.n, d.b, d.t, Mown, Moth, yown, yoth, S, Xown, Xoth, kside ? 1 : 0, dM, dXl);
    }
    prof_end(s);
    ++*launches;
    return cudaGetLastError();
}

// [V | 1] rows: the caller's fp32 values as they are, or (bf16 storage) an fp32 copy in scratch.
template <typename T>
cudaError_t value_rows(const Dims& d, const T* V, float* Vt, cc::YRows* y, cudaStream_t s, int* launches) {
    Slice sl{d.H, d.sb, d.sh, d.sn};
    if constexpr (sizeof(T) == 4) {
        *y = cc::YRows{V, sl, 1};
        return cudaSuccess;
    } else {
        const int rows = d.BH() * d.n;
        prof_begin("rows_prep_kernel", s);
        rows_prep_kernel<T><<<(rows + 15) / 16, 256, 0, s>>>(sl, d.n, rows, 0, V, nullptr, nullptr, nullptr, Vt);
        prof_end(s);
        ++*launches;
        *y = cc::YRows{Vt, Slice{d.H, (int64_t)d.H * d.n * 64, (int64_t)d.n * 64, 64}, 1};
        return cudaGetLastError();
    }
}

// Half sketches, value rows and prefix states: what the forward needs, and the backward again
// unless the forward left them in this workspace.
template <typename T, int R>
cudaError_t prefix_states(const Dims& d, const T* Q, const T* K, const T* V, const T* G1, const T* G2, char* ws,
                          const CcWorkspace& w, bool kept, cc::YRows* y, cudaStream_t s, int* launches) {
    float* Mq = (float*)(ws + w.Mq); float* Mk = (float*)(ws + w.Mk);
    if (kept) {
        *y = sizeof(T) == 4 ? cc::YRows{(const float*)V, Slice{d.H, d.sb, d.sh, d.sn}, 1}
                            : cc::YRows{(const float*)(ws + w.Vt), Slice{d.H, (int64_t)d.H * d.n * 64, (int64_t)d.n * 64, 64}, 1};
        return cudaSuccess;
    }
    PSK_TRY((launch_sketch<T, R>(d, Q, K, G1, G2, Mq, Mk, nullptr, s, launches)));
    PSK_TRY(value_rows<T>(d, V, (float*)(ws + w.Vt), y, s, launches));
    return launch_states<R>(d, Mk, *y, (float*)(ws + w.Zst), false, s, launches);
}

template <typename T, int R>
cudaError_t fwd_impl(const Dims& d, const T* Q, const T* K, const T* V, const T* G1, const T* G2,
                     T* O, float* denom, char* ws, cudaStream_t s, int* launches) {
    const CcWorkspace w = cc_workspace(d, false);
    cc::YRows y;
    PSK_TRY((prefix_states<T, R>(d, Q, K, V, G1, G2, ws, w, false, &y, s, launches)));
    return launch_rows<T, R>(d, (float*)(ws + w.Mq), (float*)(ws + w.Mk), y, (float*)(ws + w.Zst), Q, K, false, O, denom, s, launches);
}

// Chain rule through the half sketches of Q and K: dX from dM (+ `add`, the part of the gradient
// that reached X directly through exact same-block weights).  X1 may be null.
template <typename T, int R>
cudaError_t launch_sketch_bwd(const Dims& d, const T* X0, const T* X1, const T* G1, const T* G2, const float* dM0, const float* dM1,
                              const float* add0, const float* add1, T* dX0, T* dX1, cudaStream_t s, int* launches) {
    Slice sl{d.H, d.sb, d.sh, d.sn};
    const int rows = d.BH() * d.n;
    if (!d.learned && d.p == 4) {
        using L = SkBwdSmem<R>;
        PSK_TRY((allow_smem(sketch_bwd_kernel<T, R>, L::bytes)));
        prof_begin("sketch_bwd_kernel", s);
        sketch_bwd_kernel<T, R><<<dim3(d.n / 128, d.BH(), X1 != nullptr ? 2 : 1), 128, L::bytes, s>>>(
            sl, X0, X1, G1, G2, d.g_heads, d.n, dM0, dM1, add0, add1, dX0, dX1);
        prof_end(s);
        ++*launches;
        return cudaGetLastError();
    }
    for (int i = 0; i < (X1 != nullptr ? 2 : 1); ++i) {
        const T* X = i ? X1 : X0;
        const float* dM = i ? dM1 : dM0;
        const float* add = i ? add1 : add0;
        T* dX = i ? dX1 : dX0;
        if (d.learned) {          // two networks; gradients add up
            PSK_TRY(learned_sketch_bwd(d, X, dM, add, dX, s, launches));
            continue;
        }
        if (d.p == 2) {           // dX = dM (+ add)
            prof_begin("identity_sketch_bwd_kernel", s);
            identity_sketch_bwd_kernel<T><<<(rows + 7) / 8, 256, 0, s>>>(sl, d.n, rows, dM, add, dX);
        } else {
            PSK_TRY((allow_smem(sketch8_bwd_kernel<T, R>, Sk8<R>::bytes)));
            prof_begin("sketch8_bwd_kernel", s);
            sketch8_bwd_kernel<T, R><<<dim3(d.n / Sk8<R>::kRows, d.BH()), 256, Sk8<R>::bytes, s>>>(sl, X, G1, G2, d.g_heads, d.n, dM, dX);
        }
        prof_end(s);
        ++*launches;
        PSK_TRY(cudaGetLastError());
    }
    return cudaSuccess;
}

template <typename T, int R>
cudaError_t bwd_impl(const Dims& d, const T* Q, const T* K, const T* V, const T* G1, const T* G2,
                     const T* O, const float* denom, const T* dO, T* dQ, T* dK, T* dV,
                     char* ws, cudaStream_t s, int* launches) {
    const CcWorkspace w = cc_workspace(d, true);
    float* Mq = (float*)(ws + w.Mq); float* Mk = (float*)(ws + w.Mk);
    float* Z = (float*)(ws + w.Zst);
    float* E = (float*)(ws + w.E); float* Rs = (float*)(ws + w.Rst);
    float* dMq = (float*)(ws + w.dMq); float* dMk = (float*)(ws + w.dMk);
    float* dXq = d.local ? (float*)(ws + w.dXq) : nullptr;
    float* dXk = d.local ? (float*)(ws + w.dXk) : nullptr;
    const int rows = d.BH() * d.n;
    cc::YRows yv;
    PSK_TRY((prefix_states<T, R>(d, Q, K, V, G1, G2, ws, w, d.keep_states, &yv, s, launches)));
    prof_begin("rows_prep_kernel", s);
    rows_prep_kernel<T><<<(rows + 15) / 16, 256, 0, s>>>(Slice{d.H, d.sb, d.sh, d.sn}, d.n, rows, 1, nullptr, O, denom, dO, E);
    prof_end(s);
    ++*launches;
    PSK_TRY(cudaGetLastError());
    const cc::YRows ye{E, Slice{d.H, (int64_t)d.H * d.n * cc::kLd, (int64_t)d.n * cc::kLd, cc::kLd}, 0};
    PSK_TRY((launch_dphi<T, R>(d, Mq, Mk, ye, yv, Z, Q, K, false, dMq, dXq, s, launches)));
    PSK_TRY((launch_states<R>(d, Mq, ye, Rs, true, s, launches)));
    PSK_TRY((launch_dphi<T, R>(d, Mk, Mq, yv, ye, Rs, K, Q, true, dMk, dXk, s, launches)));
    PSK_TRY((launch_rows<T, R>(d, Mk, Mq, ye, Rs, K, Q, true, dV, nullptr, s, launches)));
    return launch_sketch_bwd<T, R>(d, Q, K, G1, G2, dMq, dMk, dXq, dXk, dQ, dK, s, launches);
}

#define PSK_DISPATCH(CALL_F32, CALL_BF16)                                   \
    if (d.bf16) {                                                           \
        typedef __nv_bfloat16 T;                                            \
        switch (d.r) { case 16: { constexpr int R = 16; return CALL_BF16; } \
                       case 32: { constexpr int R = 32; return CALL_BF16; } \
                       case 64: { constexpr int R = 64; return CALL_BF16; } } \
    } else {                                                                \
        typedef float T;                                                    \
        switch (d.r) { case 16: { constexpr int R = 16; return CALL_F32; }  \
                       case 32: { constexpr int R = 32; return CALL_F32; }  \
                       case 64: { constexpr int R = 64; return CALL_F32; } } \
    }                                                                       \
    return cudaErrorInvalidValue;

}  // namespace

cudaError_t cc_sketch(const Dims& d, const void* X, const void* G1, const void* G2,
                      float* M_out, float* Phi_out, cudaStream_t s, int* launches) {
#define C_ (launch_sketch<T, R>(d, (const T*)X, nullptr, (const T*)G1, (const T*)G2, M_out, nullptr, Phi_out, s, launches))
    PSK_DISPATCH(C_, C_)
#undef C_
}

cudaError_t cc_fwd(const Dims& d, const void* Q, const void* K, const void* V,
                   const void* G1, const void* G2, void* O, float* denom,
                   char* ws, cudaStream_t s, int* launches) {
#define C_ (fwd_impl<T, R>(d, (const T*)Q, (const T*)K, (const T*)V, (const T*)G1, (const T*)G2, \
                           (T*)O, denom, ws, s, launches))
    PSK_DISPATCH(C_, C_)
#undef C_
}

cudaError_t cc_bwd(const Dims& d, const void* Q, const void* K, const void* V,
                   const void* G1, const void* G2, const void* O, const float* denom,
                   const void* dO, void* dQ, void* dK, void* dV,
                   char* ws, cudaStream_t s, int* launches) {
#define C_ (bwd_impl<T, R>(d, (const T*)Q, (const T*)K, (const T*)V, (const T*)G1, (const T*)G2, \
                           (const T*)O, denom, (const T*)dO, (T*)dQ, (T*)dK, (T*)dV, ws, s, launches))
    PSK_DISPATCH(C_, C_)
#undef C_
}

}  // namespace psk
