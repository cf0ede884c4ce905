// CUDA-core path: causal Polysketch attention in fp32 arithmetic, the steps of
// Section 3.1 as separate kernels (half sketch -> per-block states H_l -> prefix scan
// Z_l -> output rows P_l + phi'(Q_l) Z_l -> division by D~).  Serves fp32 storage (the
// tensor cores' tf32 rounding cannot hold 1e-4 through a degree-4 polynomial) and
// cross-checks the tensor-core path on bf16 storage.
#include "cc_rows.cuh"

namespace psk {

// PSK_FLAG_KEEP_STATES means nothing here: every call forms all it reads, from its own arguments.
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
    // fp32 values are read where the caller has them, unless the forward writes over them
    if (d.bf16 || !backward) { w.Vt = off; off += align_up(rows * 64 * sizeof(float)); }
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
// group, two groups per CTA, one or two tensors (Q and K) per launch.  Dot form (cc_gemm.cuh): the rows
// lie in shared memory as they are in memory, only [G1 | G2] is transposed, once per CTA, which then
// walks several row tiles (the next one in flight).  A thread holds eight rows of the same columns of
// x G1 and of x G2 (two passes of 32 + 32 columns for r = 64), so their product is formed in registers.
// ---------------------------------------------------------------------------
template <int R> struct SkTile {
    static constexpr int kPasses = R == 64 ? 2 : 1, kCols = R / 8 / kPasses;       // columns per thread, matrix and pass
    static constexpr int Gt = 2 * R * cc::kLd;                                     // [2R][kLd]: rows of G1^T, then of G2^T
    static constexpr size_t bytes = (size_t)(Gt + 4 * cc::kUnit) * sizeof(float);  // two row buffers per group
};

template <typename T, int R>
__device__ __forceinline__ void load_g_transposed(float* sGt, const T* G1, const T* G2, int g, int tid, int nthr) {
#pragma unroll 4
    for (int e = tid; e < 2 * 64 * (R / 4); e += nthr) {
        const int k = e % 64, c = 4 * ((e / 64) % (R / 4)), m = e / (64 * (R / 4));
        const float4 v = cc::ld4((m ? G2 : G1) + (size_t)g * H64 * R + k * R + c);
        float* t = sGt + (m * R + c) * cc::kLd + k;
        t[0] = v.x; t[cc::kLd] = v.y; t[2 * cc::kLd] = v.z; t[3 * cc::kLd] = v.w;
    }
}
// 64 rows of a caller's tensor: asynchronous copies for fp32, converted for bf16
template <typename T>
__device__ __forceinline__ void load_x_rows(float* dst, const T* X, const Slice& sl, int bh, int i0, int lane) {
    if constexpr (sizeof(T) == 4) {
        for (int e = lane; e < 64 * 16; e += 64) cc::cp16(dst + (e / 16) * cc::kLd + 4 * (e % 16), X + sl.row(bh, i0 + e / 16) + 4 * (e % 16));
    } else {
        cc::load_raw<T, false>(dst, X, sl, bh, i0, lane, 64);
    }
    cc::cp_commit();
}
// a1, a2: rows ry + 8 i, columns base + cx + 8 j of X G1 and X G2
template <int R>
__device__ __forceinline__ void sketch_products(float (&a1)[8][SkTile<R>::kCols], float (&a2)[8][SkTile<R>::kCols],
                                                const float* X, const float* Gt, int base, int ry, int cx) {
    using namespace cc;
    constexpr int KC = SkTile<R>::kCols;
    f2 d[8][2 * KC];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 2 * KC; ++j) d[i][j] = 0ull;
    const float* x0 = X + ry * kLd;
    const float* g0 = Gt + (base + cx) * kLd;
#pragma unroll 1
    for (int k = 0; k < 64; k += 4) {
        F22 b[2 * KC];
#pragma unroll
        for (int j = 0; j < 2 * KC; ++j) b[j] = lds22(g0 + ((j / KC) * R + 8 * (j % KC)) * kLd + k);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const F22 a = lds22(x0 + 8 * i * kLd + k);
#pragma unroll
            for (int j = 0; j < 2 * KC; ++j) {
                d[i][j] = fma2(a.x, b[j].x, d[i][j]);
                d[i][j] = fma2(a.y, b[j].y, d[i][j]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < KC; ++j) { a1[i][j] = sum2(d[i][j]); a2[i][j] = sum2(d[i][KC + j]); }
}

template <typename T, int R>
__global__ void __launch_bounds__(128)
sketch_kernel(Slice sl, const T* __restrict__ X0, const T* __restrict__ X1, const T* __restrict__ G1, const T* __restrict__ G2,
              int g_heads, int n, float* __restrict__ M0, float* __restrict__ M1, float* __restrict__ Phi_out, int* status) {
    pdl_sync();
    if (status != nullptr && threadIdx.x < kStatusBytes / 4 && blockIdx.x + blockIdx.y + blockIdx.z == 0) status[threadIdx.x] = 0;
    extern __shared__ __align__(16) float smem[];
    using namespace cc;
    constexpr int KC = SkTile<R>::kCols;
    const int tid = threadIdx.x, grp = tid / 64, lane = tid % 64, ry = lane / 8, cx = lane % 8;
    float* sX = smem + SkTile<R>::Gt + grp * 2 * kUnit;
    const int bh = blockIdx.y, nt = n / 128;
    const T* X = blockIdx.z ? X1 : X0;
    float* Mbh = (blockIdx.z ? M1 : M0) + (size_t)bh * n * R;
    load_x_rows<T>(sX, X, sl, bh, blockIdx.x * 128 + grp * 64, lane);
    load_g_transposed<T, R>(smem, G1, G2, g_heads == 1 ? 0 : bh % sl.H, tid, 128);
    __syncthreads();
    const float rs = rsqrtf((float)R);
    int buf = 0;
    for (int tile = blockIdx.x; tile < nt; tile += gridDim.x, buf ^= 1) {
        if (tile + gridDim.x < nt) { load_x_rows<T>(sX + (buf ^ 1) * kUnit, X, sl, bh, (tile + gridDim.x) * 128 + grp * 64, lane); cp_wait<1>(); }
        else cp_wait<0>();
        group_sync(grp);
        float* M = Mbh + (size_t)(tile * 128 + grp * 64) * R;
#pragma unroll 1
        for (int base = 0; base < R; base += 8 * KC) {
            float a1[8][KC], a2[8][KC];
            sketch_products<R>(a1, a2, sX + buf * kUnit, smem, base, ry, cx);
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < KC; ++j) M[(ry + 8 * i) * R + base + cx + 8 * j] = a1[i][j] * a2[i][j] * rs;
        }
        group_sync(grp);
        if (Phi_out != nullptr) {           // phi'(x)[a*R+b] = m_a m_b (Section 1.2 ordering)
            float* phi = Phi_out + ((size_t)bh * n + tile * 128 + grp * 64) * R * R;      // (the group's rows of M are written)
            for (int e = lane; e < 64 * R * R / 4; e += 64) {
                const int rr = e / (R * R / 4), f = 4 * (e % (R * R / 4));
                const float ma = M[rr * R + f / R];
                const float4 mb = *reinterpret_cast<const float4*>(M + rr * R + f % R);
                *reinterpret_cast<float4*>(phi + (size_t)rr * R * R + f) = make_float4(ma * mb.x, ma * mb.y, ma * mb.z, ma * mb.w);
            }
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
    pdl_sync();
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
// A1 = X G1, A2 = X G2 recomputed.  Groups, tiles and tensors as in sketch_kernel; the second product
// contracts over the 2r sketch columns, [G1 | G2] as it lies in memory.  `add` (optional, [rows][64]):
// gradient that reached X without passing through the sketch, added before the result is rounded.
// ---------------------------------------------------------------------------
template <int R> struct SkBwdSmem {
    static constexpr int ldu = 2 * R + 4;
    static constexpr int Gt = 2 * R * cc::kLd, Gc = 64 * ldu;       // [G1 | G2]^T, and [64][G1 | G2]
    // per group: the rows, and U = [dM*A2 | dM*A1]
    static constexpr int X = cc::kUnit, U = 64 * ldu;
    static constexpr size_t bytes = (size_t)(Gt + Gc + 2 * (X + U)) * sizeof(float);
};

template <typename T, int R>
__global__ void __launch_bounds__(128)
sketch_bwd_kernel(Slice sl, const T* __restrict__ X0, const T* __restrict__ X1, const T* __restrict__ G1, const T* __restrict__ G2,
                  int g_heads, int n, const float* __restrict__ dM0, const float* __restrict__ dM1,
                  const float* __restrict__ add0, const float* __restrict__ add1, T* __restrict__ dX0, T* __restrict__ dX1) {
    pdl_sync();
    extern __shared__ __align__(16) float smem[];
    using namespace cc;
    using L = SkBwdSmem<R>;
    constexpr int KC = SkTile<R>::kCols, LDU = L::ldu;
    const int tid = threadIdx.x, grp = tid / 64, lane = tid % 64, ry = lane / 8, cx = lane % 8;
    float* sGc = smem + L::Gt;
    float* sX = sGc + L::Gc + grp * (L::X + L::U);
    float* sU = sX + L::X;
    const int bh = blockIdx.y, nt = n / 128;
    const T* X = blockIdx.z ? X1 : X0;
    const float* dM = (blockIdx.z ? dM1 : dM0) + (size_t)bh * n * R;
    const float* add = blockIdx.z ? add1 : add0;
    T* dX = blockIdx.z ? dX1 : dX0;
    const int g = (g_heads == 1) ? 0 : (bh % sl.H);
    load_x_rows<T>(sX, X, sl, bh, blockIdx.x * 128 + grp * 64, lane);
    load_g_transposed<T, R>(smem, G1, G2, g, tid, 128);
    for (int e = tid; e < 2 * 64 * (R / 4); e += 128) {
        const int k = (e / (R / 4)) % 64, c = 4 * (e % (R / 4)), m = e / (64 * (R / 4));
        *reinterpret_cast<float4*>(sGc + k * LDU + m * R + c) = ld4((m ? G2 : G1) + (size_t)g * H64 * R + k * R + c);
    }
    __syncthreads();
    const float rs = rsqrtf((float)R);
    for (int tile = blockIdx.x; tile < nt; tile += gridDim.x) {
        cp_wait<0>();
        group_sync(grp);
        const int i0 = tile * 128 + grp * 64;
#pragma unroll 1
        for (int base = 0; base < R; base += 8 * KC) {
            float a1[8][KC], a2[8][KC];
            sketch_products<R>(a1, a2, sX, smem, base, ry, cx);
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < KC; ++j) {
                    const int c = base + cx + 8 * j;
                    const float m = dM[(size_t)(i0 + ry + 8 * i) * R + c] * rs;
                    sU[(ry + 8 * i) * LDU + c] = m * a2[i][j];
                    sU[(ry + 8 * i) * LDU + R + c] = m * a1[i][j];
                }
        }
        group_sync(grp);
        // the rows have been read: the next tile's may arrive while the second product runs
        if (tile + gridDim.x < nt) load_x_rows<T>(sX, X, sl, bh, (tile + gridDim.x) * 128 + grp * 64, lane);
        f2 d[8][8];
        dot_full<LDU, LDU>(d, sU, sGc, R / 2, ry, cx);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int rr = i0 + ry + 8 * i;
            T* dst = dX + sl.row(bh, rr) + cx;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                float v = sum2(d[i][j]);
                if (add != nullptr) v += add[((size_t)bh * n + rr) * 64 + cx + 8 * j];
                stf(dst + 8 * j, v);
            }
        }
        group_sync(grp);
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

// CTAs along a head's 128-row tiles: about eight per SM in all, so that a CTA transposes the sketch matrices
// once for several tiles when there are many, and every tile has a CTA of its own when there are few.
inline unsigned sketch_grid(const Dims& d, int tensors) {
    const int nt = d.n / 128;
    const long want = 148L * 8 / ((long)d.BH() * tensors);
    const long per = want >= nt ? 1 : want < 1 ? nt : (nt + want - 1) / want;      // tiles per CTA, the same for all but the last
    return (unsigned)((nt + per - 1) / per);
}

// Half sketches of one tensor, or (X1 != nullptr) of two tensors of the same layout.
template <typename T, int R>
cudaError_t launch_sketch(const Dims& d, const T* X0, const T* X1, const T* G1, const T* G2, float* M0, float* M1, float* Phi,
                          int* status, cudaStream_t s, int* launches) {
    Slice sl{d.H, d.sb, d.sh, d.sn};
    if (!d.learned && d.p == 4) {
        PSK_TRY((allow_smem(sketch_kernel<T, R>, SkTile<R>::bytes)));
        const int nx = X1 != nullptr ? 2 : 1;
        prof_begin("sketch_kernel", s);
        launch_pdl(sketch_kernel<T, R>, dim3(sketch_grid(d, nx), d.BH(), nx), 128, SkTile<R>::bytes, s, sl, X0, X1, G1, G2, d.g_heads, d.n, M0, M1, Phi, status);
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
    launch_pdl(cc::cc_state_kernel<R>, dim3((NC + G - 1) / G, d.t - 1, d.BH()), 64 * G, cc::kStateSmem<R>, s, M, y, d.n, d.b, d.t, reverse ? 1 : 0, S);
    prof_end(s);
    ++*launches;
    PSK_TRY(cudaGetLastError());
    if (d.t == 2) return cudaSuccess;            // the only state there is needs no sum
    const size_t elems = (size_t)NC * cc::kChunkFloats / 4;
    prof_begin("scan_kernel", s);
    launch_pdl(cc::cc_scan_kernel, dim3((unsigned)((elems + 255) / 256), d.BH()), 256, 0, s, reinterpret_cast<float4*>(S), elems, d.t, reverse ? 1 : 0);
    prof_end(s);
    ++*launches;
    return cudaGetLastError();
}

// Groups of 64 threads per CTA of the row kernels: two, so that two CTAs share an SM and one's
// loads and final sums overlap the other's products, wherever their shared memory allows it (r <= 32,
// sketched weights) and there are CTAs enough for every SM; else as many as fit one CTA, which also
// spreads a few rows' work over the most warps.  (Training, four groups against two: r = 16, 128 CTAs 171 and 226 us, 320:
// 308 and 310, 640: 465 and 445, 1536: 998 and 911; r = 32, 128: 333 and 424, 320: 608 and 633, 640: 967 and 962,
// 1536: 2084 and 2018.)
inline bool two_per_sm(const Dims& d) { return (long)d.BH() * (d.n / 64) >= 2 * 148; }

template <typename T, int R, bool LOCAL, int NG>
cudaError_t launch_rows_ng(const Dims& d, const float* Mown, const float* Moth, const cc::YRows& y, const float* S, const T* Xown,
                           const T* Xoth, bool dv, T* Out, float* denom, cudaStream_t s, int* launches) {
    using L = cc::RowsSmem<R, LOCAL, NG>;
    PSK_TRY((allow_smem(cc::cc_rows_kernel<T, R, LOCAL, NG>, L::bytes)));
    prof_begin(dv ? "bwd_v_kernel" : "fwd_out_kernel", s);
    launch_pdl(cc::cc_rows_kernel<T, R, LOCAL, NG>, dim3(d.b / 64, d.t, d.BH()), 64 * NG, L::bytes, s, 
        Slice{d.H, d.sb, d.sh, d.sn}, d.n, d.b, d.t, Mown, Moth, y, S, Xown, Xoth, dv ? 1 : 0, Out, denom);
    prof_end(s);
    ++*launches;
    return cudaGetLastError();
}

template <typename T, int R>
cudaError_t launch_rows(const Dims& d, const float* Mown, const float* Moth, const cc::YRows& y, const float* S, const T* Xown,
                        const T* Xoth, bool dv, T* Out, float* denom, cudaStream_t s, int* launches) {
    if (d.local) return launch_rows_ng<T, R, true, 4>(d, Mown, Moth, y, S, Xown, Xoth, dv, Out, denom, s, launches);
    if constexpr (R <= 32)
        if (two_per_sm(d)) return launch_rows_ng<T, R, false, 2>(d, Mown, Moth, y, S, Xown, Xoth, dv, Out, denom, s, launches);
    return launch_rows_ng<T, R, false, 4>(d, Mown, Moth, y, S, Xown, Xoth, dv, Out, denom, s, launches);
}

template <typename T, int R, bool LOCAL, int NG>
cudaError_t launch_dphi_ng(const Dims& d, const float* Mown, const float* Moth, const cc::YRows& yown, const cc::YRows& yoth, const float* S,
                           const T* Xown, const T* Xoth, bool kside, float* dM, float* dXl, cudaStream_t s, int* launches) {
    using L = cc::DphiSmem<R, LOCAL, NG>;
    PSK_TRY((allow_smem(cc::cc_dphi_kernel<T, R, LOCAL, NG>, L::bytes)));
    prof_begin(kside ? "bwd_k_kernel" : "bwd_q_kernel", s);
    launch_pdl(cc::cc_dphi_kernel<T, R, LOCAL, NG>, dim3(d.b / 64, d.t, d.BH()), 64 * NG, L::bytes, s, 
        Slice{d.H, d.sb, d.sh, d.sn}, d.n, d.b, d.t, Mown, Moth, yown, yoth, S, Xown, Xoth, kside ? 1 : 0, dM, dXl);
    prof_end(s);
    ++*launches;
    return cudaGetLastError();
}

template <typename T, int R>
cudaError_t launch_dphi(const Dims& d, const float* Mown, const float* Moth, const cc::YRows& yown, const cc::YRows& yoth, const float* S,
                        const T* Xown, const T* Xoth, bool kside, float* dM, float* dXl, cudaStream_t s, int* launches) {
    constexpr int NG = R == 64 ? 3 : 4;
    if (d.local) return launch_dphi_ng<T, R, true, NG>(d, Mown, Moth, yown, yoth, S, Xown, Xoth, kside, dM, dXl, s, launches);
    if constexpr (R <= 32)
        if (two_per_sm(d)) return launch_dphi_ng<T, R, false, 2>(d, Mown, Moth, yown, yoth, S, Xown, Xoth, kside, dM, dXl, s, launches);
    return launch_dphi_ng<T, R, false, NG>(d, Mown, Moth, yown, yoth, S, Xown, Xoth, kside, dM, dXl, s, launches);
}

// [V | 1] rows: the caller's fp32 values as they are, or an fp32 copy in scratch: for bf16 storage, and where the
// output O (null: none that is written while V is read) may lie over V, which other rows' CTAs still read.
template <typename T>
cudaError_t value_rows(const Dims& d, const T* V, const T* O, float* Vt, cc::YRows* y, cudaStream_t s, int* launches) {
    Slice sl{d.H, d.sb, d.sh, d.sn};
    if constexpr (sizeof(T) == 4) {
        const uintptr_t v = reinterpret_cast<uintptr_t>(V), o = reinterpret_cast<uintptr_t>(O);
        const uintptr_t span = ((d.B - 1) * d.sb + (d.H - 1) * d.sh + (d.n - 1) * d.sn + 64) * sizeof(T);
        if (O == nullptr || v + span <= o || o + span <= v) {
            *y = cc::YRows{V, sl, 1};
            return cudaSuccess;
        }
    }
    const int rows = d.BH() * d.n;
    prof_begin("rows_prep_kernel", s);
    launch_pdl(rows_prep_kernel<T>, (rows + 15) / 16, 256, 0, s, sl, d.n, rows, 0, V, nullptr, nullptr, nullptr, Vt);
    prof_end(s);
    ++*launches;
    *y = cc::YRows{Vt, Slice{d.H, (int64_t)d.H * d.n * 64, (int64_t)d.n * 64, 64}, 1};
    return cudaGetLastError();
}

// Half sketches, value rows and prefix states: what the forward needs, and the backward again.
template <typename T, int R>
cudaError_t prefix_states(const Dims& d, const T* Q, const T* K, const T* V, const T* G1, const T* G2, const T* O, char* ws,
                          const CcWorkspace& w, cc::YRows* y, cudaStream_t s, int* launches) {
    float* Mq = (float*)(ws + w.Mq); float* Mk = (float*)(ws + w.Mk);
    PSK_TRY((launch_sketch<T, R>(d, Q, K, G1, G2, Mq, Mk, nullptr, d.clear_status ? (int*)(ws + w.status) : nullptr, s, launches)));
    PSK_TRY(value_rows<T>(d, V, O, (float*)(ws + w.Vt), y, s, launches));
    return launch_states<R>(d, Mk, *y, (float*)(ws + w.Zst), false, s, launches);
}

template <typename T, int R>
cudaError_t fwd_impl(const Dims& d, const T* Q, const T* K, const T* V, const T* G1, const T* G2,
                     T* O, float* denom, char* ws, cudaStream_t s, int* launches) {
    const CcWorkspace w = cc_workspace(d, false);
    cc::YRows y;
    PSK_TRY((prefix_states<T, R>(d, Q, K, V, G1, G2, O, ws, w, &y, s, launches)));
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
        const int nx = X1 != nullptr ? 2 : 1;
        launch_pdl(sketch_bwd_kernel<T, R>, dim3(sketch_grid(d, nx), d.BH(), nx), 128, L::bytes, s, 
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
    PSK_TRY((prefix_states<T, R>(d, Q, K, V, G1, G2, nullptr, ws, w, &yv, s, launches)));
    prof_begin("rows_prep_kernel", s);
    launch_pdl(rows_prep_kernel<T>, (rows + 15) / 16, 256, 0, s, Slice{d.H, d.sb, d.sh, d.sn}, d.n, rows, 1, nullptr, O, denom, dO, E);
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
#define C_ (launch_sketch<T, R>(d, (const T*)X, nullptr, (const T*)G1, (const T*)G2, M_out, nullptr, Phi_out, nullptr, s, launches))
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
