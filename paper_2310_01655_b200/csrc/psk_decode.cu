// Recurrent form of causal Polysketch attention: one new token per (batch, head) per call.
// lt(phi'(Q) phi'(K)^T) [V | 1] row by row is a running state (the "linear transformer" view
// the paper's Section 3 starts from; Section 3.1's Z_l is this state at block boundaries):
//   S_t = S_{t-1} + phi'(k_t) [v_t | 1]^T          (r^2 x 65, fp32, kept by the caller)
//   N_t = phi'(q_t)^T S_t,   d_t = 1 + N_t[64],   o_t = N_t[:64] / d_t
// so inference costs O(r^2 h) per token whatever the context length.  The step is bound by
// reading and writing the state once, or, with few heads, by latency.
#include "psk_internal.cuh"

namespace psk {
namespace {

constexpr int kCols = 65;            // [v | 1]
constexpr int kSub = 4;              // thread groups of 65 in a CTA
constexpr int kThreads = kCols * kSub;

// A head's state is dealt to a cluster of CL CTAs.
template <int R, int CL> struct Dec {
    static constexpr int kVec = R * R / CL / 4 / kSub;               // float4 of the state per thread
    static constexpr int kBatch = kVec < 8 ? kVec : 8;               // ... per batch of asynchronous copies
    static constexpr int kSlots = kVec < 16 ? kVec : 16;             // ... in flight: at most two batches
    static constexpr size_t kSmem = (size_t)kSlots * kThreads * 16;
    static constexpr int kPerSm = kSlots == 16 ? 2 : 4;              // CTAs per SM that registers are held to
};

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// State rows f = a r + b (the Kronecker order of Section 1.2) of 65 floats.  Four rows are 65 float4 and start
// on 16 bytes, so 65 threads move four rows with 16-byte accesses; a thread's four floats lie in
// the same one or two of the four rows, and in the same columns, in every group of four rows.
// The state comes through shared memory by asynchronous copies, so that what is in flight costs no
// registers.  The updated state waits there too until the cluster has been signalled: that signal is a
// release, and with the state's stores before it every CTA stayed until they had reached memory
// (r = 32, 384 heads: 52 us).
template <typename T, int R, int CL>
__global__ void __launch_bounds__(kThreads, Dec<R, CL>::kPerSm)
decode_step_kernel(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v,
                   const T* __restrict__ G1, const T* __restrict__ G2, int g_heads, int H,
                   float* __restrict__ state, T* __restrict__ o, float* __restrict__ denom) {
    constexpr int kRows = R * R / CL, NV = Dec<R, CL>::kVec, NB = Dec<R, CL>::kBatch, NS = Dec<R, CL>::kSlots;
    static_assert(NV % NB == 0 && NS % NB == 0 && (NV == NS || NS == 2 * NB), "whole batches");
    pdl_sync();
    extern __shared__ float4 sbuf[];                 // [NS][kThreads]: every thread copies and reads its own entries
    __shared__ float sx[3][64], sa[2][4][2][R], sm[2][R + 4];
    __shared__ double part[kSub][4 * kCols];
    __shared__ double red[CL][kCols];               // used in the cluster's first CTA
    const int cr = (int)(blockIdx.x % CL);
    const int bh = blockIdx.x / CL, tid = threadIdx.x;
    const int g = g_heads == 1 ? 0 : bh % H;
    const int t65 = tid % kCols, sub = tid / kCols;
    float4* S = reinterpret_cast<float4*>(state + ((size_t)bh * R * R + (size_t)cr * kRows) * kCols) + t65;       // this CTA's rows
    if (CL > 1) cluster_arrive();                   // (waited for before the first access to another CTA's memory)
    // The state is requested before anything else: it is in flight while the half sketches are computed.
    const unsigned buf = (unsigned)__cvta_generic_to_shared(sbuf + tid);
    auto request = [&](int j0) {
#pragma unroll
        for (int j = j0; j < j0 + NB; ++j)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(buf + (j % NS) * (kThreads * 16)), "l"(S + (sub + j * kSub) * kCols) : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // half sketches m(q_t), m(k_t) (Algorithm 1, degree-2 level): a thread sums 16 of the 64 terms of one
    // column of one matrix, for q and k; all its loads are independent
    constexpr int kPasses = (8 * R + 255) / 256;
    float gv[16];
    auto load_g = [&](int e) {
        const int c = e % R, mat = (e / R) % 2, part4 = e / (2 * R);
        const T* G = (mat ? G2 : G1) + (size_t)g * 64 * R + (part4 * 16) * R + c;
#pragma unroll
        for (int t = 0; t < 16; ++t) gv[t] = ldf(G + t * R);
    };
    const float x0 = tid < 192 ? ldf((tid < 64 ? q : (tid < 128 ? k : v)) + (size_t)bh * 64 + tid % 64) : 0.f;
    if (tid < 8 * R && tid < 256) load_g(tid);
#pragma unroll
    for (int j0 = 0; j0 < NS; j0 += NB) request(j0);
    if (tid < 192) sx[tid / 64][tid % 64] = x0;
    __syncthreads();
    // this thread's four floats of a group of four rows
    const int ro = 4 * t65 / kCols;
    float vc[4];
    unsigned up = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int flat = 4 * t65 + i, col = flat % kCols;
        if (flat / kCols != ro) up |= 1u << i;
        vc[i] = col < 64 ? sx[2][col] : 1.f;
    }
#pragma unroll
    for (int ps = 0; ps < kPasses; ++ps) {
        const int e = tid + ps * 256, c = e % R, mat = (e / R) % 2, part4 = e / (2 * R);
        if (e < 8 * R && tid < 256) {
            if (ps > 0) load_g(e);
            float aq = 0.f, ak = 0.f;
#pragma unroll
            for (int t = 0; t < 16; ++t) { aq = fmaf(sx[0][part4 * 16 + t], gv[t], aq); ak = fmaf(sx[1][part4 * 16 + t], gv[t], ak); }
            sa[mat][part4][0][c] = aq;
            sa[mat][part4][1][c] = ak;
        }
    }
    __syncthreads();
    for (int e = tid; e < 2 * R; e += kThreads) {
        const int w = e / R, c = e % R;
        const float a1 = (sa[0][0][w][c] + sa[0][1][w][c]) + (sa[0][2][w][c] + sa[0][3][w][c]);
        const float a2 = (sa[1][0][w][c] + sa[1][1][w][c]) + (sa[1][2][w][c] + sa[1][3][w][c]);
        sm[w][c] = a1 * a2 * rsqrtf((float)R);
    }
    __syncthreads();
    // (the sum over the r^2 features cancels heavily -- it equals a square of a short sum -- so the
    // products, rounded once to fp32, are added up in double)
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
    for (int j0 = 0; j0 < NV; j0 += NB) {
        if (NV == NS || j0 + NB >= NV) asm volatile("cp.async.wait_group 0;" ::: "memory");
        else asm volatile("cp.async.wait_group 1;" ::: "memory");
#pragma unroll
        for (int j = 0; j < NB; ++j) {
            const int grp = sub + (j0 + j) * kSub, f0 = cr * kRows + 4 * grp, a = f0 / R, b0 = f0 % R + ro;
            const float4 cur = sbuf[((j0 + j) % NS) * kThreads + tid];
            const float q0 = sm[0][a] * sm[0][b0], q1 = sm[0][a] * sm[0][b0 + 1];
            const float k0 = sm[1][a] * sm[1][b0], k1 = sm[1][a] * sm[1][b0 + 1];
            float x[4] = {cur.x, cur.y, cur.z, cur.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const bool u = (up >> i) & 1u;
                x[i] = fmaf(u ? k1 : k0, vc[i], x[i]);
                acc[i] += (double)((u ? q1 : q0) * x[i]);
            }
            const float4 nw = make_float4(x[0], x[1], x[2], x[3]);
            if (NV > NS && j0 + NS < NV) S[grp * kCols] = nw;          // (its slot is needed again)
            else sbuf[((j0 + j) % NS) * kThreads + tid] = nw;
        }
        if (NV > NS && j0 + NS < NV) request(j0 + NS);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) part[sub][4 * t65 + i] = acc[i];
    __syncthreads();
    // column sums of this CTA into the first CTA's memory
    if (CL > 1) cluster_wait();                       // every CTA of the cluster has started
    if (tid < kCols) {
        double nsum = 0.0;
#pragma unroll
        for (int i = 0; i < kSub; ++i)
#pragma unroll
            for (int r4 = 0; r4 < 4; ++r4) nsum += part[i][r4 * kCols + tid];
        if (CL == 1) {
            red[0][tid] = nsum;
        } else {
            unsigned dst;
            asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(dst) : "r"((unsigned)__cvta_generic_to_shared(&red[cr][tid])));
            asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(dst), "d"(nsum) : "memory");
        }
    }
    if (CL > 1) cluster_arrive(); else __syncthreads();
#pragma unroll
    for (int j = NV - NS; j < NV; ++j) S[(sub + j * kSub) * kCols] = sbuf[(j % NS) * kThreads + tid];
    if (cr != 0) return;                              // nobody reads this CTA's memory
    if (CL > 1) cluster_wait();
    if (tid < 96) {                                   // (three whole warps)
        const int c = tid < kCols ? tid : 64;
        double nsum = 0.0, dsum = 0.0;
#pragma unroll
        for (int i = 0; i < CL; ++i) { nsum += red[i][c]; dsum += red[i][64]; }
        const float d = 1.f + (float)dsum;
        if (tid < 64) stf(o + (size_t)bh * 64 + tid, (float)nsum / d);
        if (tid == 64 && denom != nullptr) denom[bh] = d;
    }
}

bool decode_shape_ok(const psk_shape* sh) {
    return sh != nullptr && (sh->dtype == PSK_F32 || sh->dtype == PSK_BF16) && sh->B > 0 && sh->H > 0 &&
           (int64_t)sh->B * sh->H < ((int64_t)1 << 31) && (sh->g_heads == 1 || sh->g_heads == sh->H);
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

template <typename T, int R, int CL>
cudaError_t launch_cl(const psk_shape* sh, const void* q, const void* k, const void* v, const void* G1, const void* G2,
                      float* state, void* o, float* denom, cudaStream_t s) {
    auto kern = decode_step_kernel<T, R, CL>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Dec<R, CL>::kSmem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(sh->B * sh->H * CL));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = Dec<R, CL>::kSmem;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CL; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kern, (const T*)q, (const T*)k, (const T*)v, (const T*)G1, (const T*)G2, (int)sh->g_heads, (int)sh->H, state,
                              (T*)o, denom);
}

template <typename T, int R>
cudaError_t launch_r(const psk_shape* sh, const void* q, const void* k, const void* v, const void* G1, const void* G2,
                     float* state, void* o, float* denom, cudaStream_t s) {
    // CTAs per head.  Few heads: as many as a cluster holds, so that more SMs work on the step (12 heads,
    // r = 32: 16.4, 10.3, 8.2, 6.2 us with 1, 2, 4, 8).  Many: no more than about three CTAs per SM in all, because
    // every CTA forms the half sketches anew and the cluster's sum costs time too (384 heads, r = 32:
    // 45.7, 47.8, 52.8, 48.5 us with 1, 2, 4, 8).  With r = 64 a CTA's part is long enough for four to pay (192 heads: 77.8 us
    // with 4, 86.6 with 2).
    const long heads = (long)sh->B * sh->H, most = 444;
    if (heads * 8 <= most) return launch_cl<T, R, 8>(sh, q, k, v, G1, G2, state, o, denom, s);
    if (R == 64 || heads * 4 <= most) return launch_cl<T, R, 4>(sh, q, k, v, G1, G2, state, o, denom, s);
    if constexpr (R != 64) {
        if (heads * 2 <= most) return launch_cl<T, R, 2>(sh, q, k, v, G1, G2, state, o, denom, s);
        return launch_cl<T, R, 1>(sh, q, k, v, G1, G2, state, o, denom, s);
    }
}

template <typename T>
cudaError_t launch(const psk_shape* sh, const void* q, const void* k, const void* v, const void* G1, const void* G2,
                   float* state, void* o, float* denom, cudaStream_t s) {
    cudaError_t e;
    prof_begin("decode_step_kernel", s);
    switch (sh->r) {
        case 16: e = launch_r<T, 16>(sh, q, k, v, G1, G2, state, o, denom, s); break;
        case 32: e = launch_r<T, 32>(sh, q, k, v, G1, G2, state, o, denom, s); break;
        default: e = launch_r<T, 64>(sh, q, k, v, G1, G2, state, o, denom, s); break;
    }
    prof_end(s);
    return e == cudaSuccess ? cudaGetLastError() : e;
}

}  // namespace
}  // namespace psk

using namespace psk;

extern "C" {

size_t psk_decode_state_bytes(const psk_shape* shape) {
    if (!decode_shape_ok(shape) || (shape->r != 16 && shape->r != 32 && shape->r != 64)) return 0;
    return (size_t)shape->B * shape->H * shape->r * shape->r * kCols * sizeof(float);
}

int psk_decode_step(const psk_shape* shape, const void* q, const void* k, const void* v, const void* G1,
                    const void* G2, float* state, void* o, float* denom, void* stream) {
    if (shape == nullptr) return PSK_ERR_INVALID_ARG;
    if (shape->dtype != PSK_F32 && shape->dtype != PSK_BF16) return PSK_ERR_INVALID_ARG;
    if (!decode_shape_ok(shape)) return PSK_ERR_SHAPE;
    if (shape->p != 4 || shape->h != 64 || (shape->r != 16 && shape->r != 32 && shape->r != 64) || shape->flags != 0)
        return PSK_ERR_UNSUPPORTED;
    if (!q || !k || !v || !G1 || !G2 || !state || !o) return PSK_ERR_INVALID_ARG;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(G1) || !aligned16(G2) || !aligned16(state) ||
        !aligned16(o))
        return PSK_ERR_ALIGN;
    cudaStream_t s = (cudaStream_t)stream;
    const cudaError_t e = shape->dtype == PSK_BF16
                              ? launch<__nv_bfloat16>(shape, q, k, v, G1, G2, state, o, denom, s)
                              : launch<float>(shape, q, k, v, G1, G2, state, o, denom, s);
    return e == cudaSuccess ? PSK_OK : PSK_ERR_CUDA;
}

}  // extern "C"
