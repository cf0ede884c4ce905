// lt(A B^T) C for arbitrary feature matrices by the block algorithm of Section 3.1:
//   H_l = B_l^T C_l,  Z_l = sum_{j<l} H_j,  rows of block l = lt(A_l B_l^T) C_l + A_l Z_l.
// The attention kernels specialise this to A = phi'(Q), B = phi'(K), C = [V | 1] with the
// features generated on the fly; this entry point takes the feature matrices as given (the
// paper applies the same algorithm to other feature maps, Section 4).  fp32 on the CUDA cores, in
// terms of the register-tiled products of cc_gemm.cuh; any m, k <= 128, no alignment asked for.
#include "cc_gemm.cuh"

#include <type_traits>

namespace psk {
namespace {

using namespace cc;

// Asynchronous copy of one float (zero when `in` is false), or of four.
__device__ __forceinline__ void cp4z(float* dst, const float* src, bool in) {
    const int sz = in ? 4 : 0;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "r"(sz) : "memory");
}
__device__ __forceinline__ void cp16z(float* dst, const float* src, bool in) {
    const int sz = in ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "r"(sz) : "memory");
}

// dst[ROWS][ld] = src[row0 .. ][col0 .. col0 + COLS) of a row-major matrix with `stride` columns; entries at
// or beyond (nrows, ncols) become zero.  `vec`: rows are 16-byte aligned and ncols is a multiple of 4.
template <int ROWS, int COLS>
__device__ __forceinline__ void load_tile(float* dst, int ld, const float* src, int64_t stride, int nrows, int col0, int ncols, bool vec,
                                          int tid, int nthr) {
    if (vec) {
        for (int e = tid; e < ROWS * (COLS / 4); e += nthr) {
            const int r = e / (COLS / 4), c = col0 + 4 * (e % (COLS / 4));
            const bool in = r < nrows && c < ncols;
            cp16z(dst + r * ld + c - col0, in ? src + r * stride + c : src, in);
        }
    } else {
        for (int e = tid; e < ROWS * COLS; e += nthr) {
            const int r = e / COLS, c = col0 + e % COLS;
            const bool in = r < nrows && c < ncols;
            cp4z(dst + r * ld + c - col0, in ? src + r * stride + c : src, in);
        }
    }
}
// the transpose of a [64 rows][32 columns] piece: dst[32][kLd]
__device__ __forceinline__ void load_tile_transposed(float* dst, const float* src, int64_t stride, int nrows, int col0, int ncols, int lane) {
    for (int e = lane; e < 64 * 32; e += 64) {
        const int r = e / 32, c = col0 + e % 32;
        const bool in = r < nrows && c < ncols;
        cp4z(dst + (e % 32) * kLd + r, in ? src + r * stride + c : src, in);
    }
}

// 8 rows x 4 NH columns per thread of the outer form: columns 32 h + 4 cx + 0..3, h < NH
template <int NH>
struct AccN {
    f2 s[4][2 * NH], x[4][2 * NH];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int q = 0; q < 2 * NH; ++q) s[p][q] = x[p][q] = 0ull;
    }
    __device__ __forceinline__ void step(const f2 (&a)[4], const float* b) {
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            const F22 u = lds22(b + 32 * h);
            const f2 c[2] = {u.x, u.y};
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const f2 sw = swap2(c[q]);
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    s[p][2 * h + q] = fma2(a[p], c[q], s[p][2 * h + q]);
                    x[p][2 * h + q] = fma2(a[p], sw, x[p][2 * h + q]);
                }
            }
        }
    }
    // token 8 ry + q of the diagonal tile (cc_gemm.cuh, diagonal_step)
    __device__ __forceinline__ void diagonal(const f2 (&a)[4], const float* b, int q) {
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            const F22 u = lds22(b + 32 * h);
            const f2 c[2] = {u.x, u.y};
            diagonal_step<false>(s, x, a, c, 2 * h, q);
        }
    }
    __device__ __forceinline__ float at(int i, int h, int j) const {       // row i, column 32 h + 4 cx + j
        const f2 v = ((i ^ j) & 1) ? x[i / 2][2 * h + j / 2] : s[i / 2][2 * h + j / 2];
        return (i & 1) ? hi2(v) : lo2(v);
    }
};

// ---------------------------------------------------------------------------
// H_l = B_l^T C_l into slot l + 1 (the first prefix it enters).  grid (ceil(m / 128), t - 1, batch),
// 128 threads: two groups of 64 features share the rows of C; 32 rows per step, the next in flight.
// ---------------------------------------------------------------------------
template <int NH> constexpr int kLdc = 32 * NH + 4;
template <int NH> constexpr size_t kStateSmem = 2 * (32 * 128 + 32 * kLdc<NH>) * sizeof(float);

template <int NH>
__global__ void __launch_bounds__(128, NH <= 2 ? 4 : 2)
lt_state_kernel(const float* __restrict__ B, const float* __restrict__ C, int n, int m, int k, int b, int t, bool vm, bool vk,
                float* __restrict__ S) {
    pdl_sync();
    extern __shared__ __align__(16) float smem[];
    constexpr int LDC = kLdc<NH>, kBuf = 32 * 128 + 32 * LDC;
    const int tid = threadIdx.x, grp = tid / 64, lane = tid % 64, ry = lane / 8, cx = lane % 8;
    const int f0 = blockIdx.x * 128, l = blockIdx.y, bt = blockIdx.z;
    const size_t row0 = (size_t)bt * n + (size_t)l * b;
    auto load = [&](int st) {
        float* dst = smem + (st & 1) * kBuf;
        load_tile<32, 128>(dst, 128, B + (row0 + st * 32) * m, m, 32, f0, m, vm, tid, 128);
        load_tile<32, 32 * NH>(dst + 32 * 128, LDC, C + (row0 + st * 32) * k, k, 32, 0, k, vk, tid, 128);
        cp_commit();
    };
    AccN<NH> acc;
    acc.zero();
    const int ns = b / 32;
    load(0);
    for (int st = 0; st < ns; ++st) {
        if (st + 1 < ns) { load(st + 1); cp_wait<1>(); } else { cp_wait<0>(); }
        __syncthreads();
        const float* a0 = smem + (st & 1) * kBuf + 64 * grp + 8 * ry;
        const float* c0 = smem + (st & 1) * kBuf + 32 * 128 + 4 * cx;
#pragma unroll 4
        for (int j = 0; j < 32; ++j) {
            f2 a[4];
            load_rows8(a, a0 + j * 128);
            acc.step(a, c0 + j * LDC);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int f = f0 + 64 * grp + 8 * ry + i;
        if (f >= m) continue;
        float* out = S + (((size_t)bt * t + l + 1) * m + f) * k;
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            const int c = 32 * h + 4 * cx;
            if (vk) {
                if (c < k) *reinterpret_cast<float4*>(out + c) = make_float4(acc.at(i, h, 0), acc.at(i, h, 1), acc.at(i, h, 2), acc.at(i, h, 3));
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) if (c + j < k) out[c + j] = acc.at(i, h, j);
            }
        }
    }
}

// Inclusive prefix over slots 1 .. t-1 of each batch entry, in place, eight slots in flight per thread.
template <typename V>
__device__ __forceinline__ void add_to(V& a, const V& b);
template <> __device__ __forceinline__ void add_to<float>(float& a, const float& b) { a += b; }
template <> __device__ __forceinline__ void add_to<float4>(float4& a, const float4& b) { a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w; }

template <typename V>
__global__ void __launch_bounds__(256)
lt_scan_kernel(V* __restrict__ S, size_t elems, int t) {
    pdl_sync();
    const size_t e = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (e >= elems) return;
    V* p = S + (size_t)blockIdx.y * t * elems + e;
    V run = p[elems];
    for (int k0 = 2; k0 < t; k0 += 8) {
        V v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) if (k0 + q < t) v[q] = p[(size_t)(k0 + q) * elems];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            if (k0 + q >= t) break;
            add_to<V>(run, v[q]);
            p[(size_t)(k0 + q) * elems] = run;
        }
    }
}

// ---------------------------------------------------------------------------
// 64 rows of block l:  A_l Z_l  +  sum over the block's 64-row tiles up to the own one of
// lt(A_tile B_tile^T) C_tile.  grid (ceil(b / 64), t, batch), heaviest row tiles first; two groups of 64
// threads take the tiles in turn, then the features of A_l Z_l are shared out so that both end
// together; their sums meet in shared memory.  Scores in dot form (both operands' features are
// contiguous), 32 features per step; the other two products in outer form.
// ---------------------------------------------------------------------------
constexpr int kLdf = 36;                                  // 32 features of a row, padded
template <int NH> struct OutSmem {
    static constexpr int C = 4 * 64 * kLdf;               // two steps of (A, B) pieces; also the weights [64][kLd]
    static constexpr int grp = C + 64 * kLdc<NH>;
    static constexpr int zbuf = 32 * kLd + 32 * kLdc<NH>; // one step of A_l Z_l
    static_assert(2 * zbuf <= grp && kUnit <= C && 64 * kLdc<NH> <= grp, "buffers");
    static constexpr size_t bytes = 2 * (size_t)grp * sizeof(float);
};

template <int NH>
__global__ void __launch_bounds__(128)
lt_out_kernel(const float* __restrict__ A, const float* __restrict__ B, const float* __restrict__ C,
              const float* __restrict__ Z, int n, int m, int k, int b, int t, bool vm, bool vk, float* __restrict__ Out) {
    pdl_sync();
    extern __shared__ __align__(16) float smem[];
    using L = OutSmem<NH>;
    constexpr int LDC = kLdc<NH>;
    const int tid = threadIdx.x, grp = tid / 64, lane = tid % 64, ry = lane / 8, cx = lane % 8;
    const int tile = gridDim.x - 1 - blockIdx.x, l = blockIdx.y, bt = blockIdx.z;
    float* sG = smem + grp * L::grp;
    const size_t blk0 = (size_t)bt * n + (size_t)l * b;
    const float* Ao = A + (blk0 + tile * 64) * m;
    const int nown = b - tile * 64, nf = (m + 31) / 32;   // (rows of the last tile beyond the block read as zeros)
    AccN<NH> acc;
    acc.zero();
    for (int jt = grp; jt <= tile; jt += 2) {
        const float* Bj = B + (blk0 + jt * 64) * m;
        auto load = [&](int st) {
            float* dst = sG + (st & 1) * 2 * 64 * kLdf;
            load_tile<64, 32>(dst, kLdf, Ao, m, nown, st * 32, m, vm, lane, 64);
            load_tile<64, 32>(dst + 64 * kLdf, kLdf, Bj, m, b - jt * 64, st * 32, m, vm, lane, 64);
            cp_commit();
        };
        load_tile<64, 32 * NH>(sG + L::C, LDC, C + (blk0 + jt * 64) * k, k, b - jt * 64, 0, k, vk, lane, 64);
        load(0);
        float w[8][8];
        auto steps = [&](auto full, int half) {
            constexpr int NR = decltype(full)::value ? 8 : 4;
            f2 d[NR][8];
#pragma unroll
            for (int i = 0; i < NR; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) d[i][j] = 0ull;
            for (int st = 0; st < nf; ++st) {
                if (st + 1 < nf) { load(st + 1); cp_wait<1>(); } else { cp_wait<0>(); }
                group_sync(grp);
                const float* a0 = sG + (st & 1) * 2 * 64 * kLdf + (ry + 32 * half) * kLdf;
                const float* b0 = sG + (st & 1) * 2 * 64 * kLdf + (64 + cx) * kLdf;
#pragma unroll 1
                for (int q = 0; q < 32; q += 4) {
                    F22 bv[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) bv[j] = lds22(b0 + 8 * j * kLdf + q);
#pragma unroll
                    for (int i = 0; i < NR; ++i) {
                        const F22 av = lds22(a0 + 8 * i * kLdf + q);
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            d[i][j] = fma2(av.x, bv[j].x, d[i][j]);
                            d[i][j] = fma2(av.y, bv[j].y, d[i][j]);
                        }
                    }
                }
                group_sync(grp);
            }
#pragma unroll
            for (int i = 0; i < NR; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const bool keep = jt < tile || cx + 8 * j <= ry + 32 * half + 8 * i;       // lt(): keep j <= i
                    w[4 * half + i][j] = keep ? sum2(d[i][j]) : 0.f;
                }
        };
        if constexpr (NH <= 2) {
            steps(std::true_type{}, 0);
        } else {                                          // (registers: half of the scores at a time)
            steps(std::false_type{}, 0);
            load(0);
            steps(std::false_type{}, 1);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) sG[(cx + 8 * j) * kLd + ry + 8 * i] = w[i][j];
        group_sync(grp);
        const int j1 = jt < tile ? 64 : 8 * ry;
#pragma unroll 2
        for (int j = 0; j < j1; ++j) {
            f2 a[4];
            load_rows8(a, sG + j * kLd + 8 * ry);
            acc.step(a, sG + L::C + j * LDC + 4 * cx);
        }
        if (jt == tile) {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                f2 a[4];
                load_rows8(a, sG + (8 * ry + q) * kLd + 8 * ry);
                acc.diagonal(a, sG + L::C + (8 * ry + q) * LDC + 4 * cx, q);
            }
        }
        group_sync(grp);
    }
    // earlier blocks through the prefix state: with an odd number of tiles the second group, which
    // had one less of them, takes all the features, else half
    if (l > 0) {
        const int mid = (tile & 1) ? nf / 2 : 0, lo = grp ? mid : 0, hi = grp ? nf : mid;
        const float* Zl = Z + ((size_t)bt * t + l) * m * k;
        auto load = [&](int st) {
            float* dst = sG + ((st - lo) & 1) * L::zbuf;
            load_tile_transposed(dst, Ao, m, nown, st * 32, m, lane);
            load_tile<32, 32 * NH>(dst + 32 * kLd, LDC, Zl + (size_t)st * 32 * k, k, m - st * 32, 0, k, vk, lane, 64);
            cp_commit();
        };
        if (lo < hi) load(lo);
        for (int st = lo; st < hi; ++st) {
            if (st + 1 < hi) { load(st + 1); cp_wait<1>(); } else { cp_wait<0>(); }
            group_sync(grp);
            const float* a0 = sG + ((st - lo) & 1) * L::zbuf + 8 * ry;
            const float* z0 = sG + ((st - lo) & 1) * L::zbuf + 32 * kLd + 4 * cx;
#pragma unroll 2
            for (int f = 0; f < 32; ++f) {
                f2 a[4];
                load_rows8(a, a0 + f * kLd);
                acc.step(a, z0 + f * LDC);
            }
            group_sync(grp);
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int h = 0; h < NH; ++h)
            *reinterpret_cast<float4*>(sG + (8 * ry + i) * LDC + 32 * h + 4 * cx) =
                make_float4(acc.at(i, h, 0), acc.at(i, h, 1), acc.at(i, h, 2), acc.at(i, h, 3));
    __syncthreads();
    float* out = Out + (blk0 + tile * 64) * k;
    const float* p0 = smem;
    const float* p1 = smem + L::grp;
    if (vk) {
        for (int e = tid; e < 64 * 8 * NH; e += 128) {
            const int r = e / (8 * NH), c = 4 * (e % (8 * NH));
            if (r >= nown || c >= k) continue;
            const float4 u = *reinterpret_cast<const float4*>(p0 + r * LDC + c), v = *reinterpret_cast<const float4*>(p1 + r * LDC + c);
            *reinterpret_cast<float4*>(out + (size_t)r * k + c) = make_float4(u.x + v.x, u.y + v.y, u.z + v.z, u.w + v.w);
        }
    } else {
        for (int e = tid; e < 64 * 32 * NH; e += 128) {
            const int r = e / (32 * NH), c = e % (32 * NH);
            if (r < nown && c < k) out[(size_t)r * k + c] = p0[r * LDC + c] + p1[r * LDC + c];
        }
    }
}

bool lt_args_ok(int batch, int n, int m, int k, int b) {
    return batch > 0 && n > 0 && m > 0 && k > 0 && k <= 128 && b > 0 && b % 32 == 0 && n % b == 0 &&
           (int64_t)batch * n < ((int64_t)1 << 31);
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// NH: 32-column groups of the k columns.
template <int NH>
cudaError_t lt_run(int batch, int n, int m, int k, int b, const float* A, const float* B, const float* C, float* Out, float* S,
                   cudaStream_t s) {
    const int t = n / b;
    // 16-byte copies and stores where every row of the matrices and of the states starts on 16 bytes
    const bool vm = m % 4 == 0 && aligned16(A) && aligned16(B);
    const bool vk = k % 4 == 0 && aligned16(C) && aligned16(Out) && aligned16(S);
    cudaError_t e = cudaFuncSetAttribute(lt_state_kernel<NH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStateSmem<NH>);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(lt_out_kernel<NH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OutSmem<NH>::bytes);
    if (e != cudaSuccess) return e;
    if (t > 1) {
        prof_begin("lt_state_kernel", s);
        launch_pdl(lt_state_kernel<NH>, dim3((m + 127) / 128, t - 1, batch), 128, kStateSmem<NH>, s, B, C, n, m, k, b, t, vm, vk, S);
        prof_end(s);
    }
    if (t > 2) {
        const size_t elems = (size_t)m * k;
        prof_begin("lt_scan_kernel", s);
        if (elems % 4 == 0 && aligned16(S))
            launch_pdl(lt_scan_kernel<float4>, dim3((unsigned)((elems / 4 + 255) / 256), batch), 256, 0, s, reinterpret_cast<float4*>(S), elems / 4, t);
        else
            launch_pdl(lt_scan_kernel<float>, dim3((unsigned)((elems + 255) / 256), batch), 256, 0, s, S, elems, t);
        prof_end(s);
    }
    prof_begin("lt_out_kernel", s);
    launch_pdl(lt_out_kernel<NH>, dim3((b + 63) / 64, t, batch), 128, OutSmem<NH>::bytes, s, A, B, C, S, n, m, k, b, t, vm, vk, Out);
    prof_end(s);
    return cudaGetLastError();
}

}  // namespace
}  // namespace psk

using namespace psk;

extern "C" {

size_t psk_lt_multiply_workspace_bytes(int batch, int n, int m, int k, int b) {
    if (!lt_args_ok(batch, n, m, k, b)) return 0;
    return align_up((size_t)batch * (n / b) * m * k * sizeof(float));
}

int psk_lt_multiply(int batch, int n, int m, int k, int b, const float* A, const float* B, const float* C,
                    float* Out, void* workspace, size_t workspace_bytes, void* stream) {
    if (!lt_args_ok(batch, n, m, k, b)) return PSK_ERR_SHAPE;
    if (!A || !B || !C || !Out) return PSK_ERR_INVALID_ARG;
    const size_t need = psk_lt_multiply_workspace_bytes(batch, n, m, k, b);
    if (!workspace || workspace_bytes < need) return PSK_ERR_WORKSPACE;
    cudaStream_t s = (cudaStream_t)stream;
    float* S = static_cast<float*>(workspace);
    cudaError_t e;
    switch ((k + 31) / 32) {
        case 1: e = lt_run<1>(batch, n, m, k, b, A, B, C, Out, S, s); break;
        case 2: e = lt_run<2>(batch, n, m, k, b, A, B, C, Out, S, s); break;
        case 3: e = lt_run<3>(batch, n, m, k, b, A, B, C, Out, S, s); break;
        default: e = lt_run<4>(batch, n, m, k, b, A, B, C, Out, S, s); break;
    }
    return e == cudaSuccess ? PSK_OK : PSK_ERR_CUDA;
}

}  // extern "C"
