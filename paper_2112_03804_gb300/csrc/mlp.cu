// Warm-start network: a 3-layer perceptron with BF16 weights and FP32
// accumulation, trained and evaluated by the kernels in this file.
//
//   H1 = relu(X W1 + b1),  H2 = relu(H1 W2 + b2),  Z = H2 W3 + b3,
//   P[q, a] = softmax over the node's actions a < nact[q] of Z[q, :]
//
// Loss: weighted cross-entropy against target strategies T,
//   L = - sum_q w_q sum_{a < nact_q} T[q,a] log P[q,a] / sum_q w_q,
// whose gradient at the logits is dZ = w_q (P - T) / sum w (zero for a >= nact).
// Weights live in FP32 (master copy, Adam moments) and BF16 (what the
// forward and backward products read); activations and gradients are FP32.
// The products are one tiled SIMT kernel (64x64 tile, 8x8 outputs per thread,
// k split over thread groups and CTAs) that reads either operand in either
// direction, so the same code computes X W, dZ W^T and X^T dH.  Not in the paper: a service for
// warm-starting the solver (Sec. 2's first-order methods start from a given
// strategy).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "abi_internal.h"
#include "mlp_internal.h"

using namespace kps_abi;

namespace {

constexpr int kBM = 64, kBN = 64, kBK = 8;   // output tile of a CTA, k slice of a group
constexpr int kPitch = kBM + 4;              // floats per k row of a staged operand

template <typename T> __device__ __forceinline__ float to_f(T v);
template <> __device__ __forceinline__ float to_f<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }

// 8 consecutive elements as floats (vector: 16-byte aligned).
__device__ __forceinline__ void load8(const float *p, float *v) {
    const float4 a = reinterpret_cast<const float4 *>(p)[0], b = reinterpret_cast<const float4 *>(p)[1];
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void load8(const __nv_bfloat16 *p, float *v) {
    const uint4 u = *reinterpret_cast<const uint4 *>(p);
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        v[2 * i] = __uint_as_float(w[i] << 16);
        v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
}

// A thread's 8 elements of a group's [8 k][64 r] operand slice: with k
// contiguous in memory row r = t and all 8 k, else k = t / 8 and the 8 rows
// 8 (t % 8)...; zeros outside [0, R) x [k0, kend).
template <bool KC, typename T>
__device__ __forceinline__ void fetch(const T *__restrict__ A, long long ld, int r0, int R, int k0, int kend, bool vec,
                                      int t, float *v) {
    const int r = r0 + (KC ? t : 8 * (t & 7)), k = k0 + (KC ? 0 : t >> 3);
    const T *p = KC ? A + (long long)r * ld + k : A + (long long)k * ld + r;
    const bool full = KC ? (r < R && k + 8 <= kend) : (k < kend && r + 8 <= R);
    if (full && vec) {
        load8(p, v);
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const bool in = KC ? (r < R && k + i < kend) : (k < kend && r + i < R);
            v[i] = in ? to_f<T>(p[i]) : 0.f;
        }
    }
}
template <bool KC>
__device__ __forceinline__ void stage(float *S, int t, const float *v) {
    if (KC) {
#pragma unroll
        for (int i = 0; i < 8; ++i) S[i * kPitch + t] = v[i];
    } else {
        float *q = S + (t >> 3) * kPitch + 8 * (t & 7);
        reinterpret_cast<float4 *>(q)[0] = make_float4(v[0], v[1], v[2], v[3]);
        reinterpret_cast<float4 *>(q)[1] = make_float4(v[4], v[5], v[6], v[7]);
    }
}

// Where a product's value goes: bias, ReLU, gate ([gate > 0]), store.
struct Epilogue {
    float *C;
    long long ldc;
    const float *bias;
    int relu;
    const float *gate;
    long long ldg;
    __device__ __forceinline__ void put(int m, int n, float v) const {
        if (bias) v += bias[n];
        if (relu) v = fmaxf(v, 0.f);
        if (gate && !(gate[(long long)m * ldg + n] > 0.f)) v = 0.f;
        C[(long long)m * ldc + n] = v;
    }
    // 16-byte loads and stores of its rows are aligned
    bool vec_ok() const {
        auto a = [](const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
        return a(C) && ldc % 4 == 0 && a(bias) && a(gate) && (!gate || ldg % 4 == 0);
    }
    // Columns n .. n + 3, the last ones maybe past N
    __device__ __forceinline__ void put4(int m, int n, int N, float4 v, bool vec) const {
        if (vec && n + 4 <= N) {
            if (bias) {
                const float4 b = *reinterpret_cast<const float4 *>(bias + n);
                v.x += b.x; v.y += b.y; v.z += b.z; v.w += b.w;
            }
            if (relu) v = make_float4(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f), fmaxf(v.z, 0.f), fmaxf(v.w, 0.f));
            if (gate) {
                const float4 g = *reinterpret_cast<const float4 *>(gate + (long long)m * ldg + n);
                if (!(g.x > 0.f)) v.x = 0.f;
                if (!(g.y > 0.f)) v.y = 0.f;
                if (!(g.z > 0.f)) v.z = 0.f;
                if (!(g.w > 0.f)) v.w = 0.f;
            }
            *reinterpret_cast<float4 *>(C + (long long)m * ldc + n) = v;
        } else {
            if (n < N) put(m, n, v.x);
            if (n + 1 < N) put(m, n + 1, v.y);
            if (n + 2 < N) put(m, n + 2, v.z);
            if (n + 3 < N) put(m, n + 3, v.w);
        }
    }
};

// C(m,n) = sum_k A(m,k) B(k,n), then the epilogue.  A(m,k) = A[m*lda + k] (AK)
// or A[k*lda + m]; B(k,n) = B[n*ldb + k] (BK) or B[k*ldb + n].
//
// FP32 FMAs, because the operands are FP32 activations and gradients that are
// not to be rounded: bound by the FMA pipe (4096 x 1232 x 256 is 2.6 GFLOP,
// 35 us at 152 SMs x 128 lanes).  A thread owns 8 x 8 outputs, as packed
// FP32x2 pairs along n: 4 shared loads of 16 bytes feed 32 packed FMAs, where
// the 4 x 4 tile it replaces needed a load for every two FMAs.  The network's
// products have few output tiles (256 for 4096 x 256, 80 for a 1232 x 256
// weight gradient), so the k range is cut twice: each of KG groups of 64
// threads takes every KG-th slice of 8 k (its own double-buffered staging and
// named barrier; the groups' sums meet in shared memory), and blockIdx.z takes
// a contiguous part of k when the tiles alone would leave SMs idle (partials
// to `part`, added in order by reduce_kernel).  Both orders are fixed: results
// are bit-reproducible.  KG = 1 without a z split adds k in ascending order.
// Losses and gradients of a 4096-row minibatch: 1.53 ms before (64 x 64
// tiles of 4 x 4 outputs per thread, no k split), 0.31 ms now; of 0.38 -> 0.31
// half by unrolling two k instead of eight (which spilled registers) and half
// by the tile's way out through shared memory (one group stored it 4 bytes at a
// time, each behind its gate's load).  The first layer's product takes 75 us: 57 %
// of the FMA pipe on 256 of 304 resident CTAs, short of its global loads; the
// shared loads take two thirds of the pipe's time, so A staged with every value
// twice (no register pairs to build, half as many loads again) is 1.15x slower.
template <int KG, bool AK, bool BK, typename TA, typename TB>
__global__ void __launch_bounds__(64 * KG, KG == 1 ? 8 : 2)
gemm_kernel(int M, int N, int K, int kpart, const TA *__restrict__ A, long long lda, int avec,
            const TB *__restrict__ B, long long ldb, int bvec, float *__restrict__ part, const Epilogue ep, int evec) {
    constexpr int kBuf = kBK * kPitch;                       // one operand, one stage
    constexpr int kRed = KG == 1 ? 0 : KG / 2 * kBM * kBN;   // sums handed over between groups
    __shared__ __align__(16) float sh[KG * 4 * kBuf > kRed ? KG * 4 * kBuf : kRed];
    const int t = threadIdx.x & 63, grp = threadIdx.x >> 6;
    const int m0 = blockIdx.y * kBM, n0 = blockIdx.x * kBN;
    const int kb = blockIdx.z * kpart, kend = min(K, kb + kpart);
    float *As = sh + grp * 4 * kBuf, *Bs = As + 2 * kBuf;
    const int tr = t >> 3, tc = t & 7;
    auto sync_group = [&]() {
        if (KG == 1) __syncthreads();
        else asm volatile("bar.sync %0, 64;" ::"r"(grp + 1) : "memory");
    };
    float2 acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
    float va[8], vb[8];
    int k0 = kb + grp * kBK, st = 0;
    if (k0 < kend) {
        fetch<AK>(A, lda, m0, M, k0, kend, avec, t, va);
        fetch<BK>(B, ldb, n0, N, k0, kend, bvec, t, vb);
        stage<AK>(As, t, va);
        stage<BK>(Bs, t, vb);
    }
    sync_group();
    for (; k0 < kend; k0 += KG * kBK) {
        const int kn = k0 + KG * kBK;
        if (kn < kend) {
            fetch<AK>(A, lda, m0, M, kn, kend, avec, t, va);
            fetch<BK>(B, ldb, n0, N, kn, kend, bvec, t, vb);
        }
        const float *a = As + st * kBuf + 4 * tr, *b = Bs + st * kBuf + 4 * tc;
#pragma unroll 2
        for (int kk = 0; kk < kBK; ++kk) {
            const float4 a0 = *reinterpret_cast<const float4 *>(a + kk * kPitch);
            const float4 a1 = *reinterpret_cast<const float4 *>(a + kk * kPitch + 32);
            const float4 b0 = *reinterpret_cast<const float4 *>(b + kk * kPitch);
            const float4 b1 = *reinterpret_cast<const float4 *>(b + kk * kPitch + 32);
            const float ar[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float2 br[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w), make_float2(b1.x, b1.y),
                                  make_float2(b1.z, b1.w)};
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = __ffma2_rn(make_float2(ar[i], ar[i]), br[j], acc[i][j]);
        }
        st ^= 1;
        if (kn < kend) {
            stage<AK>(As + st * kBuf, t, va);
            stage<BK>(Bs + st * kBuf, t, vb);
        }
        sync_group();
    }
    // groups g and g + s meet pairwise, s halving: a fixed order
#pragma unroll
    for (int s = KG / 2; s >= 1; s >>= 1) {
        __syncthreads();
        if (grp >= s && grp < 2 * s) {
            float2 *r = reinterpret_cast<float2 *>(sh) + (grp - s) * (kBM * kBN / 2) + t;
#pragma unroll
            for (int e = 0; e < 32; ++e) r[64 * e] = acc[e >> 2][e & 3];
        }
        __syncthreads();
        if (grp < s) {
            const float2 *r = reinterpret_cast<const float2 *>(sh) + grp * (kBM * kBN / 2) + t;
#pragma unroll
            for (int e = 0; e < 32; ++e) acc[e >> 2][e & 3] = __fadd2_rn(acc[e >> 2][e & 3], r[64 * e]);
        }
    }
    // the tile goes through shared memory, so that every thread of the CTA
    // stores (and reads bias and gate) 16 bytes at a time, rows contiguous
    Epilogue out = ep;
    if (part) out = Epilogue{part + (long long)blockIdx.z * M * N, N, nullptr, 0, nullptr, 0};
    const bool vec = part ? N % 4 == 0 : evec != 0;
    if (KG == 1) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int m = m0 + 4 * tr + (i & 3) + 32 * (i >> 2);
            if (m >= M) continue;
#pragma unroll
            for (int j = 0; j < 2; ++j)
                out.put4(m, n0 + 4 * tc + 32 * j, N,
                         make_float4(acc[i][2 * j].x, acc[i][2 * j].y, acc[i][2 * j + 1].x, acc[i][2 * j + 1].y), vec);
        }
        return;
    }
    __syncthreads();
    if (grp == 0) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j)
                *reinterpret_cast<float4 *>(sh + (4 * tr + (i & 3) + 32 * (i >> 2)) * kPitch + 4 * tc + 32 * j) =
                    make_float4(acc[i][2 * j].x, acc[i][2 * j].y, acc[i][2 * j + 1].x, acc[i][2 * j + 1].y);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < kBM * kBN / 4; e += 64 * KG) {
        const int r = e >> 4, c = 4 * (e & 15);
        if (m0 + r < M) out.put4(m0 + r, n0 + c, N, *reinterpret_cast<const float4 *>(sh + r * kPitch + c), vec);
    }
}

// C = A W for few rows, one thread an output: the same sums as gemm_kernel<1>
// (k in ascending order), which had one CTA per 64 rows walk all k with a
// barrier every 8: a whole prediction for one game (2 rows of K = 1133 among its
// products) 187 us with it, 125 here, bound by the round trips of 32 loads at a
// time.  Every row reads W once more (L2): 256 games' 512 rows are the last that
// gain (128 games 3.24 -> 3.11 ms, 300 games by tiles as before).
constexpr int kFewRows = 512;
__global__ void __launch_bounds__(64) few_rows_kernel(int N, int K, const float *__restrict__ A, long long lda,
                                                      const __nv_bfloat16 *__restrict__ W, long long ldw,
                                                      float *__restrict__ C, long long ldc) {
    const int n = blockIdx.x * 64 + threadIdx.x;
    if (n >= N) return;
    const float *a = A + (long long)blockIdx.y * lda;
    const __nv_bfloat16 *w = W + n;
    float s = 0.f;
#pragma unroll 32
    for (int k = 0; k < K; ++k) s = fmaf(a[k], __bfloat162float(w[(long long)k * ldw]), s);
    C[(long long)blockIdx.y * ldc + n] = s;
}

// The z parts of a split product added in order, then the epilogue.
__global__ void __launch_bounds__(256) reduce_kernel(int M, int N, int nz, const float *__restrict__ part,
                                                     const Epilogue ep) {
    const long long i = (long long)blockIdx.x * 256 + threadIdx.x, mn = (long long)M * N;
    if (i >= mn) return;
    float v = part[i];
    for (int z = 1; z < nz; ++z) v += part[z * mn + i];
    ep.put((int)(i / N), (int)(i % N), v);
}

// Column sums of G [M x N] (bias gradients): the rows in gridDim.y parts, a
// warp row of 32 columns per 8 rows of threads; the parts are added by
// reduce_kernel (as an [1 x N] product of gridDim.y parts).
__global__ void __launch_bounds__(256) colsum_kernel(int M, int N, int rows, const float *__restrict__ G,
                                                     float *__restrict__ part) {
    __shared__ float red[8][33];
    const int x = threadIdx.x & 31, y = threadIdx.x >> 5, n = blockIdx.x * 32 + x;
    const int m0 = blockIdx.y * rows, m1 = min(M, m0 + rows);
    float s = 0.f;
    if (n < N)
        for (int m = m0 + y; m < m1; m += 8) s += G[(long long)m * N + n];
    red[y][x] = s;
    __syncthreads();
    if (y == 0 && n < N) {
#pragma unroll
        for (int i = 1; i < 8; ++i) s += red[i][x];
        part[(long long)blockIdx.y * N + n] = s;
    }
}

// Masked softmax of each row; with targets: per-row loss terms and dZ.
// One thread per row (rows have at most 32 outputs).
__global__ void softmax_kernel(int Q, int D, const float *__restrict__ Z, const int *__restrict__ nact,
                               float *__restrict__ P, const float *__restrict__ T, const float *__restrict__ w,
                               float inv_wsum, float *__restrict__ dZ, float *__restrict__ row_loss) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= Q) return;
    const int na = nact[q];
    const float *z = Z + (long long)q * D;
    float mx = -INFINITY;
    for (int a = 0; a < na; ++a) mx = fmaxf(mx, z[a]);
    float s = 0.f;
    for (int a = 0; a < na; ++a) s += expf(z[a] - mx);
    const float ls = logf(s);
    float loss = 0.f;
    for (int a = 0; a < D; ++a) {
        const float p = a < na ? expf(z[a] - mx - ls) : 0.f;
        if (P) P[(long long)q * D + a] = p;
        if (T) {
            const float t = a < na ? T[(long long)q * D + a] : 0.f;
            if (a < na && t > 0.f) loss -= t * (z[a] - mx - ls);
            dZ[(long long)q * D + a] = a < na ? w[q] * inv_wsum * (p - t) : 0.f;
        }
    }
    if (T) row_loss[q] = w[q] * inv_wsum * loss;
}

__global__ void sum_kernel(int n, const float *__restrict__ v, float *__restrict__ out) {
    __shared__ float red[256];
    float s = 0.f;
    for (int i = threadIdx.x; i < n; i += 256) s += v[i];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int st = 128; st > 0; st >>= 1) {
        if (threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = red[0];
}

// Adam on the FP32 master weights, then the BF16 copy.
__global__ void adam_kernel(long long n, float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                            float *__restrict__ v, __nv_bfloat16 *__restrict__ ph, float lr, float b1, float b2,
                            float eps, float c1, float c2) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = pi;
    if (ph) ph[i] = __float2bfloat16_rn(pi);
}

__global__ void to_bf16_kernel(long long n, const float *__restrict__ p, __nv_bfloat16 *__restrict__ ph) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) ph[i] = __float2bfloat16_rn(p[i]);
}

template <typename T>
bool vec_ok(const T *p, long long ld) {
    return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && ld % (16 / (long long)sizeof(T)) == 0;
}

// Parts of k: enough CTAs for two per SM, each with at least kMinPart k.
constexpr int kMinPart = 256, kMaxParts = 32;
int gemm_parts(int M, int N, int K, int sms) {
    const long long tiles = (long long)((M + kBM - 1) / kBM) * ((N + kBN - 1) / kBN);
    return (int)std::max<long long>(1, std::min<long long>({2LL * sms / tiles, (long long)K / kMinPart, (long long)kMaxParts}));
}

// `part`: nz * M * N floats when nz > 1 (gemm_parts), else unused.
template <int KG, bool AK, bool BK, typename TA, typename TB>
cudaError_t gemm(int M, int N, int K, const TA *A, long long lda, const TB *B, long long ldb, const Epilogue &ep, int nz,
                 float *part, cudaStream_t st) {
    if (M <= 0 || N <= 0) return cudaSuccess;
    const int slice = KG * kBK;
    const int kpart = nz > 1 ? ((K + nz - 1) / nz + slice - 1) / slice * slice : K;
    dim3 grid((N + kBN - 1) / kBN, (M + kBM - 1) / kBM, nz);
    if (grid.y > 65535) return cudaErrorInvalidValue;
    gemm_kernel<KG, AK, BK, TA, TB><<<grid, 64 * KG, 0, st>>>(M, N, K, kpart, A, lda, vec_ok(A, lda), B, ldb,
                                                              vec_ok(B, ldb), nz > 1 ? part : nullptr, ep, ep.vec_ok());
    if (nz > 1)
        reduce_kernel<<<(unsigned)(((long long)M * N + 255) / 256), 256, 0, st>>>(M, N, nz, part, ep);
    return cudaGetLastError();
}

}  // namespace

namespace kps_abi {

cudaError_t mlp_gemm_xw(int M, int N, int K, const float *A, long long lda, const __nv_bfloat16 *W, long long ldw,
                        float *C, long long ldc, cudaStream_t st) {
    // k in ascending order: the predictor's activations are rounded to BF16
    if (M <= kFewRows) {
        if (M <= 0 || N <= 0) return cudaSuccess;
        few_rows_kernel<<<dim3((N + 63) / 64, M), 64, 0, st>>>(N, K, A, lda, W, ldw, C, ldc);
        return cudaGetLastError();
    }
    return gemm<1, true, false>(M, N, K, A, lda, W, ldw, Epilogue{C, ldc, nullptr, 0, nullptr, 0}, 1, nullptr, st);
}

}  // namespace kps_abi

namespace {

constexpr int kColParts = 64;   // row parts of a bias gradient

// Floats of the largest set of split-k partial products: a product takes more than one part only while all its parts
// are at most two tiles per SM, and a bias gradient kColParts rows.
size_t part_floats(const kps_mlp *m) {
    const size_t wide = std::max(m->width, m->dout);
    return std::max((size_t)2 * m->sms * kBM * kBN, kColParts * wide);
}

kps_status ensure_cap(kps_mlp *m, int rows) {
    if (rows <= m->cap) return KPS_OK;
    cudaFree(m->H1);
    cudaFree(m->H2);
    cudaFree(m->Z);
    cudaFree(m->dZ);
    cudaFree(m->dH1);
    cudaFree(m->dH2);
    cudaFree(m->row_loss);
    cudaFree(m->part);
    m->H1 = m->H2 = m->Z = m->dZ = m->dH1 = m->dH2 = m->row_loss = m->part = nullptr;
    m->cap = 0;
    const size_t r = (size_t)rows;
    cudaError_t e = kps::device_malloc(&m->H1, r * m->width * 4);
    if (e == cudaSuccess) e = kps::device_malloc(&m->H2, r * m->width * 4);
    if (e == cudaSuccess) e = kps::device_malloc(&m->Z, r * m->dout * 4);
    if (e == cudaSuccess) e = kps::device_malloc(&m->dZ, r * m->dout * 4);
    if (e == cudaSuccess) e = kps::device_malloc(&m->dH1, r * m->width * 4);
    if (e == cudaSuccess) e = kps::device_malloc(&m->dH2, r * m->width * 4);
    if (e == cudaSuccess) e = kps::device_malloc(&m->row_loss, r * 4);
    if (e == cudaSuccess) e = kps::device_malloc(&m->part, part_floats(m) * 4);
    if (e != cudaSuccess) return fail(KPS_ENOMEM, "network activations");
    m->cap = rows;
    return KPS_OK;
}

const __nv_bfloat16 *Wh(const kps_mlp *m, int l) { return m->ph + m->off[2 * l]; }
const float *Bf(const kps_mlp *m, int l) { return m->p + m->off[2 * l + 1]; }

// X W with W [K x N] as it is stored; split over k where the tiles are few.
cudaError_t gemm_xw(kps_mlp *m, int M, int N, int K, const float *A, const __nv_bfloat16 *W, const Epilogue &ep,
                    cudaStream_t st) {
    return gemm<4, true, false>(M, N, K, A, K, W, N, ep, gemm_parts(M, N, K, m->sms), m->part, st);
}
// G W^T with W [N x K] as it is stored.
cudaError_t gemm_gwt(kps_mlp *m, int M, int N, int K, const float *G, const __nv_bfloat16 *W, const Epilogue &ep,
                     cudaStream_t st) {
    return gemm<4, true, true>(M, N, K, G, K, W, K, ep, gemm_parts(M, N, K, m->sms), m->part, st);
}
// Weight and bias gradients of a layer: X^T G and the column sums of G.
cudaError_t gemm_xtg(kps_mlp *m, int M, int N, int Q, const float *X, const float *G, float *dW, float *db,
                     cudaStream_t st) {
    cudaError_t e = gemm<4, false, false>(M, N, Q, X, M, G, N, Epilogue{dW, N, nullptr, 0, nullptr, 0},
                                          gemm_parts(M, N, Q, m->sms), m->part, st);
    if (e != cudaSuccess) return e;
    // one part is the sum itself, a launch less (16 rows of a 33-65-12 network 75 -> 72 us)
    const int rows = Q <= 256 ? Q : std::max(64, (Q + kColParts - 1) / kColParts), parts = (Q + rows - 1) / rows;
    colsum_kernel<<<dim3((N + 31) / 32, parts), 256, 0, st>>>(Q, N, rows, G, parts > 1 ? m->part : db);
    if (parts > 1)
        reduce_kernel<<<(N + 255) / 256, 256, 0, st>>>(1, N, parts, m->part, Epilogue{db, N, nullptr, 0, nullptr, 0});
    return cudaGetLastError();
}

// Forward pass into H1, H2, Z (and P if given).
kps_status forward(kps_mlp *m, const float *X, int Q, const int *nact, float *P, cudaStream_t st) {
    const int D = m->din, W = m->width, O = m->dout;
    cudaError_t e = gemm_xw(m, Q, W, D, X, Wh(m, 0), Epilogue{m->H1, W, Bf(m, 0), 1, nullptr, 0}, st);
    if (e == cudaSuccess) e = gemm_xw(m, Q, W, W, m->H1, Wh(m, 1), Epilogue{m->H2, W, Bf(m, 1), 1, nullptr, 0}, st);
    if (e == cudaSuccess) e = gemm_xw(m, Q, O, W, m->H2, Wh(m, 2), Epilogue{m->Z, O, Bf(m, 2), 0, nullptr, 0}, st);
    if (e == cudaSuccess && P) {
        softmax_kernel<<<(Q + 127) / 128, 128, 0, st>>>(Q, O, m->Z, nact, P, nullptr, nullptr, 0.f, nullptr, nullptr);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return cuda_fail(e, "network forward");
    return KPS_OK;
}

kps_status backward(kps_mlp *m, const float *X, int Q, const int *nact, const float *T, const float *w,
                    float inv_wsum, float *loss, cudaStream_t st) {
    const int D = m->din, W = m->width, O = m->dout;
    softmax_kernel<<<(Q + 127) / 128, 128, 0, st>>>(Q, O, m->Z, nact, nullptr, T, w, inv_wsum, m->dZ, m->row_loss);
    cudaError_t e = cudaGetLastError();
    float *g = m->g;
    // layer 3: dW3 = H2^T dZ, db3 = colsum dZ, dH2 = (dZ W3^T) * [H2 > 0]
    if (e == cudaSuccess) e = gemm_xtg(m, W, O, Q, m->H2, m->dZ, g + m->off[4], g + m->off[5], st);
    if (e == cudaSuccess) e = gemm_gwt(m, Q, W, O, m->dZ, Wh(m, 2), Epilogue{m->dH2, W, nullptr, 0, m->H2, W}, st);
    // layer 2
    if (e == cudaSuccess) e = gemm_xtg(m, W, W, Q, m->H1, m->dH2, g + m->off[2], g + m->off[3], st);
    if (e == cudaSuccess) e = gemm_gwt(m, Q, W, W, m->dH2, Wh(m, 1), Epilogue{m->dH1, W, nullptr, 0, m->H1, W}, st);
    // layer 1
    if (e == cudaSuccess) e = gemm_xtg(m, D, W, Q, X, m->dH1, g + m->off[0], g + m->off[1], st);
    if (e == cudaSuccess && loss) {
        sum_kernel<<<1, 256, 0, st>>>(Q, m->row_loss, loss);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return cuda_fail(e, "network backward");
    return KPS_OK;
}

kps_status check_rows(const kps_mlp *m, const void *X, int Q) {
    if (!m) return fail(KPS_EINVAL, "network is NULL");
    if (Q < 0) return fail(KPS_EINVAL, "rows must be >= 0");
    if (Q > 0 && !X) return fail(KPS_EINVAL, "input is NULL");
    if ((long long)Q > 65535LL * kBM) return fail(KPS_ENOTSUP, "too many rows in one call (split the batch)");
    return KPS_OK;
}

}  // namespace

extern "C" {

kps_status kps_mlp_create(int32_t din, int32_t width, int32_t dout, uint64_t seed, kps_mlp **out) {
    if (!out) return fail(KPS_EINVAL, "out is NULL");
    *out = nullptr;
    if (din < 1 || width < 1 || dout < 1 || dout > 32) return fail(KPS_EINVAL, "bad layer sizes (dout <= 32)");
    kps_mlp *m = new (std::nothrow) kps_mlp;
    if (!m) return fail(KPS_ENOMEM, "network object");
    m->din = din;
    m->width = width;
    m->dout = dout;
    const long long sz[6] = {(long long)din * width, width, (long long)width * width, width, (long long)width * dout,
                             dout};
    for (int i = 0; i < 6; ++i) m->off[i + 1] = m->off[i] + sz[i];
    const long long n = m->off[6];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&m->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        m->sms = 1;
    // He initialisation (normal, std sqrt(2 / fan_in)), zero biases
    std::vector<float> host(n, 0.f);
    std::mt19937_64 rng(seed);
    const int fan[3] = {din, width, width};
    for (int l = 0; l < 3; ++l) {
        std::normal_distribution<float> nd(0.f, std::sqrt(2.f / fan[l]));
        for (long long i = m->off[2 * l]; i < m->off[2 * l + 1]; ++i) host[i] = nd(rng);
    }
    cudaError_t e = kps::device_malloc(&m->p, n * 4);
    if (e == cudaSuccess) e = kps::device_malloc(&m->g, n * 4);
    if (e == cudaSuccess) e = kps::device_malloc(&m->m, n * 4);
    if (e == cudaSuccess) e = kps::device_malloc(&m->v, n * 4);
    if (e == cudaSuccess) e = kps::device_malloc(&m->ph, n * 2);
    if (e == cudaSuccess) e = kps::device_malloc(&m->wsum, 4);
    if (e != cudaSuccess) {
        kps_mlp_destroy(m);
        return fail(KPS_ENOMEM, "network parameters");
    }
    e = cudaMemcpy(m->p, host.data(), n * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(m->m, 0, n * 4);
    if (e == cudaSuccess) e = cudaMemset(m->v, 0, n * 4);
    if (e == cudaSuccess) e = cudaMemset(m->g, 0, n * 4);
    if (e == cudaSuccess) {
        to_bf16_kernel<<<(unsigned)((n + 255) / 256), 256>>>(n, m->p, m->ph);
        e = cudaDeviceSynchronize();
    }
    if (e != cudaSuccess) {
        kps_mlp_destroy(m);
        return cuda_fail(e, "initialising the network");
    }
    *out = m;
    return KPS_OK;
}

kps_status kps_mlp_destroy(kps_mlp *m) {
    if (!m) return KPS_OK;
    for (void *q : {(void *)m->p, (void *)m->g, (void *)m->m, (void *)m->v, (void *)m->ph, (void *)m->wsum,
                    (void *)m->H1, (void *)m->H2, (void *)m->Z, (void *)m->dZ, (void *)m->dH1, (void *)m->dH2,
                    (void *)m->row_loss, (void *)m->part})
        if (q) cudaFree(q);
    delete m;
    return KPS_OK;
}

kps_status kps_mlp_num_params(const kps_mlp *m, int64_t *n) {
    if (!m || !n) return fail(KPS_EINVAL, "bad argument");
    *n = m->off[6];
    return KPS_OK;
}

kps_status kps_mlp_get(const kps_mlp *m, int32_t which, float *host) {
    if (!m || !host || which < 0 || which > 1) return fail(KPS_EINVAL, "bad argument");
    cudaError_t e = cudaMemcpy(host, which == 0 ? m->p : m->g, m->off[6] * 4, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_fail(e, "reading the network");
    return KPS_OK;
}

kps_status kps_mlp_set(kps_mlp *m, const float *host) {
    if (!m || !host) return fail(KPS_EINVAL, "bad argument");
    cudaError_t e = cudaMemcpy(m->p, host, m->off[6] * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        to_bf16_kernel<<<(unsigned)((m->off[6] + 255) / 256), 256>>>(m->off[6], m->p, m->ph);
        e = cudaDeviceSynchronize();
    }
    if (e != cudaSuccess) return cuda_fail(e, "writing the network");
    return KPS_OK;
}

// Checkpoint of a network (kps_mlp_save / kps_mlp_load): this header, then
// the FP32 parameters and Adam's first and second moments.
struct MlpCkpt {
    char magic[8];
    int32_t version, din, width, dout;
    int64_t step, n;
};
static const char kMlpMagic[8] = {'K', 'P', 'S', 'M', 'L', 'P', '0', '1'};

kps_status kps_mlp_state_bytes(const kps_mlp *m, int64_t *bytes) {
    if (!m || !bytes) return fail(KPS_EINVAL, "NULL argument");
    *bytes = (int64_t)sizeof(MlpCkpt) + 3 * 4 * m->off[6];
    return KPS_OK;
}

kps_status kps_mlp_save(const kps_mlp *m, void *host, int64_t bytes) {
    if (!m || !host) return fail(KPS_EINVAL, "NULL argument");
    const long long n = m->off[6];
    if (bytes < (int64_t)sizeof(MlpCkpt) + 12 * n) return fail(KPS_EINVAL, "buffer smaller than kps_mlp_state_bytes");
    MlpCkpt h;
    std::memset(&h, 0, sizeof(h));
    std::memcpy(h.magic, kMlpMagic, 8);
    h.version = 1;
    h.din = m->din;
    h.width = m->width;
    h.dout = m->dout;
    h.step = m->step;
    h.n = n;
    unsigned char *dst = static_cast<unsigned char *>(host);
    std::memcpy(dst, &h, sizeof(h));
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(dst + sizeof(h), m->p, 4 * n, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(dst + sizeof(h) + 4 * n, m->m, 4 * n, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(dst + sizeof(h) + 8 * n, m->v, 4 * n, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_fail(e, "saving the network");
    return KPS_OK;
}

kps_status kps_mlp_load(kps_mlp *m, const void *host, int64_t bytes) {
    if (!m || !host) return fail(KPS_EINVAL, "NULL argument");
    if (bytes < (int64_t)sizeof(MlpCkpt)) return fail(KPS_EINVAL, "buffer too small for a checkpoint");
    MlpCkpt h;
    std::memcpy(&h, host, sizeof(h));
    if (std::memcmp(h.magic, kMlpMagic, 8) != 0 || h.version != 1) return fail(KPS_EINVAL, "not a network checkpoint");
    if (h.din != m->din || h.width != m->width || h.dout != m->dout || h.n != m->off[6])
        return fail(KPS_EINVAL, "checkpoint of a network with other layer sizes");
    const long long n = m->off[6];
    if (bytes < (int64_t)sizeof(MlpCkpt) + 12 * n) return fail(KPS_EINVAL, "checkpoint truncated");
    if (h.step < 0 || h.step > 0x7fffffffLL) return fail(KPS_EINVAL, "bad step count in the checkpoint");
    const unsigned char *src = static_cast<const unsigned char *>(host) + sizeof(h);
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(m->p, src, 4 * n, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(m->m, src + 4 * n, 4 * n, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(m->v, src + 8 * n, 4 * n, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        to_bf16_kernel<<<(unsigned)((n + 255) / 256), 256>>>(n, m->p, m->ph);
        e = cudaDeviceSynchronize();
    }
    if (e != cudaSuccess) return cuda_fail(e, "loading the network");
    m->step = (int)h.step;
    return KPS_OK;
}

kps_status kps_mlp_forward(kps_mlp *m, const float *X, int32_t Q, const int32_t *nact, float *P, void *stream) {
    kps_status st = check_rows(m, X, Q);
    if (st != KPS_OK) return st;
    if (Q == 0) return KPS_OK;
    if (!nact || !P) return fail(KPS_EINVAL, "nact and P are required");
    st = ensure_cap(m, Q);
    if (st != KPS_OK) return st;
    return forward(m, X, Q, nact, P, static_cast<cudaStream_t>(stream));
}

kps_status kps_mlp_gradients(kps_mlp *m, const float *X, int32_t Q, const int32_t *nact, const float *T,
                             const float *w, float wsum, float *loss, void *stream) {
    kps_status st = check_rows(m, X, Q);
    if (st != KPS_OK) return st;
    if (Q == 0) return KPS_OK;
    if (!nact || !T || !w || !(wsum > 0.f)) return fail(KPS_EINVAL, "nact, T, w and wsum > 0 are required");
    st = ensure_cap(m, Q);
    if (st != KPS_OK) return st;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    st = forward(m, X, Q, nact, nullptr, s);
    if (st != KPS_OK) return st;
    return backward(m, X, Q, nact, T, w, 1.f / wsum, loss, s);
}

kps_status kps_mlp_adam(kps_mlp *m, float lr, float beta1, float beta2, float eps, void *stream) {
    if (!m) return fail(KPS_EINVAL, "network is NULL");
    m->step += 1;
    const float c1 = 1.f - std::pow(beta1, (float)m->step), c2 = 1.f - std::pow(beta2, (float)m->step);
    const long long n = m->off[6];
    adam_kernel<<<(unsigned)((n + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        n, m->p, m->g, m->m, m->v, m->ph, lr, beta1, beta2, eps, c1, c2);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "Adam step");
    return KPS_OK;
}

}  // extern "C"
