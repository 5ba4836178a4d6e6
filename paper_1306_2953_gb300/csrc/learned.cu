// Learned preconditioner: training targets, a small 3-D convolutional
// network, its training kernels and its inference inside the eigensolver.
// None of this is in the paper (its preconditioner is the filter of
// Sec. III); the definitions are:
//
//  Target generator: conjugate gradients for exactly n_iter iterations from
//  x = 0 on (-1/2 Lap + sigma) x = r, one system per column, with the
//  operator applied by the H psi kernels of a Hamiltonian built with
//  V = sigma and no projectors.
//
//  Network: y = L3(relu(L2(relu(L1(xhat))))), 3^3 bias-free cross-
//  correlations 1 -> 8 -> 8 -> 1 on the lattice, every layer's output zero
//  off the grid, xhat = r / rms(r) stored in BF16, weights used in BF16
//  (rounded from an FP32 master copy), FP32 accumulation; K r = rms(r) y.
//  Weights: one FP32 array of 2160 values, [8][1][27] | [8][8][27] |
//  [1][8][27], tap t = 9 (a+1) + 3 (b+1) + (c+1) for the offset (a, b, c)
//  along map axes (0, 1, 2).
//
//  Training: tiles of D^3 lattice points (a 16^3 interior plus 3 points of
//  halo) cut around random grid points of (residual, CG solution) pairs;
//  loss = mean squared error over interior grid points; Adam
//  (lr, beta = (0.9, 0.999), eps = 1e-8) on the FP32 master weights.
#include <algorithm>
#include <cuda_bf16.h>

#include <cmath>
#include <cstring>
#include <new>
#include <type_traits>
#include <vector>

#include "device.h"
#include "ham.h"
#include "learned.h"
#include "linalg.h"

namespace rs {

constexpr int NC = 8;                        // hidden channels
constexpr int W1_OFF = 0, W2_OFF = NC * 27, W3_OFF = NC * 27 + NC * NC * 27, W_TOTAL = W3_OFF + NC * 27;
static_assert(W_TOTAL == 2160, "weight layout");

__device__ __forceinline__ float bf16_round(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// ------------------------------------------------------------------- CG ---

// One iteration is four launches: AP = H P, p.Ap, the update of X and R with
// r.r, and the update of P.  Rows are [np][n] (n a power of two, X and B with
// their own leading dimension), LPP lanes to a row and V columns to a lane.  The
// few FP64 units set the time as soon as every thread uses them: a coefficient
// is divided once per CTA and column (once per element took 32 us per update of
// 16 columns of 103 331 points, once per thread 30, so 12.9 and 4.1 for the two updates), and
// sums meet in FP64 only once per warp.  The sums
// of iteration it use slot it & 1 of pap and slot (it + 1) & 1 of rr, which the
// launch before their first use clears.

// An FP64-accurate sum of products: FP32 products split exactly and added as
// an unevaluated pair with error-free additions; FP64 Kahan-compensated.
template <typename T> struct DotSum;
template <> struct DotSum<float> {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float a, float b) {
        const float pr = __fmul_rn(a, b), pe = fmaf(a, b, -pr);
        const float sum = __fadd_rn(hi, pr), bb = __fsub_rn(sum, hi);
        lo = __fadd_rn(lo, __fadd_rn(__fadd_rn(__fsub_rn(hi, __fsub_rn(sum, bb)), __fsub_rn(pr, bb)), pe));
        hi = sum;
    }
    // the sum of this and the lane `o` away, still as a pair
    __device__ __forceinline__ void merge(int o) {
        const float h = __shfl_xor_sync(0xffffffffu, hi, o), l = __shfl_xor_sync(0xffffffffu, lo, o);
        const float sum = __fadd_rn(hi, h), bb = __fsub_rn(sum, hi);
        const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(sum, bb)), __fsub_rn(h, bb));
        lo = __fadd_rn(__fadd_rn(lo, l), err);
        hi = sum;
    }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};
template <> struct DotSum<double> {
    double acc = 0.0, comp = 0.0;
    __device__ __forceinline__ void add(double a, double b) {
        const double v = a * b, y = v - comp, t = acc + y;
        comp = (t - acc) - y;
        acc = t;
    }
    __device__ __forceinline__ void merge(int o) { acc += __shfl_xor_sync(0xffffffffu, acc, o); }
    __device__ __forceinline__ double value() const { return acc; }
};

template <typename T, int V> struct __align__(sizeof(T) * V) Cols { T v[V]; };

constexpr int CG_NT = 256;

// adds the CTA's sums of the lanes' columns to out[0 .. LPP V)
template <typename T, int V, int LPP> __device__ __forceinline__ void cg_reduce(DotSum<T> (&d)[V], double *out) {
    __shared__ double red[CG_NT / 32][LPP * V];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < V; ++i) {
#pragma unroll
        for (int o = 16; o >= LPP; o >>= 1) d[i].merge(o);
        if (lane < LPP) red[warp][lane * V + i] = d[i].value();
    }
    __syncthreads();
    if (threadIdx.x < LPP * V) {
        double t = 0;
#pragma unroll
        for (int w = 0; w < CG_NT / 32; ++w) t += red[w][threadIdx.x];
        atomicAdd(out + threadIdx.x, t);
    }
}

// num / den (0 where den is 0) of the thread's columns
template <typename T, int V, int LPP> __device__ __forceinline__ void cg_ratio(const double *num, const double *den, T (&q)[V]) {
    __shared__ T ratio[LPP * V];
    if (threadIdx.x < LPP * V) {
        const double b = ld_fresh(den + threadIdx.x);
        ratio[threadIdx.x] = b != 0.0 ? (T)(ld_fresh(num + threadIdx.x) / b) : T(0);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < V; ++i) q[i] = ratio[(threadIdx.x % LPP) * V + i];
}

template <typename T, int V, int LPP>
__global__ void __launch_bounds__(CG_NT) k_cg_init(const T *__restrict__ B, int64_t ldb, T *__restrict__ X, int64_t ldx,
                                                   T *__restrict__ R, T *__restrict__ P, int64_t npts, double *rr) {
    const int c = (threadIdx.x % LPP) * V;
    DotSum<T> d[V];
    for (int64_t p = blockIdx.x * (int64_t)(CG_NT / LPP) + threadIdx.x / LPP; p < npts; p += (int64_t)gridDim.x * (CG_NT / LPP)) {
        Cols<T, V> b;
#pragma unroll
        for (int i = 0; i < V; ++i) {
            b.v[i] = B[p * ldb + c + i];
            X[p * ldx + c + i] = 0;
            d[i].add(b.v[i], b.v[i]);
        }
        *reinterpret_cast<Cols<T, V> *>(R + p * (LPP * V) + c) = b;
        *reinterpret_cast<Cols<T, V> *>(P + p * (LPP * V) + c) = b;
    }
    cg_reduce<T, V, LPP>(d, rr);
}

// pap += P.AP; clears rrn
template <typename T, int V, int LPP>
__global__ void __launch_bounds__(CG_NT) k_cg_pap(const T *__restrict__ P, const T *__restrict__ AP, int64_t npts, double *pap,
                                                  double *rrn) {
    const int c = (threadIdx.x % LPP) * V;
    pdl_wait();
    pdl_launch();
    if (blockIdx.x == 0 && threadIdx.x < LPP * V) rrn[threadIdx.x] = 0.0;
    DotSum<T> d[V];
#pragma unroll 2
    for (int64_t p = blockIdx.x * (int64_t)(CG_NT / LPP) + threadIdx.x / LPP; p < npts; p += (int64_t)gridDim.x * (CG_NT / LPP)) {
        const Cols<T, V> x = ld_fresh(reinterpret_cast<const Cols<T, V> *>(P + p * (LPP * V) + c));
        const Cols<T, V> y = ld_fresh(reinterpret_cast<const Cols<T, V> *>(AP + p * (LPP * V) + c));
#pragma unroll
        for (int i = 0; i < V; ++i) d[i].add(x.v[i], y.v[i]);
    }
    cg_reduce<T, V, LPP>(d, pap);
}

// X += alpha P, R -= alpha AP with alpha = rr / pap per column; rrn += R.R; clears papn
template <typename T, int V, int LPP>
__global__ void __launch_bounds__(CG_NT) k_cg_update1(T *__restrict__ X, int64_t ldx, int xvec, T *__restrict__ R,
                                                      const T *__restrict__ P, const T *__restrict__ AP, int64_t npts,
                                                      const double *__restrict__ rr, const double *__restrict__ pap, double *rrn,
                                                      double *papn) {
    using C = Cols<T, V>;
    const int c = (threadIdx.x % LPP) * V;
    pdl_wait();
    pdl_launch();
    if (blockIdx.x == 0 && threadIdx.x < LPP * V) papn[threadIdx.x] = 0.0;
    T a[V];
    cg_ratio<T, V, LPP>(rr, pap, a);
    DotSum<T> d[V];
    for (int64_t p = blockIdx.x * (int64_t)(CG_NT / LPP) + threadIdx.x / LPP; p < npts; p += (int64_t)gridDim.x * (CG_NT / LPP)) {
        const C pv = ld_fresh(reinterpret_cast<const C *>(P + p * (LPP * V) + c));
        const C ap = ld_fresh(reinterpret_cast<const C *>(AP + p * (LPP * V) + c));
        C r = *reinterpret_cast<const C *>(R + p * (LPP * V) + c), x;
        T *xp = X + p * ldx + c;
        if (xvec) x = *reinterpret_cast<const C *>(xp);
        else {
#pragma unroll
            for (int i = 0; i < V; ++i) x.v[i] = xp[i];
        }
#pragma unroll
        for (int i = 0; i < V; ++i) {
            x.v[i] += a[i] * pv.v[i];
            r.v[i] -= a[i] * ap.v[i];
            d[i].add(r.v[i], r.v[i]);
        }
        if (xvec) *reinterpret_cast<C *>(xp) = x;
        else {
#pragma unroll
            for (int i = 0; i < V; ++i) xp[i] = x.v[i];
        }
        *reinterpret_cast<C *>(R + p * (LPP * V) + c) = r;
    }
    cg_reduce<T, V, LPP>(d, rrn);
}

// P = R + beta P with beta = rrn / rr per column
template <typename T, int V, int LPP>
__global__ void __launch_bounds__(CG_NT) k_cg_update2(const T *__restrict__ R, T *__restrict__ P, int64_t npts,
                                                      const double *__restrict__ rr, const double *__restrict__ rrn) {
    using C = Cols<T, V>;
    const int c = (threadIdx.x % LPP) * V;
    T b[V];
    pdl_wait();
    pdl_launch();
    cg_ratio<T, V, LPP>(rrn, rr, b);
#pragma unroll 2
    for (int64_t p = blockIdx.x * (int64_t)(CG_NT / LPP) + threadIdx.x / LPP; p < npts; p += (int64_t)gridDim.x * (CG_NT / LPP)) {
        const C r = ld_fresh(reinterpret_cast<const C *>(R + p * (LPP * V) + c));
        C q = *reinterpret_cast<const C *>(P + p * (LPP * V) + c);
#pragma unroll
        for (int i = 0; i < V; ++i) q.v[i] = r.v[i] + b[i] * q.v[i];
        *reinterpret_cast<C *>(P + p * (LPP * V) + c) = q;
    }
}

int64_t cg_workspace_bytes(int64_t npts, int ncols, int dtype) {
    const int es = dtype == RS_F64 ? 8 : 4;
    return 3 * npts * ncols * es + 4 * 64 * 8 + 256;
}

template <typename T, int V, int LPP>
static int cg_t(rs_ham *h, const T *B, int64_t ldb, T *X, int64_t ldx, int n_iter, void *work, cudaStream_t st) {
    constexpr int n = V * LPP;
    const int64_t np = ham_npts(h);
    T *R = reinterpret_cast<T *>(work);
    T *P = R + np * n;
    T *AP = P + np * n;
    // the sums, 8-byte aligned behind the arrays
    double *rr = reinterpret_cast<double *>(((uintptr_t)(AP + np * n) + 7) & ~(uintptr_t)7), *pap = rr + 128;   // two slots of 64 each
    const int dt = sizeof(T) == 8 ? RS_F64 : RS_F32;
    // Every CTA adds its sums to the same n numbers, one after another, so few
    // CTAs a SM (103 331 points, 200 iterations, FP32 16 columns: 5.7 ms with two,
    // 6.6 with three, 7.6 with six); rows of 32 columns need the loads in flight
    // (10.2 with two, 9.8 with six).
    const unsigned blocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>((np + CG_NT / LPP - 1) / (CG_NT / LPP), 152 * (n >= 32 ? 6 : 2)));
    const int xvec = aligned16(X) && (ldx * sizeof(T)) % 16 == 0;
    RS_CUDA(cudaMemsetAsync(rr, 0, sizeof(double) * 256, st));
    k_cg_init<T, V, LPP><<<blocks, CG_NT, 0, st>>>(B, ldb, X, ldx, R, P, np, rr);
    RS_LAUNCH_CHECK();
    for (int it = 0; it < n_iter; ++it) {
        double *r0 = rr + 64 * (it & 1), *r1 = rr + 64 * (~it & 1), *p0 = pap + 64 * (it & 1), *p1 = pap + 64 * (~it & 1);
        RS_TRY(rs_ham_apply_block(h, P, n, AP, n, n, dt, st));
        RS_TRY(launch_overlapped(k_cg_pap<T, V, LPP>, blocks, CG_NT, 0, st, P, AP, np, p0, r1));
        RS_TRY(launch_overlapped(k_cg_update1<T, V, LPP>, blocks, CG_NT, 0, st, X, ldx, xvec, R, P, AP, np, r0, p0, r1, p1));
        RS_TRY(launch_overlapped(k_cg_update2<T, V, LPP>, blocks, CG_NT, 0, st, R, P, np, r0, r1));
    }
    return RS_OK;
}

template <typename T>
static int cg_n(rs_ham *h, const T *B, int64_t ldb, T *X, int64_t ldx, int n, int n_iter, void *work, cudaStream_t st) {
    constexpr int E = 16 / (int)sizeof(T);   // columns per 16 bytes
    switch (n) {
        case 1: return cg_t<T, 1, 1>(h, B, ldb, X, ldx, n_iter, work, st);
        case 2: return cg_t<T, 2, 1>(h, B, ldb, X, ldx, n_iter, work, st);
        case 4: return cg_t<T, E, 4 / E>(h, B, ldb, X, ldx, n_iter, work, st);
        case 8: return cg_t<T, E, 8 / E>(h, B, ldb, X, ldx, n_iter, work, st);
        case 16: return cg_t<T, E, 16 / E>(h, B, ldb, X, ldx, n_iter, work, st);
        case 32: return cg_t<T, E, 32 / E>(h, B, ldb, X, ldx, n_iter, work, st);
        case 64: return cg_t<T, E, 64 / E>(h, B, ldb, X, ldx, n_iter, work, st);
        default: return fail(RS_EINVAL, "shifted Poisson CG: the column count must be a power of two <= 64");
    }
}

int shifted_poisson_cg(rs_ham *h, const void *B, int64_t ldb, void *X, int64_t ldx, int n, int n_iter, int dtype,
                       void *work, cudaStream_t st) {
    if (dtype == RS_F64)
        return cg_n<double>(h, (const double *)B, ldb, (double *)X, ldx, n, n_iter, work, st);
    return cg_n<float>(h, (const float *)B, ldb, (float *)X, ldx, n, n_iter, work, st);
}

// ------------------------------------------------ network on dense tiles ---
// Activations [tile][C][D^3], point index p = (i D + j) D + k.

__device__ __forceinline__ int tap_offset(int t, int D) {
    const int a = t / 9 - 1, b = (t / 3) % 3 - 1, c = t % 3 - 1;
    return (a * D + b) * D + c;
}
__device__ __forceinline__ bool tap_inside(int t, int i, int j, int k, int D) {
    const int a = i + t / 9 - 1, b = j + (t / 3) % 3 - 1, c = k + t % 3 - 1;
    return (unsigned)a < (unsigned)D && (unsigned)b < (unsigned)D && (unsigned)c < (unsigned)D;
}

// z = conv(in), a = relu(z) * mask (or a = z * mask when relu == false)
template <int CIN, int COUT>
__global__ void k_tile_fwd(const float *__restrict__ in, const float *__restrict__ wq, const uint8_t *__restrict__ mask,
                           int ntiles, int D, float *__restrict__ z, float *__restrict__ a, bool relu) {
    __shared__ float w[COUT * CIN * 27];
    for (int e = threadIdx.x; e < COUT * CIN * 27; e += blockDim.x) w[e] = wq[e];
    __syncthreads();
    const int D3 = D * D * D;
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= (int64_t)ntiles * D3) return;
    const int tile = (int)(g / D3), p = (int)(g % D3);
    const int i = p / (D * D), j = (p / D) % D, k = p % D;
    float acc[COUT];
#pragma unroll
    for (int co = 0; co < COUT; ++co) acc[co] = 0.f;
    const float *src = in + (int64_t)tile * CIN * D3;
    for (int t = 0; t < 27; ++t) {
        if (!tap_inside(t, i, j, k, D)) continue;
        const int q = p + tap_offset(t, D);
#pragma unroll
        for (int ci = 0; ci < CIN; ++ci) {
            const float x = src[(int64_t)ci * D3 + q];
#pragma unroll
            for (int co = 0; co < COUT; ++co) acc[co] = fmaf(w[(co * CIN + ci) * 27 + t], x, acc[co]);
        }
    }
    const float m = mask[(int64_t)tile * D3 + p] ? 1.f : 0.f;
#pragma unroll
    for (int co = 0; co < COUT; ++co) {
        const int64_t o = ((int64_t)tile * COUT + co) * D3 + p;
        if (z) z[o] = acc[co];
        a[o] = (relu ? fmaxf(acc[co], 0.f) : acc[co]) * m;
    }
}

// gin[ci][q] = sum_co sum_t w[co][ci][t] gout[co][q - off_t]
template <int CIN, int COUT>
__global__ void k_tile_bwd_data(const float *__restrict__ gout, const float *__restrict__ wq, int ntiles, int D,
                                float *__restrict__ gin) {
    __shared__ float w[COUT * CIN * 27];
    for (int e = threadIdx.x; e < COUT * CIN * 27; e += blockDim.x) w[e] = wq[e];
    __syncthreads();
    const int D3 = D * D * D;
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= (int64_t)ntiles * D3) return;
    const int tile = (int)(g / D3), q = (int)(g % D3);
    const int i = q / (D * D), j = (q / D) % D, k = q % D;
    float acc[CIN];
#pragma unroll
    for (int ci = 0; ci < CIN; ++ci) acc[ci] = 0.f;
    const float *src = gout + (int64_t)tile * COUT * D3;
    for (int t = 0; t < 27; ++t) {
        // output point p = q - off_t exists when the mirrored tap is inside
        if (!tap_inside(26 - t, i, j, k, D)) continue;
        const int p = q - tap_offset(t, D);
#pragma unroll
        for (int co = 0; co < COUT; ++co) {
            const float gv = src[(int64_t)co * D3 + p];
#pragma unroll
            for (int ci = 0; ci < CIN; ++ci) acc[ci] = fmaf(w[(co * CIN + ci) * 27 + t], gv, acc[ci]);
        }
    }
#pragma unroll
    for (int ci = 0; ci < CIN; ++ci) gin[((int64_t)tile * CIN + ci) * D3 + q] = acc[ci];
}

// dW[co][ci][t] += sum over the tile points p (with p + d_t inside the tile)
// of gout[co][p] * in[ci][p + d_t].  CTA (tile, slab of WB_PLANES planes):
// the slab of gout and the slab plus one plane on either side of `in` are
// staged in shared memory; thread (ci, t) keeps COUT accumulators.
constexpr int WB_PLANES = 2;
template <int CIN, int COUT>
__global__ void k_tile_bwd_weight(const float *__restrict__ gout, const float *__restrict__ in, int ntiles, int D,
                                  float *__restrict__ dW) {
    extern __shared__ float wsm[];
    const int D2 = D * D, D3 = D2 * D;
    const int tile = blockIdx.x, i0 = blockIdx.y * WB_PLANES;
    const int np = min(WB_PLANES, D - i0);
    float *gs = wsm;                               // [COUT][np][D2]
    float *as = wsm + COUT * WB_PLANES * D2;       // [CIN][np + 2][D2], plane i0 - 1 first
    for (int e = threadIdx.x; e < COUT * np * D2; e += blockDim.x) {
        const int co = e / (np * D2), r = e - co * np * D2;
        gs[co * WB_PLANES * D2 + r] = gout[((int64_t)tile * COUT + co) * D3 + (int64_t)i0 * D2 + r];
    }
    for (int e = threadIdx.x; e < CIN * (np + 2) * D2; e += blockDim.x) {
        const int ci = e / ((np + 2) * D2), r = e - ci * (np + 2) * D2;
        const int pl = i0 - 1 + r / D2;
        as[ci * (WB_PLANES + 2) * D2 + r] =
            (pl >= 0 && pl < D) ? in[((int64_t)tile * CIN + ci) * D3 + (int64_t)pl * D2 + r % D2] : 0.f;
    }
    __syncthreads();
    const int w = threadIdx.x;
    if (w >= CIN * 27) return;
    const int ci = w / 27, t = w - ci * 27;
    const int di = t / 9 - 1, dj = (t / 3) % 3 - 1, dk = t % 3 - 1;
    float acc[COUT];
#pragma unroll
    for (int co = 0; co < COUT; ++co) acc[co] = 0.f;
    const float *ab = as + ci * (WB_PLANES + 2) * D2;
    for (int pl = 0; pl < np; ++pl) {
        if ((unsigned)(i0 + pl + di) >= (unsigned)D) continue;   // zero padding outside the tile
        for (int j = max(0, -dj); j < min(D, D - dj); ++j) {
            const float *arow = ab + (pl + 1 + di) * D2 + (j + dj) * D + dk;
            const int gofs = pl * D2 + j * D;
            for (int k = max(0, -dk); k < min(D, D - dk); ++k) {
                const float x = arow[k];
#pragma unroll
                for (int co = 0; co < COUT; ++co) acc[co] = fmaf(gs[co * WB_PLANES * D2 + gofs + k], x, acc[co]);
            }
        }
    }
#pragma unroll
    for (int co = 0; co < COUT; ++co) atomicAdd(dW + (co * CIN + ci) * 27 + t, acc[co]);
}

template <int CIN, int COUT> int tile_bwd_weight(const float *gout, const float *in, int ntiles, int D, float *dW,
                                                 cudaStream_t st) {
    const size_t sm = sizeof(float) * (size_t)(COUT * WB_PLANES + CIN * (WB_PLANES + 2)) * D * D;
    if (sm > 200 * 1024) return fail(RS_EINVAL, "tile_bwd_weight: tile too large");
    RS_TRY(smem_optin((const void *)k_tile_bwd_weight<CIN, COUT>, sm));
    const int threads = ((CIN * 27 + 31) / 32) * 32;
    k_tile_bwd_weight<CIN, COUT><<<dim3((unsigned)ntiles, (unsigned)((D + WB_PLANES - 1) / WB_PLANES)), threads, sm, st>>>(
        gout, in, ntiles, D, dW);
    RS_LAUNCH_CHECK();
    return RS_OK;
}

// count[n] = valid grid points of tile n (one CTA per tile)
__global__ void k_tile_count(const uint8_t *__restrict__ mask, const uint8_t *__restrict__ valid, int D3, int *__restrict__ count) {
    const uint8_t *m = mask + (int64_t)blockIdx.x * D3;
    int c = 0;
    for (int e = threadIdx.x; e < D3; e += blockDim.x) c += valid[e] && m[e];
    c = __reduce_add_sync(0xffffffffu, c);
    __shared__ int red[32];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x < 32) {
        c = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0;
        c = __reduce_add_sync(0xffffffffu, c);
        if (threadIdx.x == 0) count[blockIdx.x] = c;
    }
}

// g = d loss / d y with loss = sum_{valid} (y - t)^2 / nvalid; returns the sum in loss[0]
__global__ void k_tile_loss(const float *__restrict__ y, const float *__restrict__ tgt, const uint8_t *__restrict__ mask,
                            const uint8_t *__restrict__ valid, int ntiles, int D, double inv_n, float *__restrict__ gy,
                            double *loss) {
    __shared__ double red[256];
    const int D3 = D * D * D;
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    double l = 0.0;
    if (g < (int64_t)ntiles * D3) {
        const int p = (int)(g % D3);
        const bool v = valid[p] && mask[g];
        const float d = v ? y[g] - tgt[g] : 0.f;
        gy[g] = (float)(2.0 * inv_n) * d;
        l = (double)d * d * inv_n;
    }
    red[threadIdx.x] = l;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(loss, red[0]);
}

// g *= mask * (z > 0) (relu derivative; the mask is folded in)
__global__ void k_relu_grad(float *g, const float *z, const uint8_t *mask, int ntiles, int C, int D) {
    const int D3 = D * D * D;
    const int64_t n = (int64_t)ntiles * C * D3;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t tile = e / ((int64_t)C * D3);
        const int p = (int)(e % D3);
        if (!(mask[tile * D3 + p] && z[e] > 0.f)) g[e] = 0.f;
    }
}

__global__ void k_mask_grad(float *g, const uint8_t *mask, int64_t n) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
        if (!mask[e]) g[e] = 0.f;
}

__global__ void k_round_weights(const float *w, float *wq, int n) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) wq[e] = bf16_round(w[e]);
}

__global__ void k_round_inputs(const float *x, float *xq, int64_t n) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
        xq[e] = bf16_round(x[e]);
}

__global__ void k_adam(float *w, const float *g, float *m, float *v, int n, float lr, float b1, float b2, float eps,
                       int step) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const float gg = g[e];
    const float mm = b1 * m[e] + (1.f - b1) * gg;
    const float vv = b2 * v[e] + (1.f - b2) * gg * gg;
    m[e] = mm;
    v[e] = vv;
    const float mh = mm / (1.f - powf(b1, (float)step));
    const float vh = vv / (1.f - powf(b2, (float)step));
    w[e] -= lr * mh / (sqrtf(vh) + eps);
}

// Network forward + backward on a batch of dense tiles; activations in `ws`.
struct TileBufs {
    float *x0, *z1, *a1, *z2, *a2, *y, *g3, *ga2, *ga1, *wq;
    static size_t floats(int ntiles, int D) {
        const size_t v = (size_t)ntiles * D * D * D;
        return v * (1 + NC * 4 + 1 + 1 + NC * 2) + W_TOTAL + 64;
    }
    TileBufs(float *base, int ntiles, int D) {
        const size_t v = (size_t)ntiles * D * D * D;
        x0 = base;
        z1 = x0 + v;
        a1 = z1 + NC * v;
        z2 = a1 + NC * v;
        a2 = z2 + NC * v;
        y = a2 + NC * v;
        g3 = y + v;
        ga2 = g3 + v;
        ga1 = ga2 + NC * v;
        wq = ga1 + NC * v;
    }
};

int tile_forward(const float *wq, const float *x0, const uint8_t *mask, int ntiles, int D, TileBufs &b, cudaStream_t st) {
    const int64_t n = (int64_t)ntiles * D * D * D;
    const unsigned blocks = (unsigned)((n + 127) / 128);
    k_tile_fwd<1, NC><<<blocks, 128, 0, st>>>(x0, wq + W1_OFF, mask, ntiles, D, b.z1, b.a1, true);
    k_tile_fwd<NC, NC><<<blocks, 128, 0, st>>>(b.a1, wq + W2_OFF, mask, ntiles, D, b.z2, b.a2, true);
    k_tile_fwd<NC, 1><<<blocks, 128, 0, st>>>(b.a2, wq + W3_OFF, mask, ntiles, D, nullptr, b.y, false);
    RS_LAUNCH_CHECK();
    return RS_OK;
}

// grad (2160 floats) must be zeroed by the caller; g3 holds d loss / d y.
int tile_backward(const float *wq, const float *x0, const uint8_t *mask, int ntiles, int D, TileBufs &b, float *grad,
                  cudaStream_t st) {
    const int64_t n = (int64_t)ntiles * D * D * D;
    const unsigned blocks = (unsigned)((n + 127) / 128);

    k_mask_grad<<<1024, 256, 0, st>>>(b.g3, mask, n);
    RS_TRY((tile_bwd_weight<NC, 1>(b.g3, b.a2, ntiles, D, grad + W3_OFF, st)));
    k_tile_bwd_data<NC, 1><<<blocks, 128, 0, st>>>(b.g3, wq + W3_OFF, ntiles, D, b.ga2);
    k_relu_grad<<<1024, 256, 0, st>>>(b.ga2, b.z2, mask, ntiles, NC, D);
    RS_TRY((tile_bwd_weight<NC, NC>(b.ga2, b.a1, ntiles, D, grad + W2_OFF, st)));
    k_tile_bwd_data<NC, NC><<<blocks, 128, 0, st>>>(b.ga2, wq + W2_OFF, ntiles, D, b.ga1);
    k_relu_grad<<<1024, 256, 0, st>>>(b.ga1, b.z1, mask, ntiles, NC, D);
    RS_TRY((tile_bwd_weight<1, NC>(b.ga1, x0, ntiles, D, grad + W1_OFF, st)));
    RS_LAUNCH_CHECK();
    return RS_OK;
}

// ------------------------------------------------------ tile extraction ---
// For tile n: column col[n], interior origin (bbox-local) o[n] (a 16^3 box
// starting 3 points inside the D^3 tile).  x = r / rms, t = xcg / rms,
// mask = grid membership.
__global__ void k_cut_tiles(const int32_t *__restrict__ map, int d0, int d1, int d2, const float *__restrict__ R,
                            const float *__restrict__ X, int64_t ld, const double *__restrict__ rms,
                            const int4 *__restrict__ org, int ntiles, int D, float *__restrict__ xin,
                            float *__restrict__ tgt, uint8_t *__restrict__ mask) {
    const int D3 = D * D * D;
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= (int64_t)ntiles * D3) return;
    const int n = (int)(g / D3), p = (int)(g % D3);
    const int4 o = org[n];
    const int a = o.y + p / (D * D), b = o.z + (p / D) % D, c = o.w + p % D;
    int r = -1;
    if ((unsigned)a < (unsigned)d0 && (unsigned)b < (unsigned)d1 && (unsigned)c < (unsigned)d2)
        r = map[((int64_t)a * d1 + b) * d2 + c];
    const float s = (float)(1.0 / rms[o.x]);
    xin[g] = r >= 0 ? bf16_round(R[(int64_t)r * ld + o.x] * s) : 0.f;
    tgt[g] = r >= 0 ? X[(int64_t)r * ld + o.x] * s : 0.f;
    mask[g] = r >= 0;
}

__global__ void k_rms(const double *ss, int n, double inv_np, double *rms) {
    const int k = threadIdx.x;
    if (k < n) rms[k] = ss[k] > 0 ? sqrt(ss[k] * inv_np) : 1.0;
}

// --------------------------------------------- inference on the grid ---

// The three layers work on rows of four lattice positions along map axis 2
// (row items: 4-aligned positions), so that an activation read once serves the
// three outputs it touches in its row: 54 reads for four points instead of
// 108.  A CTA takes ITEMS consecutive items (16, or 64 of up
// to 8 columns, which would leave the CTA little work otherwise) and stages the point indices of
// their 3 x 3 x 6 neighbourhoods in shared memory; items without a grid point
// are skipped.  Measured on 654 520 points and 32 states (one thread per point
// and state and FP32 FMA before): input and layer 1 910 -> 497 us, layer 2
// 2709 -> 1295 us, layer 3 1203 -> 652 us; they wait for loads (issue active
// 46 % in layer 2, its tensor pipe 37 %).
constexpr int ROWN = 4, ROWP = ROWN + 2, NBH = 9 * ROWP;
constexpr int NET_NT = 256;

struct NetGrid {
    const int32_t *map;
    int d1, d2, n4, items;   // n4: row items per map row
    int nb;
};

// Indices of item `it` (of the CTA): qs[it][row][i], row = 3 (a + 1) + (b + 1),
// i = 0 .. 5 the positions from one before the item to one behind it; the
// item's own points are qs[it][4][1 .. 4].  False when no item has a point.
template <int ITEMS> __device__ __forceinline__ bool net_stage(const NetGrid &g, int (&qs)[ITEMS][NBH]) {
    const int t0 = blockIdx.x * ITEMS;
    bool any = false;
    for (int e = threadIdx.x; e < ITEMS * ROWN; e += NET_NT) {
        const int t = t0 + e / ROWN, o = e % ROWN;
        if (t < g.items) {
            const int r = t / g.n4, w = (t - r * g.n4) * ROWN + o;
            any = any || (w < g.d2 && __ldg(g.map + (int64_t)r * g.d2 + w) >= 0);
        }
    }
    if (!__syncthreads_or(any)) return false;
    for (int e = threadIdx.x; e < ITEMS * NBH; e += NET_NT) {
        const int it = e / NBH, k = e - it * NBH, row = k / ROWP, i = k - row * ROWP;
        const int t = t0 + it;
        int q = -1;
        if (t < g.items) {
            const int r = t / g.n4, w = (t - r * g.n4) * ROWN + i - 1;
            // (items with points lie at least four positions inside the map)
            const int64_t L = ((int64_t)r + (row / 3 - 1) * g.d1 + (row % 3 - 1)) * g.d2 + w;
            if (w >= 0 && w < g.d2 && L >= 0 && L < (int64_t)g.items / g.n4 * g.d2) q = __ldg(g.map + L);
        }
        qs[it][k] = q;
    }
    __syncthreads();
    return true;
}
__device__ __forceinline__ bool item_empty(const int (&q)[NBH]) {
    return (q[4 * ROWP + 1] & q[4 * ROWP + 2] & q[4 * ROWP + 3] & q[4 * ROWP + 4]) < 0;
}

// An FP32 value cut exactly into three BF16 pieces of 8 bits; two values to a
// word, the first in the low half.  An infinity is its first piece alone (what is left of it
// would be a NaN, which the next layer's relu turns into 0).
__device__ __forceinline__ void bf16_cut(float x, float y, uint32_t (&p)[3]) {
    auto rest = [](float v, int k) {
        const float r = v - __uint_as_float(__float_as_uint(v) & 0xffff0000u);
        return k > 0 || r == r ? r : 0.f;
    };
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        p[k] = __byte_perm(__float_as_uint(x), __float_as_uint(y), 0x7632);
        x = rest(x, k);
        y = rest(y, k);
    }
}

// Layer 1 (1 -> 8, relu), the input made on the way: xhat = bf16(r / rms).  One
// thread per (item, state).  The result is stored for layer 2's tensor-core
// operands, exactly: three BF16 pieces [point][piece][state][channel].
template <int ITEMS>
__global__ void __launch_bounds__(NET_NT) k_net_first(NetGrid g, const float *__restrict__ wq, const float *__restrict__ R,
                                                      int64_t ldr, const float *__restrict__ scale, uint4 *__restrict__ out) {
    __shared__ __align__(16) float ws[27 * NC];
    __shared__ int qs[ITEMS][NBH];
    for (int e = threadIdx.x; e < 27 * NC; e += NET_NT) ws[e] = __ldg(wq + W1_OFF + (e % NC) * 27 + e / NC);
    if (!net_stage<ITEMS>(g, qs)) return;
    for (int t = threadIdx.x; t < ITEMS * g.nb; t += NET_NT) {
        const int it = t / g.nb, s = t - it * g.nb;
        const int(&q)[NBH] = qs[it];
        if (item_empty(q)) continue;
        const float sc = __ldg(scale + s);
        float2 acc[ROWN][NC / 2];
#pragma unroll
        for (int o = 0; o < ROWN; ++o)
#pragma unroll
            for (int c = 0; c < NC / 2; ++c) acc[o][c] = make_float2(0.f, 0.f);
#pragma unroll 3
        for (int r = 0; r < 9; ++r) {
            float x[ROWP];
#pragma unroll
            for (int i = 0; i < ROWP; ++i) {
                const int n = q[r * ROWP + i];
                x[i] = n >= 0 ? bf16_round(__ldg(R + (int64_t)n * ldr + s) * sc) : 0.f;
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float4 wa = *reinterpret_cast<const float4 *>(ws + (3 * r + c) * NC);
                const float4 wb = *reinterpret_cast<const float4 *>(ws + (3 * r + c) * NC + 4);
                const float2 w[4] = {{wa.x, wa.y}, {wa.z, wa.w}, {wb.x, wb.y}, {wb.z, wb.w}};
#pragma unroll
                for (int o = 0; o < ROWN; ++o)
#pragma unroll
                    for (int k = 0; k < NC / 2; ++k) acc[o][k] = __ffma2_rn(w[k], make_float2(x[o + c], x[o + c]), acc[o][k]);
            }
        }
#pragma unroll
        for (int o = 0; o < ROWN; ++o) {
            const int p = q[4 * ROWP + 1 + o];
            if (p < 0) continue;
            uint32_t pc[4][3];
#pragma unroll
            for (int k = 0; k < 4; ++k) bf16_cut(fmaxf(acc[o][k].x, 0.f), fmaxf(acc[o][k].y, 0.f), pc[k]);
#pragma unroll
            for (int k = 0; k < 3; ++k)
                out[((int64_t)p * 3 + k) * g.nb + s] = make_uint4(pc[0][k], pc[1][k], pc[2][k], pc[3][k]);
        }
    }
}

// Layer 2 (8 -> 8, relu) on the tensor cores: a warp takes 16 (item, state)
// pairs; a tap's 16 x 8 (state, channel) activations meet its 8 x 8 weights,
// two taps of a row in one m16n8k16 and the third in an m16n8k8 (BF16 inputs,
// exact products, FP32 accumulation).  The tensor core truncates where it
// accumulates, so each row of taps starts from zero and is added to the sum
// with rounding: one chain over all taps is three times less exact.
__device__ __forceinline__ void mma_k16(float (&d)[4], const uint32_t (&a)[2], const uint32_t (&b)[2], uint32_t w0, uint32_t w1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(b[0]), "r"(b[1]), "r"(w0), "r"(w1));
}
__device__ __forceinline__ void mma_k8(float (&d)[4], const uint32_t (&a)[2], uint32_t w) {
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};\n"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(w));
}

// The next row's activations are loaded while the products of this one run; the
// weights (output channel gr, input channels 2 tq and 2 tq + 1) wait in shared
// memory, so that two CTAs fit an SM.
// UNI: nb is a multiple of 16, so a tile's rows are one item's.
template <int ITEMS, bool UNI>
__global__ void __launch_bounds__(NET_NT, 2) k_net_mid(NetGrid g, const float *__restrict__ wq, const uint32_t *__restrict__ in,
                                                       float *__restrict__ out) {
    __shared__ int qs[ITEMS][NBH];
    __shared__ uint32_t ws[27][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gr = lane >> 2, tq = lane & 3;
    for (int e = threadIdx.x; e < 27 * 32; e += NET_NT) {
        const int t = e >> 5, l = e & 31;
        const float *w = wq + W2_OFF + ((l >> 2) * NC + 2 * (l & 3)) * 27 + t;
        ws[t][l] = __byte_perm(__float_as_uint(__ldg(w)), __float_as_uint(__ldg(w + 27)), 0x7632);
    }
    if (!net_stage<ITEMS>(g, qs)) return;
    // the 16 rows of a tile: (item, state) pairs, states fastest; this lane's are
    // row gr (a) and gr + 8 (b)
    const int rows = ITEMS * g.nb;
    for (int t = warp; t * 16 < rows; t += NET_NT / 32) {
        const int ra = t * 16 + gr, rb = ra + 8;
        const int ia = UNI ? t * 16 / g.nb : min(ra, rows - 1) / g.nb, ib = UNI ? ia : min(rb, rows - 1) / g.nb;
        const int sa = ra - ia * g.nb, sb = rb - ib * g.nb;
        const int(&qa)[NBH] = qs[ia], (&qb)[NBH] = qs[ib];
        const bool ha = ra < rows && !item_empty(qa), hb = UNI ? ha : rb < rows && !item_empty(qb);
        if (!__any_sync(0xffffffffu, ha || hb)) continue;
        const uint32_t *ina = in + sa * 4 + tq, *inb = in + sb * 4 + tq;
        float acc[ROWN][4];
#pragma unroll
        for (int o = 0; o < ROWN; ++o)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[o][k] = 0.f;
        uint32_t x[2][ROWP][3][2];
        auto load = [&](int r, uint32_t (&y)[ROWP][3][2]) {
#pragma unroll
            for (int i = 0; i < ROWP; ++i) {
                const int na = UNI || ha ? qa[r * ROWP + i] : -1, nb = UNI ? na : hb ? qb[r * ROWP + i] : -1;
                const uint32_t *pa = ina + (int64_t)na * (12 * g.nb), *pb = UNI ? pa + 32 : inb + (int64_t)nb * (12 * g.nb);
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    y[i][k][0] = na >= 0 ? __ldg(pa + k * 4 * g.nb) : 0u;
                    y[i][k][1] = nb >= 0 ? __ldg(pb + k * 4 * g.nb) : 0u;
                }
            }
        };
        load(0, x[0]);
#pragma unroll
        for (int r = 0; r < 9; ++r) {
            if (r < 8) load(r + 1, x[(r + 1) & 1]);
            const uint32_t(&y)[ROWP][3][2] = x[r & 1];
            const uint32_t w0 = ws[3 * r][lane], w1 = ws[3 * r + 1][lane], w2 = ws[3 * r + 2][lane];
            float row[ROWN][4];
#pragma unroll
            for (int o = 0; o < ROWN; ++o)
#pragma unroll
                for (int k = 0; k < 4; ++k) row[o][k] = 0.f;
            // the small pieces first
#pragma unroll
            for (int k = 2; k >= 0; --k)
#pragma unroll
                for (int o = 0; o < ROWN; ++o) {
                    mma_k16(row[o], y[o][k], y[o + 1][k], w0, w1);
                    mma_k8(row[o], y[o + 2][k], w2);
                }
#pragma unroll
            for (int o = 0; o < ROWN; ++o)
#pragma unroll
                for (int k = 0; k < 4; ++k) acc[o][k] += row[o][k];
        }
        // [point][half][state][4 channels]
#pragma unroll
        for (int o = 0; o < ROWN; ++o) {
            const int pa = ha ? qa[4 * ROWP + 1 + o] : -1, pb = hb ? qb[4 * ROWP + 1 + o] : -1;
            float *y = out + 2 * (tq & 1);
            const int64_t half = tq >> 1;
            if (pa >= 0)
                *reinterpret_cast<float2 *>(y + (((int64_t)pa * 2 + half) * g.nb + sa) * 4) =
                    make_float2(fmaxf(acc[o][0], 0.f), fmaxf(acc[o][1], 0.f));
            if (pb >= 0)
                *reinterpret_cast<float2 *>(y + (((int64_t)pb * 2 + half) * g.nb + sb) * 4) =
                    make_float2(fmaxf(acc[o][2], 0.f), fmaxf(acc[o][3], 0.f));
        }
    }
}

// Layer 3 (8 -> 1) times the column's rms; one thread per (item, state), the
// activations [point][half][state][4 channels] (a warp's 16-byte reads are
// contiguous).
template <int ITEMS>
__global__ void __launch_bounds__(NET_NT) k_net_last(NetGrid g, const float *__restrict__ wq, const float *__restrict__ in,
                                                     float *__restrict__ W, int64_t ldw, const double *__restrict__ rms) {
    __shared__ __align__(16) float ws[27 * NC];
    __shared__ int qs[ITEMS][NBH];
    for (int e = threadIdx.x; e < 27 * NC; e += NET_NT) ws[e] = __ldg(wq + W3_OFF + (e % NC) * 27 + e / NC);
    if (!net_stage<ITEMS>(g, qs)) return;
    for (int t = threadIdx.x; t < ITEMS * g.nb; t += NET_NT) {
        const int it = t / g.nb, s = t - it * g.nb;
        const int(&q)[NBH] = qs[it];
        if (item_empty(q)) continue;
        float2 acc[ROWN];   // even and odd channels
#pragma unroll
        for (int o = 0; o < ROWN; ++o) acc[o] = make_float2(0.f, 0.f);
#pragma unroll 1
        for (int r = 0; r < 9; ++r) {
            float4 xa[ROWP], xb[ROWP];
#pragma unroll
            for (int i = 0; i < ROWP; ++i) {
                const int n = q[r * ROWP + i];
                const float4 *src = reinterpret_cast<const float4 *>(in) + (int64_t)n * 2 * g.nb + s;
                xa[i] = n >= 0 ? __ldg(src) : make_float4(0.f, 0.f, 0.f, 0.f);
                xb[i] = n >= 0 ? __ldg(src + g.nb) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float4 wa = *reinterpret_cast<const float4 *>(ws + (3 * r + c) * NC);
                const float4 wb = *reinterpret_cast<const float4 *>(ws + (3 * r + c) * NC + 4);
#pragma unroll
                for (int o = 0; o < ROWN; ++o) {
                    const float4 a = xa[o + c], bb = xb[o + c];
                    acc[o] = __ffma2_rn(make_float2(wa.x, wa.y), make_float2(a.x, a.y), acc[o]);
                    acc[o] = __ffma2_rn(make_float2(wa.z, wa.w), make_float2(a.z, a.w), acc[o]);
                    acc[o] = __ffma2_rn(make_float2(wb.x, wb.y), make_float2(bb.x, bb.y), acc[o]);
                    acc[o] = __ffma2_rn(make_float2(wb.z, wb.w), make_float2(bb.z, bb.w), acc[o]);
                }
            }
        }
        const float f = (float)rms[s];
#pragma unroll
        for (int o = 0; o < ROWN; ++o) {
            const int p = q[4 * ROWP + 1 + o];
            if (p >= 0) W[(int64_t)p * ldw + s] = (acc[o].x + acc[o].y) * f;
        }
    }
}

// ---- few columns and small grids: one thread per point and state, FP32 FMA ----

// xhat = bf16(r / rms) and the per-column rms
__global__ void k_net_input(const float *__restrict__ R, int64_t ldr, const double *__restrict__ rms, int nb,
                            int npts, float *__restrict__ x) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= npts * nb) return;
    const int p = t / nb, s = t - p * nb;
    x[t] = bf16_round(R[(int64_t)p * ldr + s] * (float)(1.0 / rms[s]));
}

// layer on the grid, activations [point][channel][state]: out[p][co][s] = act(sum_t sum_ci w[co][ci][t] in[nbr_t(p)][ci][s]).
// The layer's weights (BF16 values) are staged in shared memory as
// [tap][ci][co], so one 16-byte load gives four output channels' weights
// (a broadcast: every lane reads the same word).
template <int CIN, int COUT, bool RELU, bool FINAL, int WOFF>
__global__ void __launch_bounds__(256) k_net_layer(const int32_t *__restrict__ map, const int32_t *__restrict__ loc,
                                                   int d1, int d2, int npts, int nb, const float *__restrict__ wq,
                                                   const float *__restrict__ in, float *__restrict__ out, int64_t ldo,
                                                   const double *__restrict__ rms) {
    constexpr int CO4 = (COUT + 3) / 4 * 4;
    __shared__ __align__(16) float ws[27 * CIN * CO4];
    for (int e = threadIdx.x; e < 27 * CIN * CO4; e += blockDim.x) {
        const int co = e % CO4, ci = (e / CO4) % CIN, tap = e / (CO4 * CIN);
        ws[e] = co < COUT ? __ldg(wq + WOFF + (co * CIN + ci) * 27 + tap) : 0.f;
    }
    __syncthreads();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= npts * nb) return;
    const int p = t / nb, s = t - p * nb;
    const int64_t L = __ldg(loc + p);
    float acc[CO4];
#pragma unroll
    for (int co = 0; co < CO4; ++co) acc[co] = 0.f;
#pragma unroll 3
    for (int tap = 0; tap < 27; ++tap) {
        const int64_t off = ((int64_t)(tap / 9 - 1) * d1 + ((tap / 3) % 3 - 1)) * d2 + (tap % 3 - 1);
        const int q = __ldg(map + L + off);
        if (q < 0) continue;
        const float *src = in + ((int64_t)q * CIN) * nb + s;
        const float4 *w4 = reinterpret_cast<const float4 *>(ws + tap * CIN * CO4);
#pragma unroll
        for (int ci = 0; ci < CIN; ++ci) {
            const float x = __ldg(src + (int64_t)ci * nb);
#pragma unroll
            for (int c4 = 0; c4 < CO4 / 4; ++c4) {
                const float4 w = w4[ci * (CO4 / 4) + c4];
                acc[4 * c4 + 0] = fmaf(w.x, x, acc[4 * c4 + 0]);
                if (4 * c4 + 1 < COUT) acc[4 * c4 + 1] = fmaf(w.y, x, acc[4 * c4 + 1]);
                if (4 * c4 + 2 < COUT) acc[4 * c4 + 2] = fmaf(w.z, x, acc[4 * c4 + 2]);
                if (4 * c4 + 3 < COUT) acc[4 * c4 + 3] = fmaf(w.w, x, acc[4 * c4 + 3]);
            }
        }
    }
    if (FINAL) {
        out[(int64_t)p * ldo + s] = acc[0] * (float)rms[s];
    } else {
#pragma unroll
        for (int co = 0; co < COUT; ++co) out[((int64_t)p * COUT + co) * nb + s] = RELU ? fmaxf(acc[co], 0.f) : acc[co];
    }
}

// per-column input scale 1 / rms
__global__ void k_net_scale(const double *rms, int nb, float *scale) {
    if ((int)threadIdx.x < nb) scale[threadIdx.x] = (float)(1.0 / rms[threadIdx.x]);
}

}  // namespace rs

using namespace rs;

// ---------------------------------------------------------------- C ABI ---

extern "C" int64_t rs_cg_workspace_bytes(int64_t npts, int ncols, int dtype) {
    if (npts < 1 || ncols < 1 || ncols > 64) return -1;
    return cg_workspace_bytes(npts, ncols, dtype);
}

extern "C" int rs_shifted_poisson_cg(rs_ham *h, const void *B_dev, void *X_dev, int64_t ld, int ncols, int n_iter,
                                     int dtype, void *work_dev, void *stream) {
    if (!h || !B_dev || !X_dev || !work_dev) return fail(RS_EINVAL, "rs_shifted_poisson_cg: null argument");
    if (ncols < 1 || ncols > 64 || (ncols & (ncols - 1))) return fail(RS_EINVAL, "rs_shifted_poisson_cg: ncols must be a power of two <= 64");
    if (ld < ncols || n_iter < 0) return fail(RS_EINVAL, "rs_shifted_poisson_cg: bad ld or n_iter");
    if (dtype != RS_F64 && dtype != RS_F32) return fail(RS_EINVAL, "rs_shifted_poisson_cg: bad dtype");
    // the rows in the workspace are read and written 16 bytes (or a row) at a time,
    // as the H psi kernels need them
    const int es = dtype == RS_F64 ? 8 : 4, need = std::min(ncols * es, 16);
    if ((uintptr_t)work_dev % need) {
        if (n_iter > 0) return fail(RS_EINVAL, "rs_shifted_poisson_cg: misaligned workspace");
        // no iteration, no workspace: X = 0
        RS_CUDA(cudaMemset2DAsync(X_dev, (size_t)ld * es, 0, (size_t)ncols * es, (size_t)ham_npts(h), (cudaStream_t)stream));
        return RS_OK;
    }
    return shifted_poisson_cg(h, B_dev, ld, X_dev, ld, ncols, n_iter, dtype, work_dev, (cudaStream_t)stream);
}

extern "C" int rs_convnet_tiles(const float *w_dev, const float *x_dev, const uint8_t *mask_dev, const float *target_dev,
                                const uint8_t *valid_dev, int ntiles, int D, float *y_dev, float *grad_dev,
                                double *loss_host, void *stream) {
    if (!w_dev || !x_dev || !mask_dev || !y_dev || ntiles < 1 || D < 3)
        return fail(RS_EINVAL, "rs_convnet_tiles: bad arguments");
    if ((grad_dev || loss_host) && (!target_dev || !valid_dev))
        return fail(RS_EINVAL, "rs_convnet_tiles: gradients need target and valid");
    cudaStream_t st = (cudaStream_t)stream;
    PoolBuf ws, dl, cnt;
    RS_TRY(ws.alloc(TileBufs::floats(ntiles, D) * sizeof(float), st));
    RS_TRY(dl.alloc(sizeof(double), st));
    TileBufs b(ws.as<float>(), ntiles, D);
    const int64_t n = (int64_t)ntiles * D * D * D;
    // the number of valid points, counted on the device while the forward pass is queued
    std::vector<int> count(grad_dev || loss_host ? ntiles : 0);
    if (!count.empty()) {
        RS_TRY(cnt.alloc(sizeof(int) * (size_t)ntiles, st));
        k_tile_count<<<(unsigned)ntiles, 256, 0, st>>>(mask_dev, valid_dev, D * D * D, cnt.as<int>());
        RS_CUDA(cudaMemcpyAsync(count.data(), cnt.p, sizeof(int) * (size_t)ntiles, cudaMemcpyDeviceToHost, st));
    }
    k_round_weights<<<9, 256, 0, st>>>(w_dev, b.wq, W_TOTAL);
    k_round_inputs<<<1024, 256, 0, st>>>(x_dev, b.x0, n);
    RS_LAUNCH_CHECK();
    RS_TRY(tile_forward(b.wq, b.x0, mask_dev, ntiles, D, b, st));
    RS_CUDA(cudaMemcpyAsync(y_dev, b.y, sizeof(float) * n, cudaMemcpyDeviceToDevice, st));
    if (grad_dev || loss_host) {
        int64_t nvalid = 0;
        for (int c : count) nvalid += c;   // (the copy to pageable memory has completed)
        RS_CUDA(cudaMemsetAsync(dl.p, 0, sizeof(double), st));
        k_tile_loss<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(b.y, target_dev, mask_dev, valid_dev, ntiles, D,
                                                                1.0 / (double)std::max<int64_t>(nvalid, 1), b.g3, dl.as<double>());
        RS_LAUNCH_CHECK();
        if (grad_dev) {
            RS_CUDA(cudaMemsetAsync(grad_dev, 0, sizeof(float) * W_TOTAL, st));
            RS_TRY(tile_backward(b.wq, b.x0, mask_dev, ntiles, D, b, grad_dev, st));
        }
        if (loss_host) RS_CUDA(cudaMemcpyAsync(loss_host, dl.p, sizeof(double), cudaMemcpyDeviceToHost, st));
    }
    RS_CUDA(cudaStreamSynchronize(st));
    return RS_OK;
}

// splitmix64: the seeded generator of the tile positions
static uint64_t splitmix64(uint64_t &s) {
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

namespace rs {

// Adam on dense tiles already cut: `epochs` passes over the tiles in order,
// one step per batch of `batch` consecutive tiles (a last partial batch is
// dropped), moments zero at the start.  loss_host[ep] (may be NULL) gets the
// mean batch loss of epoch ep.  Blocking.
int train_tiles_impl(float *w_dev, const float *xin, const float *tgt, const uint8_t *msk, const uint8_t *dvalid,
                     int ntiles, int D, int batch, int epochs, float lr, float *loss_host, cudaStream_t st) {
    const int D3 = D * D * D;
    const int B = std::min(batch, ntiles);
    DevBuf ws, grad, m, v, dl;
    RS_TRY(ws.alloc(TileBufs::floats(B, D) * sizeof(float)));
    RS_TRY(grad.alloc(sizeof(float) * W_TOTAL));
    RS_TRY(m.alloc(sizeof(float) * W_TOTAL));
    RS_TRY(v.alloc(sizeof(float) * W_TOTAL));
    RS_TRY(dl.alloc(sizeof(double)));
    RS_CUDA(cudaMemsetAsync(m.p, 0, sizeof(float) * W_TOTAL, st));
    RS_CUDA(cudaMemsetAsync(v.p, 0, sizeof(float) * W_TOTAL, st));
    // number of valid points (interior grid points) of every tile, for the mean
    std::vector<int> tvalid((size_t)ntiles, 0);
    {
        PoolBuf cnt;
        RS_TRY(cnt.alloc(sizeof(int) * (size_t)ntiles, st));
        k_tile_count<<<(unsigned)ntiles, 256, 0, st>>>(msk, dvalid, D3, cnt.as<int>());
        RS_LAUNCH_CHECK();
        RS_CUDA(cudaMemcpyAsync(tvalid.data(), cnt.p, sizeof(int) * (size_t)ntiles, cudaMemcpyDeviceToHost, st));
        RS_CUDA(cudaStreamSynchronize(st));
    }
    TileBufs b(ws.as<float>(), B, D);
    int step = 0;
    for (int ep = 0; ep < epochs; ++ep) {
        RS_CUDA(cudaMemsetAsync(dl.p, 0, sizeof(double), st));
        int nbatches = 0;
        for (int t0 = 0; t0 + B <= ntiles; t0 += B, ++nbatches) {
            int nvalid = 0;
            for (int n = t0; n < t0 + B; ++n) nvalid += tvalid[n];
            const float *x0 = xin + (int64_t)t0 * D3;
            const uint8_t *mk = msk + (int64_t)t0 * D3;
            k_round_weights<<<9, 256, 0, st>>>(w_dev, b.wq, W_TOTAL);
            RS_LAUNCH_CHECK();
            RS_TRY(tile_forward(b.wq, x0, mk, B, D, b, st));
            const int64_t n = (int64_t)B * D3;
            k_tile_loss<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(b.y, tgt + (int64_t)t0 * D3, mk, dvalid, B, D,
                                                                    1.0 / std::max(nvalid, 1), b.g3, dl.as<double>());
            RS_CUDA(cudaMemsetAsync(grad.p, 0, sizeof(float) * W_TOTAL, st));
            RS_TRY(tile_backward(b.wq, x0, mk, B, D, b, grad.as<float>(), st));
            ++step;
            k_adam<<<(W_TOTAL + 255) / 256, 256, 0, st>>>(w_dev, grad.as<float>(), m.as<float>(), v.as<float>(), W_TOTAL,
                                                          lr, 0.9f, 0.999f, 1e-8f, step);
            RS_LAUNCH_CHECK();
        }
        double tot = 0;
        RS_CUDA(cudaMemcpyAsync(&tot, dl.p, sizeof(double), cudaMemcpyDeviceToHost, st));
        RS_CUDA(cudaStreamSynchronize(st));
        if (loss_host) loss_host[ep] = (float)(tot / std::max(nbatches, 1));
    }
    RS_CUDA(cudaStreamSynchronize(st));
    return RS_OK;
}

// Cuts c.n_tiles tiles around random grid points of the column pairs (R, X),
// inputs and targets scaled by the residual column's rms, and trains on them.
int train_pairs_impl(const rs_ham *h, const rs_grid *g, const float *R_dev, const float *X_dev, int64_t ld, int ncols,
                     const rs_train_cfg &c, float *w_dev, float *loss_host, cudaStream_t st) {
    const int D = c.tile + 6, D3 = D * D * D;
    const int64_t np = g->npts;
    // tile positions: a random grid point of a random column at the tile centre
    std::vector<int4> org((size_t)c.n_tiles);
    uint64_t seed = c.seed;
    for (int n = 0; n < c.n_tiles; ++n) {
        const int col = (int)(splitmix64(seed) % (uint64_t)ncols);
        const int64_t p = (int64_t)(splitmix64(seed) % (uint64_t)np);
        const int a = g->ijk[3 * p] - g->origin[0], b = g->ijk[3 * p + 1] - g->origin[1], cc = g->ijk[3 * p + 2] - g->origin[2];
        org[n] = make_int4(col, a - D / 2, b - D / 2, cc - D / 2);
    }
    std::vector<uint8_t> valid((size_t)D3, 0);
    for (int i = 3; i < D - 3; ++i)
        for (int j = 3; j < D - 3; ++j)
            for (int k = 3; k < D - 3; ++k) valid[((size_t)i * D + j) * D + k] = 1;
    DevBuf dorg, dvalid, xin, tgt, msk, ss, rms;
    RS_TRY(dorg.upload(org.data(), org.size() * sizeof(int4)));
    RS_TRY(dvalid.upload(valid.data(), valid.size()));
    RS_TRY(xin.alloc((size_t)c.n_tiles * D3 * sizeof(float)));
    RS_TRY(tgt.alloc((size_t)c.n_tiles * D3 * sizeof(float)));
    RS_TRY(msk.alloc((size_t)c.n_tiles * D3));
    RS_TRY(ss.alloc(sizeof(double) * 256));
    RS_TRY(rms.alloc(sizeof(double) * 256));
    RS_TRY(coldots(RS_F32, R_dev, ld, R_dev, ld, ncols, np, ss.as<double>(), st));
    k_rms<<<1, 256, 0, st>>>(ss.as<double>(), ncols, 1.0 / (double)np, rms.as<double>());
    RS_LAUNCH_CHECK();
    const int64_t ntot = (int64_t)c.n_tiles * D3;
    k_cut_tiles<<<(unsigned)((ntot + 255) / 256), 256, 0, st>>>(
        ham_map(h), g->dims[0], g->dims[1], g->dims[2], R_dev, X_dev, ld, rms.as<double>(), dorg.as<int4>(), c.n_tiles,
        D, xin.as<float>(), tgt.as<float>(), msk.as<uint8_t>());
    RS_LAUNCH_CHECK();
    return train_tiles_impl(w_dev, xin.as<float>(), tgt.as<float>(), msk.as<uint8_t>(), dvalid.as<uint8_t>(), c.n_tiles,
                            D, c.batch, c.epochs, c.lr, loss_host, st);
}

}  // namespace rs

extern "C" int rs_precond_train_pairs(rs_ham *h, const rs_grid *g, const float *R_dev, const float *X_dev, int64_t ld,
                                      int ncols, const rs_train_cfg *cfg, float *w_dev, float *loss_host, void *stream) {
    if (!h || !g || !R_dev || !X_dev || !cfg || !w_dev) return fail(RS_EINVAL, "rs_precond_train_pairs: null argument");
    const rs_train_cfg c = *cfg;
    if (ncols < 1 || ncols > 256 || ld < ncols || c.n_tiles < 1 || c.batch < 1 || c.epochs < 0 || c.tile < 1)
        return fail(RS_EINVAL, "rs_precond_train_pairs: bad sizes");
    if (ham_npts(h) != g->npts) return fail(RS_EINVAL, "rs_precond_train_pairs: grid and Hamiltonian differ");
    return train_pairs_impl(h, g, R_dev, X_dev, ld, ncols, c, w_dev, loss_host, (cudaStream_t)stream);
}

extern "C" int rs_precond_train_tiles(float *w_dev, const float *x_dev, const uint8_t *mask_dev, const float *target_dev,
                                      const uint8_t *valid_dev, int ntiles, int D, int batch, int epochs, float lr,
                                      float *loss_host, void *stream) {
    if (!w_dev || !x_dev || !mask_dev || !target_dev || !valid_dev) return fail(RS_EINVAL, "rs_precond_train_tiles: null argument");
    if (ntiles < 1 || D < 3 || D > 64 || batch < 1 || epochs < 0 || !(lr > 0))
        return fail(RS_EINVAL, "rs_precond_train_tiles: bad sizes");
    return train_tiles_impl(w_dev, x_dev, target_dev, mask_dev, valid_dev, ntiles, D, batch, epochs, lr, loss_host,
                            (cudaStream_t)stream);
}

// ----------------------------------------------------- solver plug-in ---

namespace rs {

// Points below which nb columns go a thread to a point and state.  The row
// kernels win by reading each activation once for three taps, but a CTA's rows (ITEMS nb)
// leave its last round of 256 threads part empty, and small grids do not fill the GPU.
// us, thread per point / row kernels:
//   points   8 052    15 915   28 872   41 625   72 344   120 681  138 507  654 520
//   1 col.   75/77    74/82    74/87    89/105   93/125   133/161  138/167  442/454
//   3        67/81    71/90    80/95    94/121   125/150  181/206  195/214  742/663
//   4        70/81    82/91    99/99    140/129  211/164  315/209  340/219
//   5        72/93    73/105   87/117   114/156  166/181  233/251  259/269
//   6        70/97    78/113   105/121  145/153  197/185  294/272  325/288
//   7        70/104   80/117   106/132  141/165  201/208  288/312  329/332
//   8        73/103   90/116   119/131  176/168  246/226  378/296  420/315
//   9        69/78    87/100   137/146  167/180  241/231  367/360  417/392
//   11       71/83    96/107   150/157  178/189  277/250  425/396  479/433
//   12       74/83    99/108   165/155  210/188  312/260  489/405  552/446
//   16       77/81    128/100  163/140
//   32       117/118  175/146  261/198
// (8 columns, 33 429 points: 148/138; 4 columns, 20 724: 99/92; 5 and 7 columns, 154 249: 285/283, 354/348.)
static int64_t per_point_below(int nb) {
    if (nb <= 3) return INT64_MAX;
    if (nb == 5 || nb == 7) return 150000;
    if (nb == 8) return 31000;
    if (nb >= 6 && nb <= 11) return 50000;
    return nb <= 15 ? 18000 : nb <= 32 ? 10000 : 0;
}

int learned_apply(const rs_ham *h, const float *R, int64_t ldr, float *W, int64_t ldw, int nb, const float *wq_dev,
                  float *act, double *dots, cudaStream_t st) {
    const int64_t np = ham_npts(h);
    double *ss = dots, *rms = dots + 64;
    RS_TRY(coldots(RS_F32, R, ldr, R, ldr, nb, np, ss, st));
    k_rms<<<1, 64, 0, st>>>(ss, nb, 1.0 / (double)np, rms);
    if (np * nb >= (int64_t)INT32_MAX) return fail(RS_EINVAL, "learned preconditioner: npts * nb above 2^31");
    // (the scale array shares the activations' buffer: 64 floats ahead of them)
    const bool per_point = np < per_point_below(nb);
    if (per_point) {
        const int n32 = (int)np;
        float *x = act, *a1 = x + np * nb, *a2 = a1 + np * NC * nb;
        const unsigned blocks = (unsigned)((np * nb + 255) / 256);
        const int32_t *map = ham_map(h), *loc = ham_loc(h);
        const int d1 = ham_dim(h, 1), d2 = ham_dim(h, 2);
        k_net_input<<<blocks, 256, 0, st>>>(R, ldr, rms, nb, n32, x);
        k_net_layer<1, NC, true, false, W1_OFF><<<blocks, 256, 0, st>>>(map, loc, d1, d2, n32, nb, wq_dev, x, a1, 0, rms);
        k_net_layer<NC, NC, true, false, W2_OFF><<<blocks, 256, 0, st>>>(map, loc, d1, d2, n32, nb, wq_dev, a1, a2, 0, rms);
        k_net_layer<NC, 1, false, true, W3_OFF><<<blocks, 256, 0, st>>>(map, loc, d1, d2, n32, nb, wq_dev, a2, W, ldw, rms);
        RS_LAUNCH_CHECK();
        return RS_OK;
    }
    float *scale = act;
    uint32_t *a1 = reinterpret_cast<uint32_t *>(act + 64);   // three BF16 pieces of 8 channels
    float *a2 = reinterpret_cast<float *>(a1 + np * nb * (3 * NC / 2));
    k_net_scale<<<1, 64, 0, st>>>(rms, nb, scale);
    NetGrid g;
    g.map = ham_map(h);
    g.d1 = ham_dim(h, 1), g.d2 = ham_dim(h, 2);
    g.n4 = (g.d2 + ROWN - 1) / ROWN;
    g.items = ham_dim(h, 0) * g.d1 * g.n4;
    g.nb = nb;
    auto layers = [&](auto items, auto uni) {
        constexpr int ITEMS = decltype(items)::value;
        const unsigned blocks = (unsigned)((g.items + ITEMS - 1) / ITEMS);
        k_net_first<ITEMS><<<blocks, NET_NT, 0, st>>>(g, wq_dev, R, ldr, scale, reinterpret_cast<uint4 *>(a1));
        k_net_mid<ITEMS, decltype(uni)::value><<<blocks, NET_NT, 0, st>>>(g, wq_dev, a1, a2);
        k_net_last<ITEMS><<<blocks, NET_NT, 0, st>>>(g, wq_dev, a2, W, ldw, rms);
    };
    using std::integral_constant;
    if (nb <= 8) layers(integral_constant<int, 64>{}, integral_constant<bool, false>{});
    else if (nb % 16) layers(integral_constant<int, 16>{}, integral_constant<bool, false>{});
    else layers(integral_constant<int, 16>{}, integral_constant<bool, true>{});
    RS_LAUNCH_CHECK();
    return RS_OK;
}

int64_t learned_act_floats(int64_t npts, int nb) { return npts * nb * (3 * NC / 2 + NC) + 64; }

int learned_round_weights(const float *w, float *wq, cudaStream_t st) {
    k_round_weights<<<9, 256, 0, st>>>(w, wq, W_TOTAL);
    RS_LAUNCH_CHECK();
    return RS_OK;
}

}  // namespace rs

extern "C" int rs_precond_apply(rs_ham *h, const float *w_dev, const float *R_dev, int64_t ldr, float *W_dev, int64_t ldw,
                                int nb, void *stream) {
    if (!h || !w_dev || !R_dev || !W_dev) return fail(RS_EINVAL, "rs_precond_apply: null argument");
    if (nb < 1 || nb > 64 || ldr < nb || ldw < nb) return fail(RS_EINVAL, "rs_precond_apply: bad nb or ld");
    cudaStream_t st = (cudaStream_t)stream;
    DevBuf *ws = ham_scratch(h, (sizeof(float) * (size_t)(LEARNED_WEIGHTS + learned_act_floats(ham_npts(h), nb))) +
                                    sizeof(double) * 128);
    if (!ws) return fail(RS_ENOMEM, "rs_precond_apply: device allocation failed");
    double *dots = ws->as<double>();
    float *wq = reinterpret_cast<float *>(dots + 128);
    float *act = wq + LEARNED_WEIGHTS;
    RS_TRY(learned_round_weights(w_dev, wq, st));
    return learned_apply(h, R_dev, ldr, W_dev, ldw, nb, wq, act, dots, st);
}
