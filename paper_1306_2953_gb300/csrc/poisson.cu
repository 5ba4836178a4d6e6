// Hartree potential by fast Fourier transforms (Sec. X; Eq. 2, the Poisson
// equation lap V_H = -4 pi n), the paper's steps on the GPU:
//   1. the density is copied from the grid to a cube (zero elsewhere);
//   2. forward 3-D FFT;
//   3. multiplication by the Coulomb-interaction kernel;
//   4. inverse 3-D FFT;
//   5. the potential is copied back to the grid.
// Free boundary conditions: an enlarged cube and the spherical-cutoff kernel
// of Rozzi et al. (2006), the Coulomb potential cut off at r = R_c,
//   v(G) = 4 pi (1 - cos(|G| R_c)) / |G|^2,   v(0) = 2 pi R_c^2,
// with R_c = D + h (D: the diagonal of the grid's bounding box) and N_a
// points along axis a, the smallest 2^p 3^q >= extent_a + ceil(R_c / h) + 1,
// so that no periodic image of the density lies within R_c of it.
//
// The transforms are complex FP64 and bound by GB300's few FP64 units (about
// 554 G fused operations a second), so the work is cut to what the cube needs:
//  - The density and the potential are real: along axis 2 two lines make one
//    complex transform, and only the N_2 / 2 + 1 frequencies are kept.
//  - They are zero, or not asked for, outside the grid's bounding box (e_a of
//    N_a points, at most half): axis 2 transforms only the e_0 e_1 lines that
//    hold points, axis 1 only the e_0 planes; axis 0, all lines, goes forward,
//    through the kernel and back in one launch, reading and writing only its
//    e_0 planes.
//  - Stockham passes (Govindaraju et al. 2008 formulation: pass with radix R
//    and span Ns reads R inputs N/R apart, twiddles them by
//    exp(-+2 pi i r (j mod Ns) / (Ns R)), takes an R-point DFT and writes R
//    outputs Ns apart) of radix 9, 3, 8, 4, 2: 9 and 8 take 4.9 operations per
//    point and factor 3, 2.2 per factor 2, before their twiddles; the first
//    pass has none, and when it is one of radix 9 it skips the inputs that are
//    zero.  Twiddles come from a table of exp(2 pi i m / N) in shared memory.
// On the 288^3 cube of the 100-atom molecule (655 k points, e = 105 .. 109)
// that is 126 k lines instead of 498 k and 26.8 operations per point instead of
// 33: a solve takes 2.02 ms (1.76 at the FP64 units' rate), 10.3 ms before, when
// every line of the complex cube was transformed with radices 3, 4 and 2.
#include <algorithm>
#include <cmath>
#include <new>
#include <vector>

#include "device.h"

namespace {

constexpr int LN = 8;          // lines per CTA
constexpr int FFT_NT = 256;
constexpr int MAX_N = 768;     // largest axis length (two LN-line buffers and the table fit in shared memory)

struct __align__(16) Cplx {
    double x, y;
};
__device__ __forceinline__ Cplx cmul(Cplx a, Cplx b) { return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x}; }
__device__ __forceinline__ Cplx cadd(Cplx a, Cplx b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ Cplx csub(Cplx a, Cplx b) { return {a.x - b.x, a.y - b.y}; }

struct Radices {
    int r[16];
    int n;
};

// DFTs in place, S = -1 forward, +1 inverse (unnormalised).
template <int S> __device__ __forceinline__ void dft2(Cplx (&v)[2]) {
    const Cplx a = v[0];
    v[0] = cadd(a, v[1]);
    v[1] = csub(a, v[1]);
}
constexpr double S3 = 0.86602540378443864676;   // sin(2 pi / 3)
template <int S> __device__ __forceinline__ void dft3(Cplx &a, Cplx &b, Cplx &c) {
    const Cplx t = cadd(b, c), d = csub(b, c);
    const Cplx m = {fma(-0.5, t.x, a.x), fma(-0.5, t.y, a.y)};
    a = cadd(a, t);
    // m +- S i sin(2 pi / 3) d
    b = {fma(-S * S3, d.y, m.x), fma(S * S3, d.x, m.y)};
    c = {fma(S * S3, d.y, m.x), fma(-S * S3, d.x, m.y)};
}
template <int S> __device__ __forceinline__ void dft4(Cplx &v0, Cplx &v1, Cplx &v2, Cplx &v3) {
    const Cplx a = cadd(v0, v2), b = csub(v0, v2), c = cadd(v1, v3), d = csub(v1, v3);
    v0 = cadd(a, c);
    v1 = {b.x - S * d.y, b.y + S * d.x};
    v2 = csub(a, c);
    v3 = {b.x + S * d.y, b.y - S * d.x};
}
template <int S> __device__ __forceinline__ void dft8(Cplx (&v)[8]) {
    constexpr double H = 0.70710678118654752440;
    dft4<S>(v[0], v[2], v[4], v[6]);   // even inputs: results 0 .. 3 in v[0], v[2], v[4], v[6]
    dft4<S>(v[1], v[3], v[5], v[7]);   // odd inputs
    const Cplx e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o2 = v[5];
    // odd result k times exp(S 2 pi i k / 8), the factor 1 / sqrt(2) of k = 1, 3 in the last sums
    const Cplx t1 = {v[3].x - S * v[3].y, v[3].y + S * v[3].x};
    const Cplx t2 = {-S * o2.y, S * o2.x};
    const Cplx t3 = {-v[7].x - S * v[7].y, -v[7].y + S * v[7].x};
    v[0] = cadd(e0, o0);
    v[4] = csub(e0, o0);
    v[1] = {fma(H, t1.x, e1.x), fma(H, t1.y, e1.y)};
    v[5] = {fma(-H, t1.x, e1.x), fma(-H, t1.y, e1.y)};
    v[2] = cadd(e2, t2);
    v[6] = csub(e2, t2);
    v[3] = {fma(H, t3.x, e3.x), fma(H, t3.y, e3.y)};
    v[7] = {fma(-H, t3.x, e3.x), fma(-H, t3.y, e3.y)};
}
// FEW: inputs 4 .. 8 are zero
template <int S, bool FEW> __device__ __forceinline__ void dft9(Cplx (&v)[9]) {
    constexpr double C1 = 0.76604444311897803520, S1 = 0.64278760968653932632;    // cos, sin of 2 pi / 9
    constexpr double C2 = 0.17364817766693034885, S2 = 0.98480775301220805937;    // 4 pi / 9
    constexpr double C4 = -0.93969262078590838405, S4 = 0.34202014332566873304;   // 8 pi / 9
    if constexpr (FEW) {
        // three-point transforms of (v0, v3, 0), (v1, 0, 0), (v2, 0, 0)
        const Cplx b = v[3];
        const Cplx m = {fma(-0.5, b.x, v[0].x), fma(-0.5, b.y, v[0].y)};
        v[0] = cadd(v[0], b);
        v[3] = {fma(-S * S3, b.y, m.x), fma(S * S3, b.x, m.y)};
        v[6] = {fma(S * S3, b.y, m.x), fma(-S * S3, b.x, m.y)};
        v[4] = v[7] = v[1];
        v[5] = v[8] = v[2];
    } else {
        dft3<S>(v[0], v[3], v[6]);
        dft3<S>(v[1], v[4], v[7]);
        dft3<S>(v[2], v[5], v[8]);
    }
    v[4] = cmul(v[4], {C1, S * S1});
    v[7] = cmul(v[7], {C2, S * S2});
    v[5] = cmul(v[5], {C2, S * S2});
    v[8] = cmul(v[8], {C4, S * S4});
    dft3<S>(v[0], v[1], v[2]);
    dft3<S>(v[3], v[4], v[5]);
    dft3<S>(v[6], v[7], v[8]);
    // result 3 b + a of group a, element b
    const Cplx t1 = v[1], t2 = v[2], t5 = v[5];
    v[1] = v[3];
    v[2] = v[6];
    v[3] = t1;
    v[5] = v[7];
    v[6] = t2;
    v[7] = t5;
}

// One pass of radix R over nl lines (stride np in x and y).
template <int R, int S, bool FEW>
__device__ __forceinline__ void fft_pass(const Cplx *x, Cplx *y, const Cplx *T, int nl, int np, int N, int Ns) {
    const int M = N / R, step = N / (Ns * R);
    for (int e = threadIdx.x; e < nl * M; e += FFT_NT) {
        const int l = e / M, j = e - l * M;
        const Cplx *xl = x + l * np + j;
        const int q = j / Ns, k = j - q * Ns;
        Cplx v[R];
#pragma unroll
        for (int r = 0; r < (FEW ? 4 : R); ++r) v[r] = xl[r * M];
        if (!FEW && k) {
            // input r times exp(S 2 pi i r k / (Ns R))
            const int ks = k * step;
#pragma unroll
            for (int r = 1; r < R; ++r) {
                const Cplx w = T[r * ks];
                v[r] = cmul(v[r], {w.x, S * w.y});
            }
        }
        if constexpr (R == 2) dft2<S>(v);
        else if constexpr (R == 3) dft3<S>(v[0], v[1], v[2]);
        else if constexpr (R == 4) dft4<S>(v[0], v[1], v[2], v[3]);
        else if constexpr (R == 8) dft8<S>(v);
        else dft9<S, FEW>(v);
        Cplx *yl = y + l * np + q * Ns * R + k;
#pragma unroll
        for (int r = 0; r < R; ++r) yl[r * Ns] = v[r];
    }
    __syncthreads();
}

// Transforms nl lines of length N held in a (line stride np), with b as the
// other buffer; ein: inputs from there on are zero.  Returns the buffer that
// holds the result.  Ends with a barrier.
template <int S> __device__ Cplx *fft_lines(Cplx *a, Cplx *b, const Cplx *T, int nl, int np, int N, const Radices &rad, int ein) {
    int Ns = 1;
    for (int p = 0; p < rad.n; ++p) {
        const int R = rad.r[p];
        if (R == 9) {
            if (p == 0 && 9 * ein <= 4 * N) fft_pass<9, S, true>(a, b, T, nl, np, N, Ns);
            else fft_pass<9, S, false>(a, b, T, nl, np, N, Ns);
        } else if (R == 8) fft_pass<8, S, false>(a, b, T, nl, np, N, Ns);
        else if (R == 4) fft_pass<4, S, false>(a, b, T, nl, np, N, Ns);
        else if (R == 3) fft_pass<3, S, false>(a, b, T, nl, np, N, Ns);
        else fft_pass<2, S, false>(a, b, T, nl, np, N, Ns);
        Cplx *t = a;
        a = b;
        b = t;
        Ns *= R;
    }
    return a;
}

struct Shape {
    int N[3], e[3];   // cube and bounding box
    int H;            // frequencies kept along axis 2: N[2] / 2 + 1
};

// shared memory: two buffers of LN lines (an odd stride, so that one element
// of eight lines falls in distinct banks) and the twiddles
__host__ __device__ inline int line_stride(int N) { return N | 1; }
__device__ __forceinline__ void fft_buffers(int N, const Cplx *tw, Cplx *&A, Cplx *&B, Cplx *&T) {
    extern __shared__ __align__(16) unsigned char fsm[];
    A = reinterpret_cast<Cplx *>(fsm);
    B = A + LN * line_stride(N);
    T = B + LN * line_stride(N);
    for (int m = threadIdx.x; m < N; m += FFT_NT) T[m] = tw[m];
}

// Axis 2 forward: pairs of real lines (i0, 2q), (i0, 2q + 1) of the box ->
// C1[i0][i1][k2], k2 < H.
__global__ void __launch_bounds__(FFT_NT) k_fft2_fwd(const double *__restrict__ box, Cplx *__restrict__ C1, Shape s, Radices rad,
                                                      const Cplx *__restrict__ tw) {
    Cplx *A, *B, *T;
    const int N = s.N[2], np = line_stride(N), hp = (s.e[1] + 1) / 2;
    fft_buffers(N, tw, A, B, T);
    const int l0 = blockIdx.x * LN, nl = min(LN, s.e[0] * hp - l0);
    for (int e = threadIdx.x; e < nl * N; e += FFT_NT) {
        const int l = e / N, j = e - l * N, i0 = (l0 + l) / hp, i1 = 2 * ((l0 + l) - i0 * hp);
        const double *r = box + ((int64_t)i0 * s.e[1] + i1) * s.e[2] + j;
        const bool in = j < s.e[2];
        A[l * np + j] = {in ? r[0] : 0.0, in && i1 + 1 < s.e[1] ? r[s.e[2]] : 0.0};
    }
    __syncthreads();
    const Cplx *z = fft_lines<-1>(A, B, T, nl, np, N, rad, s.e[2]);
    for (int e = threadIdx.x; e < nl * s.H; e += FFT_NT) {
        const int l = e / s.H, k = e - l * s.H, i0 = (l0 + l) / hp, i1 = 2 * ((l0 + l) - i0 * hp);
        const Cplx p = z[l * np + k], m = z[l * np + (k ? N - k : 0)];
        Cplx *c = C1 + ((int64_t)i0 * s.e[1] + i1) * s.H + k;
        // Z = A + i B with A, B of real lines: conj(Z[-k]) = A - i B
        c[0] = {0.5 * (p.x + m.x), 0.5 * (p.y - m.y)};
        if (i1 + 1 < s.e[1]) c[s.H] = {0.5 * (p.y + m.y), 0.5 * (m.x - p.x)};
    }
}

// Axis 2 inverse: C1 -> real box.
__global__ void __launch_bounds__(FFT_NT) k_fft2_inv(const Cplx *__restrict__ C1, double *__restrict__ box, Shape s, Radices rad,
                                                      const Cplx *__restrict__ tw) {
    Cplx *A, *B, *T;
    const int N = s.N[2], np = line_stride(N), hp = (s.e[1] + 1) / 2;
    fft_buffers(N, tw, A, B, T);
    const int l0 = blockIdx.x * LN, nl = min(LN, s.e[0] * hp - l0);
    for (int e = threadIdx.x; e < nl * s.H; e += FFT_NT) {
        const int l = e / s.H, k = e - l * s.H, i0 = (l0 + l) / hp, i1 = 2 * ((l0 + l) - i0 * hp);
        const Cplx *c = C1 + ((int64_t)i0 * s.e[1] + i1) * s.H + k;
        Cplx a = c[0], b = i1 + 1 < s.e[1] ? c[s.H] : Cplx{0.0, 0.0};
        Cplx *z = A + l * np;
        if (k == 0 || 2 * k == N) {
            z[k] = {a.x, b.x};   // the spectra of real lines are real there
        } else {
            z[k] = {a.x - b.y, a.y + b.x};
            z[N - k] = {a.x + b.y, b.x - a.y};
        }
    }
    __syncthreads();
    const Cplx *z = fft_lines<1>(A, B, T, nl, np, N, rad, N);
    for (int e = threadIdx.x; e < nl * s.e[2]; e += FFT_NT) {
        const int l = e / s.e[2], j = e - l * s.e[2], i0 = (l0 + l) / hp, i1 = 2 * ((l0 + l) - i0 * hp);
        double *r = box + ((int64_t)i0 * s.e[1] + i1) * s.e[2] + j;
        const Cplx v = z[l * np + j];
        r[0] = v.x;
        if (i1 + 1 < s.e[1]) r[s.e[2]] = v.y;
    }
}

// Axis 1: C1[i0][i1 < e1][k2] -> C2[i0][k1][k2] (S = -1) and back (S = 1); a CTA
// takes LN adjacent k2 of one plane i0.
template <int S>
__global__ void __launch_bounds__(FFT_NT) k_fft1(const Cplx *__restrict__ in, Cplx *__restrict__ out, Shape s, Radices rad,
                                                  const Cplx *__restrict__ tw) {
    Cplx *A, *B, *T;
    const int N = s.N[1], np = line_stride(N);
    fft_buffers(N, tw, A, B, T);
    const int k20 = blockIdx.x * LN, nl = min(LN, s.H - k20);
    const int ni = S < 0 ? s.e[1] : N, no = S < 0 ? N : s.e[1];
    in += (int64_t)blockIdx.y * ni * s.H + k20;
    out += (int64_t)blockIdx.y * no * s.H + k20;
    for (int e = threadIdx.x; e < nl * N; e += FFT_NT) {
        const int j = e / nl, l = e - j * nl;
        A[l * np + j] = j < ni ? in[(int64_t)j * s.H + l] : Cplx{0.0, 0.0};
    }
    __syncthreads();
    const Cplx *z = fft_lines<S>(A, B, T, nl, np, N, rad, ni);
    for (int e = threadIdx.x; e < nl * no; e += FFT_NT) {
        const int j = e / nl, l = e - j * nl;
        out[(int64_t)j * s.H + l] = z[l * np + j];
    }
}

// Axis 0 forward, the Coulomb kernel (with the transforms' normalisation), axis
// 0 inverse, in place on C2[i0 < e0][line]; a CTA takes LN adjacent lines.
__global__ void __launch_bounds__(FFT_NT) k_fft0(Cplx *__restrict__ C2, const double *__restrict__ vg, Shape s, Radices rad,
                                                  const Cplx *__restrict__ tw) {
    Cplx *A, *B, *T;
    const int N = s.N[0], np = line_stride(N);
    fft_buffers(N, tw, A, B, T);
    const int64_t lines = (int64_t)s.N[1] * s.H, l0 = (int64_t)blockIdx.x * LN;
    const int nl = lines - l0 < LN ? (int)(lines - l0) : LN;
    for (int e = threadIdx.x; e < nl * N; e += FFT_NT) {
        const int j = e / nl, l = e - j * nl;
        A[l * np + j] = j < s.e[0] ? C2[j * lines + l0 + l] : Cplx{0.0, 0.0};
    }
    __syncthreads();
    Cplx *z = fft_lines<-1>(A, B, T, nl, np, N, rad, s.e[0]);
    for (int e = threadIdx.x; e < nl * N; e += FFT_NT) {
        const int j = e / nl, l = e - j * nl;
        const double v = __ldg(vg + j * lines + l0 + l);
        Cplx &c = z[l * np + j];
        c = {c.x * v, c.y * v};
    }
    __syncthreads();
    z = fft_lines<1>(z, z == A ? B : A, T, nl, np, N, rad, N);
    for (int e = threadIdx.x; e < nl * s.e[0]; e += FFT_NT) {
        const int j = e / nl, l = e - j * nl;
        C2[j * lines + l0 + l] = z[l * np + j];
    }
}

__global__ void k_to_box(const double *__restrict__ n, const int32_t *__restrict__ idx, int64_t npts, double *__restrict__ box) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < npts; p += (int64_t)gridDim.x * blockDim.x)
        box[idx[p]] = n[p];
}

__global__ void k_from_box(const double *__restrict__ box, const int32_t *__restrict__ idx, int64_t npts, double *__restrict__ v) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < npts; p += (int64_t)gridDim.x * blockDim.x)
        v[p] = box[idx[p]];
}

// v(G) / (N_0 N_1 N_2) at the kept frequencies: G_a = 2 pi f_a / (N_a h), f_a the
// signed frequency of index i_a (computed once per plan)
__global__ void k_kernel_values(double *__restrict__ vg, int n0, int n1, int n2, int nh, double h, double rc) {
    const int64_t tot = (int64_t)n0 * n1 * nh;
    const double tp = 2.0 * 3.14159265358979323846, cube = (double)n0 * (double)n1 * (double)n2;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
        const int i2 = (int)(e % nh), i1 = (int)((e / nh) % n1), i0 = (int)(e / ((int64_t)n1 * nh));
        const int f0 = i0 < (n0 + 1) / 2 ? i0 : i0 - n0, f1 = i1 < (n1 + 1) / 2 ? i1 : i1 - n1, f2 = i2;
        const double g0 = tp * f0 / (n0 * h), g1 = tp * f1 / (n1 * h), g2 = tp * f2 / (n2 * h);
        const double G2 = g0 * g0 + g1 * g1 + g2 * g2;
        vg[e] = (e == 0 ? tp * rc * rc : 2.0 * tp * (1.0 - cos(sqrt(G2) * rc)) / G2) / cube;
    }
}

int smooth_size(int n) {
    int best = -1;
    for (int64_t p2 = 1; p2 < 2 * (int64_t)n + 2; p2 *= 2)
        for (int64_t p3 = p2; p3 < 2 * (int64_t)n + 2; p3 *= 3)
            if (p3 >= n && (best < 0 || p3 < best)) best = (int)p3;
    return best;
}

Radices radices(int n) {
    Radices r{};
    for (int R : {9, 3, 8, 4, 2})
        while (n % R == 0) {
            r.r[r.n++] = R;
            n /= R;
        }
    return r;
}

}  // namespace

struct rs_poisson {
    int64_t npts = 0;
    Shape s{};
    double h = 0, rc = 0;
    // real box, half-transformed planes, v(G), twiddles exp(2 pi i m / N[a])
    rs::DevBuf box, c1, c2, idx, vg, tw[3];
};

using rs::fail;

extern "C" int rs_poisson_create(const rs_grid *g, rs_poisson **out) {
    if (!g || !out) return fail(RS_EINVAL, "rs_poisson_create: null argument");
    *out = nullptr;
    if (g->npts < 1) return fail(RS_EINVAL, "rs_poisson_create: empty grid");
    int32_t lo[3], hi[3];
    for (int d = 0; d < 3; ++d) lo[d] = hi[d] = g->ijk[d];
    for (int64_t p = 0; p < g->npts; ++p)
        for (int d = 0; d < 3; ++d) {
            lo[d] = std::min(lo[d], g->ijk[3 * p + d]);
            hi[d] = std::max(hi[d], g->ijk[3 * p + d]);
        }
    double D2 = 0;
    for (int d = 0; d < 3; ++d) D2 += (double)(hi[d] - lo[d]) * (double)(hi[d] - lo[d]);
    const double rc = g->h * std::sqrt(D2) + g->h;
    rs_poisson *P = new (std::nothrow) rs_poisson;
    if (!P) return fail(RS_ENOMEM, "host allocation failed");
    P->npts = g->npts;
    P->h = g->h;
    P->rc = rc;
    Shape &s = P->s;
    int64_t tot = 1;
    for (int d = 0; d < 3; ++d) {
        s.e[d] = hi[d] - lo[d] + 1;
        s.N[d] = smooth_size((hi[d] - lo[d]) + (int)std::ceil(rc / g->h) + 1);
        if (s.N[d] > MAX_N) {
            const int n = s.N[d];
            delete P;
            return fail(RS_EINVAL, "rs_poisson_create: cube of %d points along an axis exceeds %d", n, MAX_N);
        }
        tot *= s.N[d];
    }
    if (tot > INT32_MAX) {
        delete P;
        return fail(RS_EINVAL, "rs_poisson_create: cube too large");
    }
    s.H = s.N[2] / 2 + 1;
    std::vector<int32_t> idx((size_t)g->npts);
    for (int64_t p = 0; p < g->npts; ++p)
        idx[p] = (int32_t)(((int64_t)(g->ijk[3 * p] - lo[0]) * s.e[1] + (g->ijk[3 * p + 1] - lo[1])) * s.e[2] +
                           (g->ijk[3 * p + 2] - lo[2]));
    int rc2;
    const size_t nbox = (size_t)s.e[0] * s.e[1] * s.e[2];
    if ((rc2 = P->idx.upload(idx.data(), idx.size() * sizeof(int32_t))) || (rc2 = P->box.alloc(nbox * sizeof(double))) ||
        (rc2 = P->c1.alloc((size_t)s.e[0] * s.e[1] * s.H * sizeof(Cplx))) ||
        (rc2 = P->c2.alloc((size_t)s.e[0] * s.N[1] * s.H * sizeof(Cplx))) ||
        (rc2 = P->vg.alloc((size_t)s.N[0] * s.N[1] * s.H * sizeof(double)))) {
        delete P;
        return rc2;
    }
    k_kernel_values<<<152 * 16, 256>>>(P->vg.as<double>(), s.N[0], s.N[1], s.N[2], s.H, P->h, P->rc);
    if (cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) {
        delete P;
        return fail(RS_ECUDA, "rs_poisson_create: kernel table failed");
    }
    for (int d = 0; d < 3; ++d) {
        std::vector<Cplx> t((size_t)s.N[d]);
        const double tp = 2.0 * 3.14159265358979323846;
        for (int m = 0; m < s.N[d]; ++m) t[m] = {std::cos(tp * m / s.N[d]), std::sin(tp * m / s.N[d])};
        if ((rc2 = P->tw[d].upload(t.data(), t.size() * sizeof(Cplx)))) {
            delete P;
            return rc2;
        }
    }
    *out = P;
    return RS_OK;
}

extern "C" int rs_poisson_info(const rs_poisson *P, int32_t shape[3], double *r_cut, int64_t *cube_bytes) {
    if (!P) return fail(RS_EINVAL, "rs_poisson_info: null handle");
    for (int d = 0; d < 3 && shape; ++d) shape[d] = P->s.N[d];
    if (r_cut) *r_cut = P->rc;
    if (cube_bytes) *cube_bytes = (int64_t)P->s.N[0] * P->s.N[1] * P->s.N[2] * (int64_t)sizeof(Cplx);
    return RS_OK;
}

extern "C" int rs_poisson_solve(rs_poisson *P, const double *n_dev, double *vh_dev, void *stream) {
    if (!P || !n_dev || !vh_dev) return fail(RS_EINVAL, "rs_poisson_solve: null argument");
    cudaStream_t st = (cudaStream_t)stream;
    const Shape s = P->s;
    double *box = P->box.as<double>();
    Cplx *c1 = P->c1.as<Cplx>(), *c2 = P->c2.as<Cplx>();
    size_t smem[3];
    Radices rad[3];
    for (int d = 0; d < 3; ++d) {
        smem[d] = (2 * (size_t)LN * line_stride(s.N[d]) + s.N[d]) * sizeof(Cplx);
        rad[d] = radices(s.N[d]);
    }
    RS_TRY(rs::smem_optin((const void *)k_fft2_fwd, smem[2]));
    RS_TRY(rs::smem_optin((const void *)k_fft2_inv, smem[2]));
    RS_TRY(rs::smem_optin((const void *)k_fft1<-1>, smem[1]));
    RS_TRY(rs::smem_optin((const void *)k_fft1<1>, smem[1]));
    RS_TRY(rs::smem_optin((const void *)k_fft0, smem[0]));
    const unsigned pb = (unsigned)std::min<int64_t>((P->npts + 255) / 256, 152 * 16);
    const unsigned b2 = (unsigned)((s.e[0] * ((s.e[1] + 1) / 2) + LN - 1) / LN);
    const dim3 b1((unsigned)((s.H + LN - 1) / LN), (unsigned)s.e[0]);
    const unsigned b0 = (unsigned)(((int64_t)s.N[1] * s.H + LN - 1) / LN);
    // (the inverse leaves values at box positions that are not grid points)
    RS_CUDA(cudaMemsetAsync(box, 0, sizeof(double) * (size_t)s.e[0] * s.e[1] * s.e[2], st));
    k_to_box<<<pb, 256, 0, st>>>(n_dev, P->idx.as<int32_t>(), P->npts, box);
    k_fft2_fwd<<<b2, FFT_NT, smem[2], st>>>(box, c1, s, rad[2], P->tw[2].as<Cplx>());
    k_fft1<-1><<<b1, FFT_NT, smem[1], st>>>(c1, c2, s, rad[1], P->tw[1].as<Cplx>());
    k_fft0<<<b0, FFT_NT, smem[0], st>>>(c2, P->vg.as<double>(), s, rad[0], P->tw[0].as<Cplx>());
    k_fft1<1><<<b1, FFT_NT, smem[1], st>>>(c2, c1, s, rad[1], P->tw[1].as<Cplx>());
    k_fft2_inv<<<b2, FFT_NT, smem[2], st>>>(c1, box, s, rad[2], P->tw[2].as<Cplx>());
    k_from_box<<<pb, 256, 0, st>>>(box, P->idx.as<int32_t>(), P->npts, vh_dev);
    RS_LAUNCH_CHECK();
    return RS_OK;
}

extern "C" int rs_poisson_destroy(rs_poisson *P) {
    delete P;
    return RS_OK;
}
