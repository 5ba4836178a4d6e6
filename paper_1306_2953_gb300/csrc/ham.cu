// Kohn-Sham Hamiltonian applied to a block of orbitals (Sec. V, Eq. 3).
//
// Two launches per block:
//  1. k_project: the Kleinman-Bylander projection integrals of Eq. (4),
//     c[A,q,s] = E[A,q] dV sum_{p in S_A} gamma_Aq(p) psi(p,s), PSPLIT CTAs
//     per (atom, state group), each a block-wide tree reduction over its share
//     of the sphere points; the last of them adds the shares up; stored
//     [atom][state][q] so that one 16-byte load gives a state's four.
//     FP32 blocks of 32-state groups take k_project_f32 (four states per lane
//     and four sphere entries per warp step, the atom split sized to fill the
//     GPU).
//  2. k_gather: the 25-point star kinetic stencil (Sec. V.A), the local
//     potential (Sec. V.B) and the nonlocal sum of Eq. (4), fused: every
//     point reads its 24 neighbours' rows.  The nonlocal term is a gather too
//     (each output point sums over the atoms whose spheres cover it), so
//     overlapping spheres need neither atom colouring (Sec. V.C, Fig. 10) nor
//     atomics, and the output is written exactly once.
// Orbitals are [npts][ld] with the state index fastest (Sec. IV, Fig. 4b);
// grid points are addressed through the int32 point map (Sec. V.A).
// FP32 blocks whose state count is a multiple of 32 take the persistent
// ring-buffer kernel of stencil_ring.cu for step 2 instead; k_gather serves
// FP64 blocks, narrower state groups and layouts that kernel cannot copy.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "device.h"
#include "ham.h"
#include "stencil_ring.h"

// 1: FP32 blocks of 32 states go to the persistent ring-buffer kernel
// (stencil_ring.cu) when the block's layout allows 16-byte row copies.
#ifndef RS_STENCIL_RING
#define RS_STENCIL_RING 1
#endif

// Height (planes) of the z-slabs the ring kernel lays its columns out in
// before cutting them into per-CTA runs (the default: whole columns).
#ifndef RS_RING_SLAB
#define RS_RING_SLAB 4096
#endif

namespace rs {

template <typename T> struct HamDev {
    const int4 *pinfo;  // per point: nonlocal entry range [x, y) and V (z: float bits; z,w: double bits)
    const int32_t *map;
    int d0, d1, d2;
    const T *V;
    const int32_t *cov_off, *cov_atom;
    const T *cov_gam;   // [entries][4]
    const int32_t *sph_off, *sph_idx;
    const T *sph_gam;   // [entries][4]
    const T *E;         // [atoms][4]
    T dV;
    T w[5];             // w[0] = 3 kin c_0, w[j] = kin c_j, kin = -1/(2h^2)
};

// ---------------------------------------------------------------- helpers --

template <typename T> __device__ __forceinline__ T point_v(int4 inf);
template <> __device__ __forceinline__ float point_v<float>(int4 inf) { return __int_as_float(inf.z); }
template <> __device__ __forceinline__ double point_v<double>(int4 inf) { return __hiloint2double(inf.w, inf.z); }

template <typename T> struct Four { T a, b, c, d; };
__device__ __forceinline__ Four<float> load4(const float *p) {
    float4 v = __ldg(reinterpret_cast<const float4 *>(p));
    return {v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ Four<double> load4(const double *p) {
    double2 u = __ldg(reinterpret_cast<const double2 *>(p));
    double2 v = __ldg(reinterpret_cast<const double2 *>(p) + 1);
    return {u.x, u.y, v.x, v.y};
}

__device__ __forceinline__ Four<float> fresh4(const float *p) {
    const float4 v = ld_fresh(reinterpret_cast<const float4 *>(p));
    return {v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ Four<double> fresh4(const double *p) {
    const double2 u = ld_fresh(reinterpret_cast<const double2 *>(p)), v = ld_fresh(reinterpret_cast<const double2 *>(p) + 1);
    return {u.x, u.y, v.x, v.y};
}

// ------------------------------------------------- projection integrals ---

// Grid (atoms * split, state groups): each CTA sums 1 / split of an atom's
// sphere points and writes its partial sums to `part` [atom, group][split][n];
// the CTA that comes last (`count`, which returns to zero) adds the parts in
// their order and writes the group's coefficients.
// (Atomic additions to zeroed coefficients needed a memset before each block and
// gave sums that depended on the order.)
constexpr int PSPLIT = 8;

// True in the whole CTA that is the last of the `split` of its atom and group;
// the parts of the others are visible to it.
__device__ __forceinline__ bool last_part(unsigned *count, int split) {
    __shared__ int last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicInc(count, (unsigned)split - 1) == (unsigned)split - 1;
    __syncthreads();
    if (last) __threadfence();
    return last;
}

template <typename T, int SGP, int NT>
__global__ void __launch_bounds__(NT) k_project(HamDev<T> d, const T *__restrict__ psi, int64_t ldp, int nb,
                                                T *part, unsigned *count, T *__restrict__ cproj) {
    constexpr int R = NT / SGP;
    __shared__ T red[4][NT];
    const int A = blockIdx.x / PSPLIT, piece = blockIdx.x % PSPLIT;
    const int sg0 = blockIdx.y * SGP;
    const int s = threadIdx.x % SGP, r = threadIdx.x / SGP;
    const int o = __ldg(d.sph_off + A), e = __ldg(d.sph_off + A + 1);
    const int len = e - o, per = (len + PSPLIT - 1) / PSPLIT;
    const int i0 = o + piece * per, i1 = min(e, i0 + per);
    pdl_wait();
    const T *ps = psi + sg0 + s;
    T a0 = 0, a1 = 0, a2 = 0, a3 = 0;
#pragma unroll 8
    for (int i = i0 + r; i < i1; i += R) {
        const int p = __ldg(d.sph_idx + i);
        const T v = ld_fresh(ps + (int64_t)p * ldp);
        const Four<T> g = load4(d.sph_gam + 4 * (int64_t)i);
        a0 += g.a * v;
        a1 += g.b * v;
        a2 += g.c * v;
        a3 += g.d * v;
    }
    red[0][threadIdx.x] = a0;
    red[1][threadIdx.x] = a1;
    red[2][threadIdx.x] = a2;
    red[3][threadIdx.x] = a3;
    __syncthreads();
    for (int st = R / 2; st > 0; st >>= 1) {
        if (r < st) {
#pragma unroll
            for (int q = 0; q < 4; ++q) red[q][threadIdx.x] += red[q][threadIdx.x + st * SGP];
        }
        __syncthreads();
    }
    const int slot = A * gridDim.y + blockIdx.y;
    part += (int64_t)slot * PSPLIT * 4 * SGP;
    if (threadIdx.x < 4 * SGP) part[piece * 4 * SGP + threadIdx.x] = red[threadIdx.x % 4][threadIdx.x / 4];
    if (last_part(count + slot, PSPLIT) && threadIdx.x < 4 * SGP) {
        T t = 0;
#pragma unroll
        for (int k = 0; k < PSPLIT; ++k) t += __ldcg(part + k * 4 * SGP + threadIdx.x);
        cproj[((int64_t)A * nb + sg0) * 4 + threadIdx.x] = __ldg(d.E + 4 * A + threadIdx.x % 4) * d.dV * t;
    }
}

#ifndef RS_PROJ_CTAS
#define RS_PROJ_CTAS 4
#endif

// FP32 blocks of 32-state groups: lane l of a warp takes sphere entry
// l / 8 of the warp's four and the states 4 (l % 8) .. + 3 (one 16-byte
// load of the psi row), so a warp reads four psi rows per step, four steps
// at a time; the point indices are read one round ahead of their rows.  The
// grid is (atoms * split,
// state groups) with the split sized to fill the GPU.  SUM: the last part adds
// them up; else (the ring kernel, whose CTAs read few atoms each) the reader
// does, which spares the fences at the kernel's end, 2.3 us a block.
constexpr int NTP4 = 256;

template <bool SUM>
__global__ void __launch_bounds__(NTP4, RS_PROJ_CTAS) k_project_f32(HamDev<float> d, const float *__restrict__ psi, int64_t ldp, int nb,
                                                     int split, float *part, unsigned *count, float *__restrict__ cproj) {
    constexpr int STEP = 4 * (NTP4 / 32), UN = 4;
    __shared__ float red[NTP4 / 32][8][16];
    const int A = blockIdx.x / split, piece = blockIdx.x - A * split;
    const int sg0 = blockIdx.y * 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, q = lane & 7;
    const int o = __ldg(d.sph_off + A), e = __ldg(d.sph_off + A + 1);
    const int per = (e - o + split - 1) / split;
    const int i0 = o + piece * per, i1 = min(e, i0 + per);
    const float *ps = psi + sg0 + 4 * q;
    float acc[16];   // [projector][state]
#pragma unroll
    for (int k = 0; k < 16; ++k) acc[k] = 0.f;
    int i = i0 + 4 * warp + (lane >> 3);
    int p[UN];
#pragma unroll
    for (int u = 0; u < UN; ++u) p[u] = i + u * STEP < i1 ? __ldg(d.sph_idx + i + u * STEP) : -1;
    pdl_wait();
    pdl_launch();
    for (; i < i1; i += UN * STEP) {
        float4 v[UN], g[UN];
#pragma unroll
        for (int u = 0; u < UN; ++u) {
            v[u] = g[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (p[u] >= 0) {
                v[u] = ld_fresh(reinterpret_cast<const float4 *>(ps + (int64_t)p[u] * ldp));
                g[u] = __ldg(reinterpret_cast<const float4 *>(d.sph_gam) + i + u * STEP);
            }
        }
#pragma unroll
        for (int u = 0; u < UN; ++u) {
            const int n = i + (UN + u) * STEP;
            p[u] = n < i1 ? __ldg(d.sph_idx + n) : -1;
        }
#pragma unroll
        for (int u = 0; u < UN; ++u) {
            const float gv[4] = {g[u].x, g[u].y, g[u].z, g[u].w}, vv[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
            for (int l = 0; l < 4; ++l)
#pragma unroll
                for (int st = 0; st < 4; ++st) acc[4 * l + st] = fmaf(gv[l], vv[st], acc[4 * l + st]);
        }
    }
    // the four entries of a warp, then the warps
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], 8);
        acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], 16);
    }
    if (lane < 8) {
#pragma unroll
        for (int k = 0; k < 16; ++k) red[warp][q][k] = acc[k];
    }
    __syncthreads();
    // thread t < 128: state t / 4 of the group, projector t % 4
    const int slot = A * gridDim.y + blockIdx.y, l = threadIdx.x & 3, st = threadIdx.x >> 2;
    part += (int64_t)slot * split * 128;
    if (threadIdx.x < 128) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < NTP4 / 32; ++w) t += red[w][st >> 2][4 * l + (st & 3)];
        part[piece * 128 + threadIdx.x] = __ldg(d.E + 4 * A + l) * d.dV * t;
    }
    if constexpr (SUM)
        if (last_part(count + slot, split) && threadIdx.x < 128) {
            float t = 0.f;
            for (int k = 0; k < split; ++k) t += __ldcg(part + k * 128 + threadIdx.x);
            cproj[((int64_t)A * nb + sg0) * 4 + threadIdx.x] = t;
        }
}

// ------------------------------------------- fused stencil + V + nonlocal ---

// V states of one point, read and written as one access.
template <typename T, int V> struct __align__(sizeof(T) * V) Pack { T v[V]; };

template <typename T, int V> __device__ __forceinline__ void add_to(Pack<T, V> &a, const Pack<T, V> &b) {
    if constexpr (sizeof(T) == 4 && V % 2 == 0) {
#pragma unroll
        for (int i = 0; i < V; i += 2) {
            const float2 r = __fadd2_rn(make_float2(a.v[i], a.v[i + 1]), make_float2(b.v[i], b.v[i + 1]));
            a.v[i] = r.x;
            a.v[i + 1] = r.y;
        }
    } else {
#pragma unroll
        for (int i = 0; i < V; ++i) a.v[i] += b.v[i];
    }
}
template <typename T, int V> __device__ __forceinline__ void fma_to(Pack<T, V> &acc, T w, const Pack<T, V> &b) {
    if constexpr (sizeof(T) == 4 && V % 2 == 0) {
#pragma unroll
        for (int i = 0; i < V; i += 2) {
            const float2 r = __ffma2_rn(make_float2(w, w), make_float2(b.v[i], b.v[i + 1]), make_float2(acc.v[i], acc.v[i + 1]));
            acc.v[i] = r.x;
            acc.v[i + 1] = r.y;
        }
    } else {
#pragma unroll
        for (int i = 0; i < V; ++i) acc.v[i] = fma(w, b.v[i], acc.v[i]);
    }
}

// A CTA takes PTS consecutive points in storage order.  First the 24 neighbour
// indices of every point go from the point map to shared memory (four along
// one direction at a time); then LPP lanes a point, V states a lane, read the 24
// rows, sum the six at each distance, and add the potential and the nonlocal
// terms.  The rows come from L1 and L2: points that follow one another in
// storage are lattice neighbours, so a CTA's rows overlap.
// Why no march with register queues (the kernel before this one): a march
// needs long columns per CTA, which left most SMs without work on small grids
// and one CTA of latency-bound steps on each of the others.  Measured, us per
// block, march -> gather: 103 331 points, FP32 16 states 68 -> 15.7, FP64 16
// states 699 -> 115; 654 520 points, FP32 16 states 273 -> 91, FP64 32 states
// 2338 -> 1211 (1060 at the FP64 pipe's rate, 25 operations per value: bound
// by that pipe; the FP32 blocks by the rows' way from L2).
constexpr int GT_NT = 256;
template <typename T, int V, int LPP> struct GatherCfg {
    static constexpr int PP = GT_NT / LPP;                 // points per pass
    static constexpr int PTS = PP > 64 ? PP : 64;
};

template <typename T, int V, int LPP>
__global__ void __launch_bounds__(GT_NT) k_gather(HamDev<T> d, const int32_t *__restrict__ loc, int npts,
                                                  const T *__restrict__ psi, int64_t ldp, T *__restrict__ hpsi, int64_t ldh,
                                                  const T *__restrict__ cproj, int nb) {
    using C = GatherCfg<T, V, LPP>;
    using P = Pack<T, V>;
    __shared__ int4 nbr[6][C::PTS];
    const int tid = threadIdx.x;
    const int p0 = blockIdx.x * C::PTS;
    const int np = min(C::PTS, npts - p0);
    const int strides[3] = {d.d1 * d.d2, d.d2, 1};
    for (int e = tid; e < 6 * C::PTS; e += GT_NT) {
        const int g = e / C::PTS, q = e - g * C::PTS;
        if (q >= np) continue;
        const int st = (g & 1) ? -strides[g >> 1] : strides[g >> 1];
        const int32_t *m = d.map + __ldg(loc + p0 + q);
        nbr[g][q] = make_int4(__ldg(m + st), __ldg(m + 2 * st), __ldg(m + 3 * st), __ldg(m + 4 * st));
    }
    __syncthreads();
    pdl_wait();
    const int lane = tid % LPP;
    const T *ps = psi + lane * V;
    for (int q = tid / LPP; q < C::PTS; q += C::PP) {
        if (q >= np) break;
        int id[6][4];
        bool all = true;
#pragma unroll
        for (int g = 0; g < 6; ++g) {
            const int4 n = nbr[g][q];
            id[g][0] = n.x, id[g][1] = n.y, id[g][2] = n.z, id[g][3] = n.w;
            all = all && (n.x | n.y | n.z | n.w) >= 0;
        }
        const int p = p0 + q;
        const int4 inf = ld_fresh(d.pinfo + p);
        const P c = ld_fresh(reinterpret_cast<const P *>(ps + (int64_t)p * ldp));
        // from the smallest weight to the largest, so that the roundings of the
        // large terms come last
        P acc;
#pragma unroll
        for (int i = 0; i < V; ++i) acc.v[i] = T(0);
        if (all) {
#pragma unroll
            for (int j = 3; j >= 0; --j) {
                P n[6];
#pragma unroll
                for (int g = 0; g < 6; ++g) n[g] = ld_fresh(reinterpret_cast<const P *>(ps + (int64_t)id[g][j] * ldp));
                add_to(n[0], n[1]);
                add_to(n[2], n[3]);
                add_to(n[4], n[5]);
                add_to(n[0], n[2]);
                add_to(n[0], n[4]);
                fma_to(acc, d.w[j + 1], n[0]);
            }
        } else {
            // a neighbour off the grid contributes nothing
#pragma unroll
            for (int j = 3; j >= 0; --j) {
                P n[6];
#pragma unroll
                for (int g = 0; g < 6; ++g) {
#pragma unroll
                    for (int i = 0; i < V; ++i) n[g].v[i] = T(0);
                    if (id[g][j] >= 0) n[g] = ld_fresh(reinterpret_cast<const P *>(ps + (int64_t)id[g][j] * ldp));
                }
                add_to(n[0], n[1]);
                add_to(n[2], n[3]);
                add_to(n[4], n[5]);
                add_to(n[0], n[2]);
                add_to(n[0], n[4]);
                fma_to(acc, d.w[j + 1], n[0]);
            }
        }
        fma_to(acc, d.w[0], c);
        fma_to(acc, point_v<T>(inf), c);
        for (int e = inf.x; e < inf.y; ++e) {
            const int A = __ldg(d.cov_atom + e);
            const Four<T> g = load4(d.cov_gam + 4 * (int64_t)e);
            const T *cp = cproj + ((int64_t)A * nb + lane * V) * 4;
#pragma unroll
            for (int i = 0; i < V; ++i) {
                const Four<T> c4 = fresh4(cp + 4 * i);
                acc.v[i] += g.a * c4.a + g.b * c4.b + g.c * c4.c + g.d * c4.d;
            }
        }
        *reinterpret_cast<P *>(hpsi + (int64_t)p * ldh + lane * V) = acc;
    }
}

// ----------------------------------------------- face-neighbour filter ---
// W = alpha R + beta sum_{6 face neighbours} R (zero off the grid); one thread
// per (point, state), state fastest.
template <typename T>
__global__ void k_filter(const int32_t *__restrict__ map, const int32_t *__restrict__ loc, int64_t npts, int d1, int d2,
                         const T *__restrict__ R, int64_t ldr, T *__restrict__ W, int64_t ldw, int nb, T alpha,
                         T beta) {
    // block (nb, 256 / nb): threadIdx.x is the state, threadIdx.y the point
    const int s = threadIdx.x;
    const int64_t p = blockIdx.x * (int64_t)blockDim.y + threadIdx.y;
    if (p >= npts) return;
    const int64_t L = __ldg(loc + p);
    const int64_t plane = (int64_t)d1 * d2;
    const int64_t offs[6] = {1, -1, d2, -(int64_t)d2, plane, -plane};
    T acc = 0;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const int q = __ldg(map + L + offs[k]);
        if (q >= 0) acc += __ldg(R + (int64_t)q * ldr + s);
    }
    W[p * ldw + s] = alpha * __ldg(R + p * ldr + s) + beta * acc;
}

}  // namespace rs

using namespace rs;

// ------------------------------------------------------------ host side ---

struct rs_ham {
    int64_t npts = 0;
    int32_t d[3] = {0, 0, 0};
    double h = 0, dV = 0;
    int order = 4;
    int n_atoms = 0;
    int64_t n_entries = 0;
    int device = 0;
    int n_sm = 1;                  // SMs of the device (grid sizing)
    double w[5] = {0, 0, 0, 0, 0};
    DevBuf pinfo64, pinfo32, map, loc, V64, V32, cov_off, cov_atom, cov_gam64, cov_gam32, sph_off, sph_idx, sph_gam64, sph_gam32, E64, E32,
        cproj, cpart, ccount, dummy, scratch;
    RingPlan *ring = nullptr;      // tables of the ring-buffer FP32 kernel (nullptr: not usable)
    int kernel = RS_KERNEL_AUTO;   // rs_ham_select_kernel
    // optional per-launch timing (rs_ham_timing)
    bool timing = false;
    std::vector<cudaEvent_t> events;   // 3 per recorded call
    size_t n_recorded = 0;
    ~rs_ham() {
        ring_plan_destroy(ring);
        for (cudaEvent_t e : events) cudaEventDestroy(e);
    }
    // events for the next recorded call (nullptr when timing is off)
    cudaEvent_t *next_events() {
        if (!timing) return nullptr;
        if (events.size() < 3 * (n_recorded + 1)) {
            for (int i = 0; i < 3; ++i) {
                cudaEvent_t e;
                if (cudaEventCreate(&e) != cudaSuccess) return nullptr;
                events.push_back(e);
            }
        }
        return &events[3 * n_recorded++];
    }
    template <typename T> HamDev<T> view() const;
    // parts of an atom's sphere in k_project_f32: one wave of at most
    // RS_PROJ_CTAS CTAs of 256 threads per SM in all
    int proj_split() const { return std::max(1, std::min(64, RS_PROJ_CTAS * n_sm / std::max(1, n_atoms))); }
};

template <> HamDev<double> rs_ham::view<double>() const {
    HamDev<double> v;
    v.pinfo = pinfo64.as<int4>();
    v.map = map.as<int32_t>();
    v.d0 = d[0], v.d1 = d[1], v.d2 = d[2];
    v.V = V64.as<double>();
    v.cov_off = cov_off.as<int32_t>();
    v.cov_atom = cov_atom.as<int32_t>();
    v.cov_gam = cov_gam64.as<double>();
    v.sph_off = sph_off.as<int32_t>();
    v.sph_idx = sph_idx.as<int32_t>();
    v.sph_gam = sph_gam64.as<double>();
    v.E = E64.as<double>();
    v.dV = dV;
    for (int j = 0; j < 5; ++j) v.w[j] = w[j];
    return v;
}
template <> HamDev<float> rs_ham::view<float>() const {
    HamDev<float> v;
    v.pinfo = pinfo32.as<int4>();
    v.map = map.as<int32_t>();
    v.d0 = d[0], v.d1 = d[1], v.d2 = d[2];
    v.V = V32.as<float>();
    v.cov_off = cov_off.as<int32_t>();
    v.cov_atom = cov_atom.as<int32_t>();
    v.cov_gam = cov_gam32.as<float>();
    v.sph_off = sph_off.as<int32_t>();
    v.sph_idx = sph_idx.as<int32_t>();
    v.sph_gam = sph_gam32.as<float>();
    v.E = E32.as<float>();
    v.dV = (float)dV;
    for (int j = 0; j < 5; ++j) v.w[j] = (float)w[j];
    return v;
}

// Central second-derivative weights of half-width m (closed form):
// c_j = 2 (-1)^(j+1) (m!)^2 / (j^2 (m-j)! (m+j)!), c_0 = -2 sum_{j>=1} c_j.
static void fd_weights(int m, double c[5]) {
    auto fact = [](int n) {
        double f = 1;
        for (int i = 2; i <= n; ++i) f *= i;
        return f;
    };
    for (int j = 0; j < 5; ++j) c[j] = 0;
    double sum = 0;
    for (int j = 1; j <= m; ++j) {
        c[j] = 2.0 * ((j & 1) ? 1.0 : -1.0) * fact(m) * fact(m) / ((double)j * j * fact(m - j) * fact(m + j));
        sum += c[j];
    }
    c[0] = -2.0 * sum;
}

extern "C" int rs_ham_create(const rs_grid *g, const double *V_host, const rs_proj *pr, int order, rs_ham **out) {
    if (!g || !V_host || !out) return fail(RS_EINVAL, "rs_ham_create: null argument");
    if (order < 1 || order > 4) return fail(RS_EINVAL, "rs_ham_create: order must be in 1..4");
    *out = nullptr;
    int dev = 0;
    RS_CUDA(cudaGetDevice(&dev));
    rs_ham *H = new (std::nothrow) rs_ham;
    if (!H) return fail(RS_ENOMEM, "host allocation failed");
    auto bail = [&](int rc) {
        delete H;
        return rc;
    };
    H->device = dev;
    if (cudaDeviceGetAttribute(&H->n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || H->n_sm < 1)
        return bail(fail(RS_ECUDA, "device query failed"));
    H->npts = g->npts;
    for (int i = 0; i < 3; ++i) H->d[i] = g->dims[i];
    H->h = g->h;
    H->dV = g->h * g->h * g->h;
    H->order = order;
    double c[5];
    fd_weights(order, c);
    const double kin = -0.5 / (g->h * g->h);
    H->w[0] = 3.0 * kin * c[0];
    for (int j = 1; j < 5; ++j) H->w[j] = kin * c[j];

    int rc;
    const int64_t np = g->npts;
    if ((rc = H->map.upload(g->map.data(), g->map.size() * sizeof(int32_t)))) return bail(rc);
    {
        std::vector<int32_t> loc((size_t)g->npts);
        for (int64_t p = 0; p < g->npts; ++p)
            loc[p] = (int32_t)(((int64_t)(g->ijk[3 * p] - g->origin[0]) * g->dims[1] + (g->ijk[3 * p + 1] - g->origin[1])) *
                                   g->dims[2] + (g->ijk[3 * p + 2] - g->origin[2]));
        if ((rc = H->loc.upload(loc.data(), loc.size() * sizeof(int32_t)))) return bail(rc);
    }
    std::vector<float> v32((size_t)np);
    for (int64_t p = 0; p < np; ++p) v32[p] = (float)V_host[p];
    if ((rc = H->V64.upload(V_host, (size_t)np * sizeof(double)))) return bail(rc);
    if ((rc = H->V32.upload(v32.data(), (size_t)np * sizeof(float)))) return bail(rc);

    // projector tables: atom-major (projection) and point-major (gather)
    const int na = pr ? pr->n_atoms : 0;
    const int64_t ne = pr ? (int64_t)pr->idx.size() : 0;
    if (ne > (int64_t)INT32_MAX) return bail(fail(RS_EINVAL, "too many projector entries"));
    H->n_atoms = na;
    H->n_entries = ne;
    std::vector<int32_t> soff((size_t)na + 1, 0), coff((size_t)np + 1, 0), catom((size_t)std::max<int64_t>(ne, 1));
    std::vector<double> cg64((size_t)std::max<int64_t>(ne, 1) * 4), sg64((size_t)std::max<int64_t>(ne, 1) * 4),
        E64((size_t)std::max(na, 1) * 4);
    for (int A = 0; A < na; ++A) soff[A + 1] = (int32_t)pr->off[A + 1];
    for (int64_t e = 0; e < ne; ++e) coff[(size_t)pr->idx[e] + 1]++;
    for (int64_t p = 0; p < np; ++p) coff[p + 1] += coff[p];
    {
        std::vector<int32_t> fill(coff.begin(), coff.end() - 1);
        for (int A = 0; A < na; ++A)
            for (int64_t e = pr->off[A]; e < pr->off[A + 1]; ++e) {
                const int32_t slot = fill[pr->idx[e]]++;
                catom[slot] = A;
                for (int q = 0; q < 4; ++q) cg64[(size_t)slot * 4 + q] = pr->gam[e * 4 + q];
            }
    }
    for (int64_t e = 0; e < ne * 4; ++e) sg64[e] = pr->gam[e];
    for (int A = 0; A < na * 4; ++A) E64[A] = pr->E[A];
    std::vector<float> cg32(cg64.begin(), cg64.end()), sg32(sg64.begin(), sg64.end()), E32(E64.begin(), E64.end());
    std::vector<int32_t> sidx(pr && ne ? pr->idx : std::vector<int32_t>(1, 0));
    if ((rc = H->sph_off.upload(soff.data(), soff.size() * 4)) || (rc = H->sph_idx.upload(sidx.data(), sidx.size() * 4)) ||
        (rc = H->sph_gam64.upload(sg64.data(), sg64.size() * 8)) ||
        (rc = H->sph_gam32.upload(sg32.data(), sg32.size() * 4)) || (rc = H->E64.upload(E64.data(), E64.size() * 8)) ||
        (rc = H->E32.upload(E32.data(), E32.size() * 4)) || (rc = H->cov_off.upload(coff.data(), coff.size() * 4)) ||
        (rc = H->cov_atom.upload(catom.data(), catom.size() * 4)) ||
        (rc = H->cov_gam64.upload(cg64.data(), cg64.size() * 8)) ||
        (rc = H->cov_gam32.upload(cg32.data(), cg32.size() * 4)))
        return bail(rc);
    if ((rc = H->cproj.alloc((size_t)std::max(na, 1) * 4 * 64 * sizeof(double)))) return bail(rc);
    {
        // partial sums: PSPLIT parts of 64 FP64 states, or as many FP32 parts as proj_split allows
        const size_t a64 = (size_t)std::max(na, 1) * PSPLIT * 4 * 64 * sizeof(double);
        const size_t a32 = (size_t)std::max(na, 1) * H->proj_split() * 4 * 64 * sizeof(float);
        if ((rc = H->cpart.alloc(std::max(a64, a32)))) return bail(rc);
        // one count per atom and state group (at most two groups)
        if ((rc = H->ccount.alloc((size_t)std::max(na, 1) * 2 * sizeof(unsigned)))) return bail(rc);
        if (cudaMemset(H->ccount.p, 0, (size_t)std::max(na, 1) * 2 * sizeof(unsigned)) != cudaSuccess)
            return bail(fail(RS_ECUDA, "cudaMemset failed"));
    }
    {
        std::vector<int4> p64((size_t)np), p32((size_t)np);
        for (int64_t p = 0; p < np; ++p) {
            int64_t bits;
            memcpy(&bits, &V_host[p], 8);
            int32_t fbits;
            memcpy(&fbits, &v32[p], 4);
            p64[p] = make_int4(coff[p], coff[p + 1], (int32_t)(bits & 0xffffffffll), (int32_t)(bits >> 32));
            p32[p] = make_int4(coff[p], coff[p + 1], fbits, 0);
        }
        if ((rc = H->pinfo64.upload(p64.data(), p64.size() * sizeof(int4))) ||
            (rc = H->pinfo32.upload(p32.data(), p32.size() * sizeof(int4))))
            return bail(rc);
    }
#if RS_STENCIL_RING
    if ((rc = ring_plan_build(&H->ring, g, coff, catom, cg32, v32, (float)H->w[0], na, RS_RING_SLAB))) return bail(rc);
#endif
    *out = H;
    return RS_OK;
}

extern "C" int rs_ham_destroy(rs_ham *h) {
    delete h;
    return RS_OK;
}

// nb states of the block, V to a lane (16-byte accesses where the rows allow it)
template <typename T, int V, int LPP>
static int launch_gather(rs_ham *H, const HamDev<T> &d, const T *psi, int64_t ldp, T *hpsi, int64_t ldh, int nb,
                         cudaStream_t st) {
    constexpr int PTS = GatherCfg<T, V, LPP>::PTS;
    return launch_overlapped(k_gather<T, V, LPP>, dim3((unsigned)((H->npts + PTS - 1) / PTS)), GT_NT, 0, st, d,
                             H->loc.as<int32_t>(), (int)H->npts, psi, ldp, hpsi, ldh, H->cproj.as<T>(), nb);
}

template <typename T>
static int apply_t(rs_ham *H, const T *psi, int64_t ldp, T *hpsi, int64_t ldh, int nb, cudaStream_t st) {
    const HamDev<T> d = H->view<T>();
    cudaEvent_t *ev = H->next_events();
    if (ev) RS_CUDA(cudaEventRecord(ev[0], st));
    bool ring = false;
    if constexpr (sizeof(T) == 4) ring = H->kernel == RS_KERNEL_AUTO && ring_usable(H->ring, psi, ldp, ldh, nb);
    if (H->n_atoms > 0) {
        const int sgp = std::min(nb, 32);
        const dim3 grid((unsigned)(H->n_atoms * PSPLIT), (unsigned)(nb / sgp));
        T *cp = H->cproj.as<T>(), *part = H->cpart.as<T>();
        unsigned *cnt = H->ccount.as<unsigned>();
        bool done = false;
        if constexpr (sizeof(T) == 4) {
            if (nb % 32 == 0 && ldp % 4 == 0 && aligned16(psi)) {
                const int split = H->proj_split();
                RS_TRY(launch_overlapped(ring ? k_project_f32<false> : k_project_f32<true>, dim3((unsigned)(H->n_atoms * split), (unsigned)(nb / 32)), NTP4, 0, st,
                                         d, psi, ldp, nb, split, part, cnt, cp));
                done = true;
            }
        }
        if (!done) switch (sgp) {
            case 1: RS_TRY(launch_overlapped(k_project<T, 1, 512>, grid, 512, 0, st, d, psi, ldp, nb, part, cnt, cp)); break;
            case 2: RS_TRY(launch_overlapped(k_project<T, 2, 512>, grid, 512, 0, st, d, psi, ldp, nb, part, cnt, cp)); break;
            case 4: RS_TRY(launch_overlapped(k_project<T, 4, 512>, grid, 512, 0, st, d, psi, ldp, nb, part, cnt, cp)); break;
            case 8: RS_TRY(launch_overlapped(k_project<T, 8, 512>, grid, 512, 0, st, d, psi, ldp, nb, part, cnt, cp)); break;
            case 16: RS_TRY(launch_overlapped(k_project<T, 16, 512>, grid, 512, 0, st, d, psi, ldp, nb, part, cnt, cp)); break;
            default: RS_TRY(launch_overlapped(k_project<T, 32, 512>, grid, 512, 0, st, d, psi, ldp, nb, part, cnt, cp)); break;
        }
    }
    if (ev) RS_CUDA(cudaEventRecord(ev[1], st));
    int rc = -1;
    if constexpr (sizeof(T) == 4)
        if (ring) {
            float w[5];
            for (int j = 0; j < 5; ++j) w[j] = (float)H->w[j];
            rc = ring_launch(H->ring, psi, ldp, hpsi, ldh, H->cpart.as<float>(), H->proj_split(), nb, w, st);
        }
    constexpr int E = 16 / (int)sizeof(T);   // states per 16 bytes
    if (!ring) switch (nb) {
        case 1: rc = launch_gather<T, 1, 1>(H, d, psi, ldp, hpsi, ldh, nb, st); break;
        case 2: rc = launch_gather<T, 2, 1>(H, d, psi, ldp, hpsi, ldh, nb, st); break;
        case 4: rc = launch_gather<T, E, 4 / E>(H, d, psi, ldp, hpsi, ldh, nb, st); break;
        case 8: rc = launch_gather<T, E, 8 / E>(H, d, psi, ldp, hpsi, ldh, nb, st); break;
        case 16: rc = launch_gather<T, E, 16 / E>(H, d, psi, ldp, hpsi, ldh, nb, st); break;
        case 32: rc = launch_gather<T, E, 32 / E>(H, d, psi, ldp, hpsi, ldh, nb, st); break;
        case 64: rc = launch_gather<T, E, 64 / E>(H, d, psi, ldp, hpsi, ldh, nb, st); break;
        default: return fail(RS_EINVAL, "unsupported state group");
    }
    if (rc == RS_OK && ev) RS_CUDA(cudaEventRecord(ev[2], st));
    return rc;
}

extern "C" int rs_ham_apply_block(rs_ham *h, const void *psi_dev, int64_t ld_psi, void *hpsi_dev, int64_t ld_hpsi,
                                  int nb, int dtype, void *stream) {
    if (!h || !psi_dev || !hpsi_dev) return fail(RS_EINVAL, "rs_ham_apply_block: null argument");
    if (nb < 1 || nb > 64 || (nb & (nb - 1))) return fail(RS_EINVAL, "rs_ham_apply_block: nb must be a power of two <= 64");
    if (ld_psi < nb || ld_hpsi < nb) return fail(RS_EINVAL, "rs_ham_apply_block: ld < nb");
    if (dtype != RS_F64 && dtype != RS_F32) return fail(RS_EINVAL, "rs_ham_apply_block: bad dtype");
    const int es = dtype == RS_F64 ? 8 : 4;
    const int sgbytes = std::min(nb, 128 / es) * es;
    const int need = std::min(sgbytes, 16);
    if (((uintptr_t)psi_dev % need) || ((uintptr_t)hpsi_dev % need) || ((ld_psi * es) % need) || ((ld_hpsi * es) % need))
        return fail(RS_EINVAL, "rs_ham_apply_block: misaligned pointer or leading dimension");
    const char *a = (const char *)psi_dev, *b = (const char *)hpsi_dev;
    const int64_t span_a = ((h->npts - 1) * ld_psi + nb) * es, span_b = ((h->npts - 1) * ld_hpsi + nb) * es;
    if (a < b + span_b && b < a + span_a) return fail(RS_EINVAL, "rs_ham_apply_block: psi and hpsi overlap");
    cudaStream_t st = (cudaStream_t)stream;
    if (dtype == RS_F64)
        return apply_t<double>(h, (const double *)psi_dev, ld_psi, (double *)hpsi_dev, ld_hpsi, nb, st);
    return apply_t<float>(h, (const float *)psi_dev, ld_psi, (float *)hpsi_dev, ld_hpsi, nb, st);
}

extern "C" int64_t rs_ham_apply_bytes(const rs_ham *h, int nb, int dtype) {
    // psi read once, hpsi written once, V and the point map, one copy of the
    // projector tables and the coefficients: the bytes of the fused launch
    // (the projection pass re-reads rows that stay in L2 and its own copy of
    // the tables, which are not counted again)
    int64_t b = 0;
    if (rs_ham_launch_bytes(h, nb, dtype, nullptr, &b) != RS_OK) return -1;
    return b;
}

extern "C" int rs_ham_launch_bytes(const rs_ham *h, int nb, int dtype, int64_t *project_bytes, int64_t *stencil_bytes) {
    if (!h) return fail(RS_EINVAL, "rs_ham_launch_bytes: null handle");
    const int64_t s = dtype == RS_F64 ? 8 : 4;
    const int64_t np = h->npts, ne = h->n_entries, nc = (int64_t)h->n_atoms * 4 * nb * s;
    if (project_bytes) *project_bytes = ne * (4 + 4 * s) + (h->n_atoms + 1) * 4 + nc;
    if (stencil_bytes) *stencil_bytes = np * nb * 2 * s + np * s + np * 4 + ne * (4 + 4 * s) + (np + 1) * 4 + nc;
    return RS_OK;
}

extern "C" int rs_ham_status(rs_ham *h, int *flags) {
    if (!h || !flags) return fail(RS_EINVAL, "rs_ham_status: null argument");
    int f = 0;
    RS_TRY(ring_status(h->ring, &f));
    *flags = f;
    return RS_OK;
}

__global__ void k_set_potential(const double *__restrict__ V, int64_t np, double *__restrict__ V64,
                                float *__restrict__ V32, int4 *__restrict__ p64, int4 *__restrict__ p32) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < np; p += (int64_t)gridDim.x * blockDim.x) {
        const double v = V[p];
        const float f = __double2float_rn(v);
        V64[p] = v;
        V32[p] = f;
        const long long bits = __double_as_longlong(v);
        int4 a = p64[p];
        a.z = (int)(bits & 0xffffffffll);
        a.w = (int)(bits >> 32);
        p64[p] = a;
        int4 b = p32[p];
        b.z = __float_as_int(f);
        p32[p] = b;
    }
}

extern "C" int rs_ham_set_potential(rs_ham *h, const double *V_dev, void *stream) {
    if (!h || !V_dev) return fail(RS_EINVAL, "rs_ham_set_potential: null argument");
    cudaStream_t st = (cudaStream_t)stream;
    k_set_potential<<<(unsigned)std::min<int64_t>((h->npts + 255) / 256, 152 * 16), 256, 0, st>>>(
        V_dev, h->npts, h->V64.as<double>(), h->V32.as<float>(), h->pinfo64.as<int4>(), h->pinfo32.as<int4>());
    RS_LAUNCH_CHECK();
    return ring_set_potential(h->ring, h->V32.as<float>(), st);
}

extern "C" int rs_ham_select_kernel(rs_ham *h, int which) {
    if (!h || (which != RS_KERNEL_AUTO && which != RS_KERNEL_GENERIC)) return fail(RS_EINVAL, "rs_ham_select_kernel: bad argument");
    h->kernel = which;
    return RS_OK;
}

extern "C" int rs_ham_reset_status(rs_ham *h) {
    if (!h) return fail(RS_EINVAL, "rs_ham_reset_status: null handle");
    return ring_reset_status(h->ring);
}

extern "C" int rs_ham_set_wait_limit(rs_ham *h, int tests) {
    if (!h) return fail(RS_EINVAL, "rs_ham_set_wait_limit: null handle");
    ring_set_wait_limit(h->ring, tests);
    return RS_OK;
}

namespace rs {
int *ham_status_word(rs_ham *h) { return ring_status_word(h->ring); }
}  // namespace rs

extern "C" int rs_ham_timing(rs_ham *h, int enable) {
    if (!h) return fail(RS_EINVAL, "rs_ham_timing: null handle");
    if (enable) h->n_recorded = 0;
    h->timing = enable != 0;
    return RS_OK;
}

extern "C" int rs_ham_timing_read(rs_ham *h, double *project_ms, double *stencil_ms, int64_t *calls) {
    if (!h) return fail(RS_EINVAL, "rs_ham_timing_read: null handle");
    double pm = 0, sm = 0;
    for (size_t i = 0; i < h->n_recorded; ++i) {
        cudaEvent_t *e = &h->events[3 * i];
        RS_CUDA(cudaEventSynchronize(e[2]));
        float a = 0, b = 0;
        RS_CUDA(cudaEventElapsedTime(&a, e[0], e[1]));
        RS_CUDA(cudaEventElapsedTime(&b, e[1], e[2]));
        pm += a;
        sm += b;
    }
    if (project_ms) *project_ms = pm;
    if (stencil_ms) *stencil_ms = sm;
    if (calls) *calls = (int64_t)h->n_recorded;
    return RS_OK;
}

namespace rs {

int64_t ham_npts(const rs_ham *h) { return h->npts; }
const int32_t *ham_map(const rs_ham *h) { return h->map.as<int32_t>(); }
const int32_t *ham_loc(const rs_ham *h) { return h->loc.as<int32_t>(); }
int ham_dim(const rs_ham *h, int axis) { return h->d[axis]; }
DevBuf *ham_scratch(rs_ham *h, size_t bytes) {
    if (h->scratch.bytes >= bytes) return &h->scratch;
    if (h->scratch.alloc(bytes) != RS_OK) return nullptr;
    return &h->scratch;
}
double ham_dV(const rs_ham *h) { return h->dV; }

int ham_filter(const rs_ham *h, const void *R, int64_t ldr, void *W, int64_t ldw, int nb, int dtype, double alpha,
               cudaStream_t st) {
    const dim3 blk((unsigned)nb, (unsigned)std::max(1, 256 / nb));
    const unsigned blocks = (unsigned)((h->npts + blk.y - 1) / blk.y);
    const double beta = (1.0 - alpha) / 6.0;
    if (dtype == RS_F64)
        k_filter<double><<<blocks, blk, 0, st>>>(h->map.as<int32_t>(), h->loc.as<int32_t>(), h->npts, h->d[1], h->d[2],
                                                 (const double *)R, ldr, (double *)W, ldw, nb, alpha, beta);
    else
        k_filter<float><<<blocks, blk, 0, st>>>(h->map.as<int32_t>(), h->loc.as<int32_t>(), h->npts, h->d[1], h->d[2],
                                                (const float *)R, ldr, (float *)W, ldw, nb, (float)alpha, (float)beta);
    RS_LAUNCH_CHECK();
    return RS_OK;
}

}  // namespace rs
