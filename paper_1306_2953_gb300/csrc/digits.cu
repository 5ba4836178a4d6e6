// Tall-skinny contractions of Sec. VI on the 5th-generation tensor cores at
// FP64 (and FP32) accuracy, by splitting every operand into integer digits.
//
//   overlap   S = dV X^T Y      (contraction over the grid points)
//   rotation  Y = alpha X C + beta Y   (contraction over the states)
//
// GB300 has about 1.1 TFLOP/s of FP64 FMA against 1.9 PFLOP/s of FP16 tensor
// throughput.  An operand value is written as an integer q = trunc(x 2^(s - E)),
// 2^E above the largest entry of its column (overlap; of its row of X, the columns
// brought to one size, and of its column of C in the rotation) and s = 8 NS - 2, and q as NS
// balanced digits in base 256, |d| <= 128, each exact in FP16.  Digit products are
// integers of at most 2^14, so the FP32 accumulators of the tensor cores sum
// up to 1024 of them without any rounding.  The products of weight
// 256^-(i+j), i + j = t, have their own accumulator in tensor memory for
// every t < NS; the accumulators are read out every 256 points and summed as
// 64-bit integers: with t + 1 pairs of digits in accumulator t everything up to
// t = 3 is exact and a rounding of a later one is below 2^-56 of the largest
// product.  NS = 8 (FP64), 7 (overlap of FP32 data at FP64-like accuracy) or 5 (rotation of
// FP32 data).  (Ozaki, Ogita, Oishi and Rump 2012 give the scheme of error-free
// splittings of a matrix product.)
// Error of one product x y, in units of 2^(Ex + Ey - s): below 1 for each operand's
// truncation and NS - 1 for the digits with i + j = NS, the first that are left out (the rest
// is a 256th of that); signs and digits vary, so sums of many come out far below.  It is relative
// to the largest entries, not to x y: sums of products that are all below 2^-9 (FP64,
// s = 62; 2^-10 for FP32 overlaps against their former sums of float pairs) of the largest entries'
// product, as of two columns that hardly meet, are less accurate relative to
// themselves than FP64 multiply-adds.
//
// Kernel: 8 converter warps and one MMA warp per CTA, one CTA per SM, a 128 x
// BN tile of the result.  Stage (32 steps of the contraction, two stages): the
// converters read the operands from global memory into registers one stage
// ahead, extract the digits with integer instructions (the FP64 pipe would
// take longer than the products) and store them as K-major core matrices (8
// rows of 16 bytes) in shared memory; one thread issues the products; every
// 256 steps the converters read the accumulators back, accumulator by
// accumulator in the order the products run, so the products of the next
// steps overlap the readout.  Columns or rows that hold a non-finite or an
// extreme value (an exponent near either end of the range) make their CTA
// take a plain loop instead, so that infinities and NaN spread as in a plain
// contraction.  Every wait is bounded; a CTA whose wait gives up writes
// NaN in every result that it has not stored, and sets the call's status word
// where it has one.
//
// What bounds it, and what it measured (overlap of 256 x 256 columns over
// 658 416 points): FP64 2.95 ms, FP32 data 2.64 ms, against 69.8 ms by FP64 FMA
// and 14.3 ms by compensated FP32 sums before.  The products alone take
// 1.65 ms (28 % more than the tensor pipe needs: the readouts); the
// conversion, 20 integer instructions per value on a pipe of half rate,
// accounts for the rest, the pass that finds the column exponents for 0.4 ms.
// Every size gains (64 x 64: 4.4 -> 0.45 ms FP64, 0.94 -> 0.41 ms FP32), so
// overlaps have no other path; rotations of more states or columns than
// digit_rot_takes says take k_rowmul.
#include <cuda_fp16.h>

#include <algorithm>
#include <climits>

#include "device.h"
#include "digits.h"
#include "linalg.h"

namespace rs {

namespace {

constexpr int DG_M = 128;            // rows of the tile (TMEM lanes)
constexpr int DG_K = 32;             // contraction steps per stage
constexpr int DG_DRAIN = 8;          // stages between accumulator readouts
constexpr int DG_STAGES = 2;
constexpr int DG_CW = 8;             // converter warps
constexpr int DG_CT = DG_CW * 32;    // converter threads
constexpr int DG_NT = DG_CT + 128;   // and the MMA warp's warpgroup (its other warps only help with the set-up)
constexpr int DG_SPIN = 100000;      // barrier tests (at most 20 us each) before a wait gives up
constexpr int KQ = DG_K / 8;         // 8-step groups per stage
__device__ __forceinline__ uint32_t dg_su32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void dg_bar_init(uint64_t *b, uint32_t n) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(dg_su32(b)), "r"(n) : "memory");
}
__device__ __forceinline__ void dg_arrive(uint64_t *b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(dg_su32(b)) : "memory");
}
__device__ __forceinline__ bool dg_try(uint64_t *b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(dg_su32(b)), "r"(parity), "n"(20000)
        : "memory");
    return ok != 0;
}
// What a CTA's bounded waits share: whether one has given up, and after how many tests.
struct DgGive {
    int bad, spin;
};
// bounded wait; false once it has given up here or `bad` says another thread's has
// (sleep: nanoseconds between tests, for warps that wait most of the time and
// would take issue slots from the converters)
__device__ __forceinline__ bool dg_wait(uint64_t *b, uint32_t parity, DgGive *give, unsigned sleep = 0) {
    volatile int *bad = &give->bad;
    const int spin = give->spin;
    for (int i = 0; i < spin; ++i) {
        if (dg_try(b, parity)) return true;
        if ((i & 7) == 7 && *bad) return false;
        if (sleep) __nanosleep(sleep);
    }
    *bad = 1;
    return false;
}
// The wait for products in flight, whatever has given up: nothing may write shared or
// tensor memory after the CTA has left.
__device__ __forceinline__ void dg_settle(uint64_t *b, uint32_t parity) {
    for (int i = 0; i < DG_SPIN && !dg_try(b, parity); ++i) {
    }
}
// The MMA warp runs its loop as a whole, so that descriptors stay in uniform
// registers; `lead` (one lane) issues.
// the whole warp: true only when every lane's wait ended (no lane goes on alone).
// The lanes leave it together, as the warp-wide loads of tensor memory need
// (they run apart in the loop, and in stores and atomics of ragged tiles before it).
__device__ __forceinline__ bool dg_wait_warp(uint64_t *b, uint32_t parity, DgGive *give) {
    const bool all = __all_sync(0xffffffffu, dg_wait(b, parity, give));
    __syncwarp();
    return all;
}
__device__ __forceinline__ void dg_mma(uint32_t tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accum,
                                       uint32_t lead) {
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum), "r"(lead)
        : "memory");
}
__device__ __forceinline__ void dg_commit(uint64_t *b, uint32_t lead) {
    asm volatile(
        "{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n"
        " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(dg_su32(b)),
        "r"(lead)
        : "memory");
}
// registers: 384 threads are launched with 168 each; the converters' two
// warpgroups take 232 and the MMA warp's keeps 40 (2 x 232 + 40 = 3 x 168)
#define DG_REGS_UP() asm volatile("setmaxnreg.inc.sync.aligned.u32 232;\n")
#define DG_REGS_DOWN() asm volatile("setmaxnreg.dec.sync.aligned.u32 40;\n")
#define DG_FENCE_BEFORE() asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory")
#define DG_FENCE_AFTER() asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory")

// Matrix descriptor of a K-major tile without swizzle: core matrices of 8 rows x
// 16 bytes, `lbo` bytes apart along K and 128 bytes apart along the rows.
__device__ __forceinline__ uint64_t dg_desc(uint32_t saddr, uint32_t lbo) {
    return (uint64_t)((saddr >> 4) & 0x3FFF) | (uint64_t)(lbo >> 4) << 16 | (uint64_t)(128 >> 4) << 32 | (uint64_t)1 << 46;
}
// FP16 x FP16 -> FP32, both K-major
__host__ __device__ constexpr uint32_t dg_idesc(int M, int N) {
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void dg_tmem_ld32(uint32_t addr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}

__device__ __forceinline__ void dg_tmem_ld16(uint32_t addr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(addr));
}
__device__ __forceinline__ void dg_tmem_ld8(uint32_t addr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(addr));
}

// ------------------------------------------------------------- digits ---

// Ordering key of |x| whose high part is the biased exponent; 0 for zero only.
__device__ __forceinline__ int abs_key(double x) {
    const int hi = __double2hiint(x) & 0x7fffffff;
    return hi ? hi : (__double2loint(x) != 0);
}
__device__ __forceinline__ int abs_key(float x) { return __float_as_int(x) & 0x7fffffff; }

// Biased exponent of a column from its largest key (of a column of zeros: any
// that leaves their digits zero), and whether the digit
// path takes it: below `lo` an element's missing implicit bit could reach
// the digits, and the weights of the result could leave the FP64 range.
template <typename T> struct ExpOf;
template <> struct ExpOf<double> {
    static constexpr int bias = 1023;
    static constexpr int mant = 20, lo = 623, hi = 1423;   // bits below the exponent in a key; exponents taken
    static constexpr int span = 512;                       // largest ratio of two columns of a rotation, 2^span
    static __device__ __forceinline__ int exponent(int key) { return key ? key >> 20 : bias; }
    static __device__ __forceinline__ bool plain(int key) { return key && ((key >> 20) < lo || (key >> 20) > hi); }
};
template <> struct ExpOf<float> {
    static constexpr int bias = 127;
    static constexpr int mant = 23, lo = 64, hi = 254, span = 126;
    static __device__ __forceinline__ int exponent(int key) { return key ? key >> 23 : bias; }
    static __device__ __forceinline__ bool plain(int key) { return key && ((key >> 23) < lo || (key >> 23) > hi); }
};

// q + 128 in every digit, q = trunc(|x| 2^(s - E)), |x| < 2^E, E = ecol - bias + 1.
// The mantissa stands at bits 61 .. 9 (38) and is shifted right by `room` plus
// the distance of the exponents; room = 62 - s.  sh: of an FP64 number, an exponent to
// take off it (at bit 20).
template <int NS> struct Bias {
    static constexpr uint64_t b = 0x8080808080808080ull >> (64 - 8 * NS);
    static constexpr int room = 62 - (8 * NS - 2);
};
template <int NS> __device__ __forceinline__ uint64_t biased_int(double x, int ecol, int sh) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const int d = ((ecol + Bias<NS>::room) << 20) + sh - (int)(hi & 0x7ff00000u);
    const uint32_t mh = (hi & 0xfffffu) | 0x100000u;
    const uint64_t l = (uint64_t)lo * 512u;
    const uint64_t m = ((uint64_t)(mh * 512u + (uint32_t)(l >> 32)) << 32) | (uint32_t)l;
    return (m >> min((uint32_t)(d >> 20), 63u)) + Bias<NS>::b;
}
template <int NS> __device__ __forceinline__ uint64_t biased_int(float x, int ecol, int) {
    const uint32_t b = __float_as_uint(x);
    const int d = ((ecol + Bias<NS>::room) << 23) - (int)(b & 0x7f800000u);
    const uint32_t mh = ((b & 0x7fffffu) | 0x800000u) << 6;
    return (((uint64_t)mh << 32) >> min((uint32_t)(d >> 23), 63u)) + Bias<NS>::b;
}
__device__ __forceinline__ uint32_t top_word(double x) { return (uint32_t)__double2hiint(x); }
__device__ __forceinline__ uint32_t top_word(float x) { return __float_as_uint(x); }

// The digits of eight consecutive steps of one row: slice i (most significant
// first) is one core-matrix row of 16 bytes at dst + i * stride.  A byte b
// becomes the FP16 number 1024 + b by its bit pattern (two elements to a
// word), then the signed digit +-(b - 128) by one exact fused multiply-add:
// a byte permutation and a logic operation per two digits on the integer
// pipe, whose half rate bounds the conversion, the rest on the FP16 pipe.
template <typename T, int NS>
__device__ __forceinline__ void store_digits(const T (&v)[8], int ecol, unsigned char *dst, int stride,
                                             const int (&sh)[8] = {0, 0, 0, 0, 0, 0, 0, 0}) {
    uint32_t lo[8], hi[8], mul[4], add[4];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const uint64_t u = biased_int<NS>(v[k], ecol, sh[k]);
        lo[k] = (uint32_t)u;
        hi[k] = (uint32_t)(u >> 32);
    }
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const uint32_t sg = __byte_perm(top_word(v[2 * p]), top_word(v[2 * p + 1]), 0x7632) & 0x80008000u;
        mul[p] = sg ^ 0x3c003c00u;   // +-1
        add[p] = sg ^ 0xe480e480u;   // -+1152
    }
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        constexpr int last = NS - 1;
        const int b = last - i;      // byte of the integer
        uint32_t w[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            const uint32_t x0 = b < 4 ? lo[2 * p] : hi[2 * p], x1 = b < 4 ? lo[2 * p + 1] : hi[2 * p + 1];
            // bytes 0 and 2: the two elements' digits
            const uint32_t h = (__byte_perm(x0, x1, (unsigned)(b & 3) | ((unsigned)(4 + (b & 3)) << 8)) & 0x00ff00ffu) | 0x64006400u;
            const __half2 d = __hfma2(*reinterpret_cast<const __half2 *>(&h), *reinterpret_cast<const __half2 *>(&mul[p]),
                                      *reinterpret_cast<const __half2 *>(&add[p]));
            w[p] = *reinterpret_cast<const uint32_t *>(&d);
        }
        *reinterpret_cast<uint4 *>(dst + i * stride) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// ------------------------------------------------------- shared pieces ---

template <int NS, int BN, int PAD> struct DgCfg {
    // A: slice by slice, each KQ columns of core matrices; B: the slices of one
    // column group behind one another, so that several are one wide operand
    static constexpr int LBO_A = DG_M * 16 + PAD, LBO_B = NS * BN * 16;
    static constexpr int SL_A = KQ * LBO_A, SL_B = BN * 16;      // bytes from slice to slice
    static constexpr int A_BYTES = NS * SL_A, STAGE = A_BYTES + KQ * LBO_B;
    static constexpr int TMEM = NS * BN <= 128 ? 128 : NS * BN <= 256 ? 256 : 512;
    static constexpr size_t SMEM = (size_t)DG_STAGES * STAGE + 128;
    static_assert(NS * BN <= 512, "tensor memory columns");
    static_assert(LBO_A % 16 == 0, "core matrix stride");
};

struct DgBars {
    uint64_t full[DG_STAGES], empty[DG_STAGES], accfull[8], accfree, done;
    uint32_t tmem;
    DgGive give;
    int plain;
};

template <int NS> __device__ __forceinline__ void dg_setup(DgBars &b, int tmem_cols, int spin) {
    if (threadIdx.x == 0) {
        for (int i = 0; i < DG_STAGES; ++i) {
            dg_bar_init(&b.full[i], DG_CT);
            dg_bar_init(&b.empty[i], 1);
        }
        for (int t = 0; t < NS; ++t) dg_bar_init(&b.accfull[t], 1);
        dg_bar_init(&b.accfree, DG_CT);
        dg_bar_init(&b.done, 1);
        b.give = {0, spin};
        b.plain = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (threadIdx.x >> 5 == DG_CW) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(dg_su32(&b.tmem)),
                     "r"(tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    DG_FENCE_BEFORE();
    __syncthreads();
    DG_FENCE_AFTER();
}

// The MMA warp: all products of nst stages, in blocks of kst (a readout
// interval ends with its block).  Slice i of A meets slices 0 .. NS - 1 - i of
// B as one operand of (NS - i) BN columns (at most 256 to an instruction),
// whose products fall in accumulators i .. NS - 1: a third of the instructions
// and reads of A that single pairs of slices would take (those ran at 68
// cycles each, twice what 64 columns need).  Accumulator t is complete after
// slice t of the last stage.
template <int NS, int BN, int PAD> struct DgIssue {
    using C = DgCfg<NS, BN, PAD>;
    uint32_t tmem, lead;
    uint64_t da0, db0;
    int g = 0, iv = -1;   // stages taken, readout interval
    __device__ __forceinline__ DgIssue(DgBars &b, unsigned char *base) {
        tmem = __shfl_sync(0xffffffffu, b.tmem, 0);
        lead = (threadIdx.x & 31) == 0;
        da0 = dg_desc(dg_su32(base), C::LBO_A);
        db0 = dg_desc(dg_su32(base) + C::A_BYTES, C::LBO_B);
    }
    __device__ __forceinline__ bool run(DgBars &b, int nst, int kst) {
        int kb = 0;   // stage within the block
        bool ok = true;
        for (int it = 0; it < nst && ok; ++it, ++g) {
            const int s = g % DG_STAGES;
            const bool first = kb % DG_DRAIN == 0, last = kb % DG_DRAIN == DG_DRAIN - 1 || kb == kst - 1;
            iv += first;
            if (++kb == kst) kb = 0;
            ok = __all_sync(0xffffffffu, dg_wait(&b.full[s], (g / DG_STAGES) & 1, &b.give, 40));
            DG_FENCE_AFTER();
            const uint64_t da = da0 + (uint64_t)(s * (C::STAGE >> 4)), db = db0 + (uint64_t)(s * (C::STAGE >> 4));
            if (first && iv > 0 && ok) {
                ok = __all_sync(0xffffffffu, dg_wait(&b.accfree, (iv - 1) & 1, &b.give));
                DG_FENCE_AFTER();
            }
            if (ok) {
#pragma unroll
                for (int i = 0; i < NS; ++i) {
#pragma unroll
                    for (int k = 0; k < DG_K / 16; ++k)
#pragma unroll
                        for (int c = 0; c < (NS - i) * BN; c += 256) {
                            const int n = (NS - i) * BN - c < 256 ? (NS - i) * BN - c : 256;
                            dg_mma(tmem + i * BN + c, da + (uint64_t)((i * C::SL_A + 2 * k * C::LBO_A) >> 4),
                                   db + (uint64_t)((c * 16 + 2 * k * C::LBO_B) >> 4), dg_idesc(DG_M, n),
                                   (first && i == 0 && k == 0) ? 0u : 1u, lead);
                        }
                    if (last) dg_commit(&b.accfull[i], lead);
                }
            }
            dg_commit(&b.empty[s], lead);
        }
        return ok;
    }
    // after the last stage: waits for every product in flight
    __device__ __forceinline__ void finish(DgBars &b) {
        dg_commit(&b.done, lead);
        dg_settle(&b.done, 0);
    }
};

// One readout (in the order in which the accumulators complete) of CPT columns of
// the converter thread's row: H += accumulators 0 .. 2 in units of accumulator
// 2, L += the later ones in units of accumulator NS - 2, the last one rounded to
// them.
template <int NS, int BN, int CPT>
__device__ __forceinline__ bool dg_drain(DgBars &b, int iv, int col0, int64_t (&H)[CPT], int64_t (&L)[CPT], bool release = true) {
    const int warp = threadIdx.x >> 5;
    const uint32_t lane_base = b.tmem + ((uint32_t)(warp & 3) * 32 << 16) + (uint32_t)col0;
#pragma unroll
    for (int t = 0; t < NS - 2; ++t) {
        if (!dg_wait_warp(&b.accfull[t], iv & 1, &b.give)) return false;
        DG_FENCE_AFTER();
#pragma unroll
        for (int c = 0; c < CPT; c += CPT < 32 ? CPT : 32) {
            constexpr int W = CPT < 32 ? CPT : 32;
            uint32_t r[W];
            if constexpr (W == 32) dg_tmem_ld32(lane_base + t * BN + c, r);
            else dg_tmem_ld16(lane_base + t * BN + c, r);
#pragma unroll
            for (int j = 0; j < W; ++j) {
                // accumulators 0 and 1 stay within 2^22: their integers stand in the
                // mantissa after one addition (the conversion unit is slow)
                const int64_t v = t < 2 ? (int64_t)((int)__float_as_uint(__fadd_rn(__uint_as_float(r[j]), 12582912.f)) - 0x4b400000)
                                        : (int64_t)__float2int_rn(__uint_as_float(r[j]));
                if (t < 3) H[c + j] += v * (int64_t)(1 << (8 * (2 - t)));
                else L[c + j] += v * (int64_t)(1 << (8 * (NS - 2 - t)));
            }
        }
    }
    // the last two accumulators together, rounded at the weight of the first
    if (!dg_wait_warp(&b.accfull[NS - 1], iv & 1, &b.give)) return false;
    DG_FENCE_AFTER();
#pragma unroll
    for (int q = 0; q < CPT / 8; ++q) {
        uint32_t u[8], w[8];
        dg_tmem_ld8(lane_base + (NS - 2) * BN + 8 * q, u);
        dg_tmem_ld8(lane_base + (NS - 1) * BN + 8 * q, w);
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
        for (int j = 0; j < 8; ++j)
            L[8 * q + j] += (int64_t)__float2int_rn(fmaf(__uint_as_float(w[j]), 1.f / 256.f, __uint_as_float(u[j])));
    }
    if (release) {
        DG_FENCE_BEFORE();
        dg_arrive(&b.accfree);
    }
    return true;
}

// 2^e as FP64 (e within the normal range)
__device__ __forceinline__ double pow2d(int e) { return __hiloint2double((e + 1023) << 20, 0); }

// ------------------------------------------------------------ overlap ---

template <typename T> struct GramArgs {
    const T *X, *Y;
    int64_t ldx, ldy, npts, lds;
    int nx, ny;
    const int *kx, *ky;      // column keys
    double *S;
    double dV;
    int tiles_n, stages, per_cta;   // stages in all and per CTA
    int sym;                 // Y is X: only the elements j >= i are computed, and mirrored
    int far;                 // rows 4 GB or more apart: the digit path's row strides are 32-bit numbers of bytes
    int spin;                // barrier tests before a wait gives up
    int *err;                // status word (or nullptr): 1 once one has
};

template <typename T, int NS, int BN> __global__ void __launch_bounds__(DG_NT, 1) k_digit_gram(GramArgs<T> a) {
    using C = DgCfg<NS, BN, 0>;
    extern __shared__ __align__(128) unsigned char dgsm[];
    __shared__ DgBars b;
    __shared__ int ea[DG_M], eb[BN];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // tile (bm, bn): in the symmetric case the bn-th of those not entirely below the diagonal
    int bm = 0, bn = blockIdx.x;
    if (a.sym) {
        for (;; ++bm) {
            const int skip = bm * DG_M / BN;
            if (bn < a.tiles_n - skip) {
                bn += skip;
                break;
            }
            bn -= a.tiles_n - skip;
        }
    } else {
        bm = blockIdx.x / a.tiles_n;
        bn = blockIdx.x - bm * a.tiles_n;
    }
    const int m0 = bm * DG_M, n0 = bn * BN;
    const int st0 = blockIdx.y * a.per_cta, nst = min(a.per_cta, a.stages - st0);
    dg_setup<NS>(b, C::TMEM, a.spin);
    for (int i = tid; i < DG_M + BN; i += DG_NT) {
        const bool isa = i < DG_M;
        const int c = isa ? m0 + i : n0 + i - DG_M;
        const int key = isa ? (c < a.nx ? a.kx[c] : 0) : (c < a.ny ? a.ky[c] : 0);
        (isa ? ea[i] : eb[i - DG_M]) = ExpOf<T>::exponent(key);
        if (ExpOf<T>::plain(key) || a.far) b.plain = 1;
    }
    __syncthreads();
    const int64_t p0 = (int64_t)st0 * DG_K, p1 = min(a.npts, p0 + (int64_t)nst * DG_K);
    if (b.plain) {
        // a column beyond the digits' range, or far rows: plain FP64 sums of this tile and range
        for (int e = tid; e < DG_M * BN; e += DG_NT) {
            const int i = m0 + e / BN, j = n0 + e % BN;
            if (i >= a.nx || j >= a.ny || (a.sym && j < i)) continue;
            double s = 0;
            for (int64_t p = p0; p < p1; ++p) s = fma((double)a.X[p * a.ldx + i], (double)a.Y[p * a.ldy + j], s);
            atomicAdd(a.S + (int64_t)i * a.lds + j, a.dV * s);
            if (a.sym && j > i) atomicAdd(a.S + (int64_t)j * a.lds + i, a.dV * s);
        }
    } else if (warp >= DG_CW) {
        DG_REGS_DOWN();
        if (warp == DG_CW) {
            DgIssue<NS, BN, 0> mma(b, dgsm);
            mma.run(b, nst, nst);
            mma.finish(b);
        }
    } else {
        DG_REGS_UP();
        // converter warp: units (32 columns, 8 points) warp, warp + 8 of A and warp of B
        constexpr int NB = BN / 32 * KQ;            // units of B per stage
        constexpr int NU = 2 + (NB + DG_CW - 1) / DG_CW;
        const T *src[NU];
        unsigned char *dst[NU];
        int ec[NU], sl[NU], off[NU];
        uint32_t ld[NU];
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            const bool isa = u < 2;
            const int w = isa ? warp + DG_CW * u : warp + DG_CW * (u - 2);
            const bool has = isa || w < NB;
            const int rg = w / KQ, kq = w % KQ, row = rg * 32 + lane;
            const int c = isa ? m0 + row : n0 + row;
            // a column beyond the last reads the first one; what its digits are
            // only reaches results that are not written
            const bool in = has && c < (isa ? a.nx : a.ny);
            ec[u] = isa ? ea[row & (DG_M - 1)] : eb[row & (BN - 1)];
            ld[u] = (uint32_t)((isa ? a.ldx : a.ldy) * (int64_t)sizeof(T));
            off[u] = 8 * kq;
            src[u] = (isa ? a.X : a.Y) + (in ? c : 0);
            dst[u] = has ? dgsm + (isa ? kq * C::LBO_A : C::A_BYTES + kq * C::LBO_B) + row * 16 : nullptr;
            sl[u] = isa ? C::SL_A : C::SL_B;
        }
        T v[NU][8];
        auto load = [&](int it) {
            const int64_t pb = p0 + (int64_t)it * DG_K;
            if (pb + DG_K <= p1) {
#pragma unroll
                for (int u = 0; u < NU; ++u)
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        v[u][k] = __ldg(reinterpret_cast<const T *>(reinterpret_cast<const char *>(src[u]) +
                                                                    (uint64_t)((uint32_t)pb + off[u] + k) * ld[u]));
            } else {
#pragma unroll
                for (int u = 0; u < NU; ++u)
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        v[u][k] = pb + off[u] + k < p1
                                      ? __ldg(reinterpret_cast<const T *>(reinterpret_cast<const char *>(src[u]) +
                                                                          (uint64_t)((uint32_t)pb + off[u] + k) * ld[u]))
                                      : T(0);
            }
        };
        constexpr int CPT = 32;   // columns of the result per thread
        int64_t H[CPT], L[CPT];
#pragma unroll
        for (int j = 0; j < CPT; ++j) H[j] = L[j] = 0;
        const int col0 = (warp >> 2) * CPT;
        const bool drains = col0 < BN;   // BN = 32: the second four warps only free the accumulators
        bool ok = true;
        load(0);
        int iv = 0;   // readouts taken
        for (int it = 0; it < nst && ok; ++it) {
            const int s = it % DG_STAGES;
            if (it >= DG_STAGES && !dg_wait_warp(&b.empty[s], (it / DG_STAGES - 1) & 1, &b.give)) {
                ok = false;
                break;
            }
#pragma unroll
            for (int u = 0; u < NU; ++u)
                if (dst[u]) store_digits<T, NS>(v[u], ec[u], dst[u] + s * C::STAGE, sl[u]);
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
            dg_arrive(&b.full[s]);
            if (it + 1 < nst) load(it + 1);
            // the previous 256 points' accumulators, once the first stage after them is queued
            if (it % DG_DRAIN == 0 && it > 0) {
                ok = dg_drain<NS, BN, CPT>(b, iv, drains ? col0 : 0, H, L);
                ++iv;
            }
        }
        if (ok) ok = dg_drain<NS, BN, CPT>(b, iv, drains ? col0 : 0, H, L);
        const int row = (warp & 3) * 32 + lane, i = m0 + row;
        if (i < a.nx && drains) {
            const int s2 = 2 * (8 * NS - 2);
#pragma unroll
            for (int j = 0; j < CPT; ++j) {
                const int jc = n0 + col0 + j;
                if (jc >= a.ny || (a.sym && jc < i)) continue;
                const int e = ea[row] + eb[col0 + j] - 2 * (ExpOf<T>::bias - 1) - s2;
                double r = a.dV * fma((double)H[j], pow2d(e + 8 * (2 * NS - 4)), (double)L[j] * pow2d(e + 8 * NS));
                if (!ok) r = __longlong_as_double(0x7ff8000000000000ll);
                atomicAdd(a.S + (int64_t)i * a.lds + jc, r);
                if (a.sym && jc > i) atomicAdd(a.S + (int64_t)jc * a.lds + i, r);
            }
        }
    }
    DG_FENCE_BEFORE();
    __syncthreads();
    if (tid == 0 && a.err && b.give.bad) atomicExch(a.err, 1);
    if (warp == DG_CW)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(b.tmem), "r"(C::TMEM) : "memory");
}

// Zero S and the keys.
__global__ void k_digit_init(double *S, int64_t lds, int n, int m, int *keys, int nkeys) {
    const int64_t step = (int64_t)gridDim.x * blockDim.x, t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    for (int64_t e = t0; e < (int64_t)n * m; e += step) S[(e / m) * lds + e % m] = 0.0;
    for (int64_t e = t0; e < nkeys; e += step) keys[e] = 0;
}

// Largest key of every column of X (blocks [0, gx)) and Y: 32 columns and 8
// rows per block and pass.
template <typename T>
__global__ void __launch_bounds__(256) k_digit_keys(const T *__restrict__ X, int64_t ldx, int nx, const T *__restrict__ Y,
                                                    int64_t ldy, int ny, int64_t npts, int gx, int *keys) {
    __shared__ int red[8][32];
    const int l = threadIdx.x & 31, r = threadIdx.x >> 5;
    const bool isx = (int)blockIdx.x < gx;
    const int c = (isx ? blockIdx.x : blockIdx.x - gx) * 32 + l;
    const T *src = isx ? X : Y;
    const int64_t ld = isx ? ldx : ldy;
    int k = 0;
    if (c < (isx ? nx : ny)) {
        const int64_t step = (int64_t)gridDim.y * 8;
        int64_t p = (int64_t)blockIdx.y * 8 + r;
        for (; p + 7 * step < npts; p += 8 * step) {
            T v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = __ldg(src + (p + u * step) * ld + c);
#pragma unroll
            for (int u = 0; u < 8; ++u) k = max(k, abs_key(v[u]));
        }
        for (; p < npts; p += step) k = max(k, abs_key(__ldg(src + p * ld + c)));
    }
    red[r][l] = k;
    __syncthreads();
    if (r == 0 && c < (isx ? nx : ny)) {
#pragma unroll
        for (int q = 1; q < 8; ++q) k = max(k, red[q][l]);
        if (k) atomicMax(keys + (isx ? 0 : nx) + c, k);
    }
}

// Barrier tests before a wait of a contraction gives up, for the calls of this host
// thread (rs_contraction_wait_limit).
thread_local int t_gram_spin = DG_SPIN, t_rot_spin = DG_SPIN;

int sm_count(int *n) {
    int dev = 0;
    RS_CUDA(cudaGetDevice(&dev));
    RS_CUDA(cudaDeviceGetAttribute(n, cudaDevAttrMultiProcessorCount, dev));
    return RS_OK;
}

template <typename T, int NS, int BN> int launch_gram(GramArgs<T> a, int tiles_m, cudaStream_t st) {
    using C = DgCfg<NS, BN, 0>;
    a.tiles_n = (a.ny + BN - 1) / BN;
    int tiles = 0;
    for (int m = 0; m < tiles_m; ++m) tiles += a.tiles_n - (a.sym ? m * DG_M / BN : 0);
    int nsm = 0;
    RS_TRY(sm_count(&nsm));
    // the split of the points that leaves the fewest stages to the busiest SM
    // (a CTA's set-up and result cost about as much as 6 stages)
    a.stages = (int)((a.npts + DG_K - 1) / DG_K);
    int64_t best = INT64_MAX;
    for (int s = 1; s <= std::min(a.stages, 8 * nsm); ++s) {
        if ((int64_t)tiles * s > 8ll * nsm && s > 1) break;
        const int64_t cost = (((int64_t)tiles * s + nsm - 1) / nsm) * ((a.stages + s - 1) / s + 6);
        if (cost < best) {
            best = cost;
            a.per_cta = (a.stages + s - 1) / s;
        }
    }
    const int splits = (a.stages + a.per_cta - 1) / a.per_cta;
    RS_TRY(smem_optin((const void *)k_digit_gram<T, NS, BN>, C::SMEM));
    k_digit_gram<T, NS, BN><<<dim3((unsigned)tiles, (unsigned)splits), DG_NT, C::SMEM, st>>>(a);
    RS_LAUNCH_CHECK();
    return RS_OK;
}

}  // namespace

template <typename T>
int digit_gram(const T *X, int64_t ldx, int nx, const T *Y, int64_t ldy, int ny, int64_t npts, double dV, double *S,
               int64_t lds, int *scratch, cudaStream_t st, int *err) {
    if (npts > (int64_t)INT32_MAX - 64) return fail(RS_EINVAL, "digit_gram: too many points");
    const bool sym = X == Y && ldx == ldy && nx == ny;
    int *keys = scratch;
    PoolBuf own;
    if (!keys) {
        RS_TRY(own.alloc(sizeof(int) * (size_t)digit_gram_scratch_ints(nx, ny), st));
        keys = reinterpret_cast<int *>(own.p);
    }
    {
        const int64_t ne = std::max<int64_t>((int64_t)nx * ny, nx + ny);
        k_digit_init<<<(unsigned)std::min<int64_t>(256, (ne + 255) / 256), 256, 0, st>>>(S, lds, nx, ny, keys, nx + ny);
        RS_LAUNCH_CHECK();
        const int gx = (nx + 31) / 32, gy = sym ? 0 : (ny + 31) / 32;
        const int rows = (int)std::max<int64_t>(1, std::min<int64_t>((npts + 63) / 64, 152 * 8 / (gx + gy)));
        k_digit_keys<T><<<dim3((unsigned)(gx + gy), (unsigned)rows), 256, 0, st>>>(X, ldx, nx, Y, ldy, ny, npts, gx, keys);
        RS_LAUNCH_CHECK();
        GramArgs<T> a{};
        a.X = X, a.Y = Y, a.ldx = ldx, a.ldy = ldy, a.npts = npts, a.lds = lds, a.nx = nx, a.ny = ny;
        a.kx = keys, a.ky = sym ? keys : keys + nx;
        a.S = S, a.dV = dV, a.sym = sym, a.far = std::max(ldx, ldy) > (int64_t)(UINT32_MAX / sizeof(T)), a.spin = t_gram_spin, a.err = err;
        const int tm = (nx + DG_M - 1) / DG_M;
        // 32 columns of Y fill half of a 64-wide tile
        const bool narrow = ny <= 32;
        if constexpr (sizeof(T) == 8) return narrow ? launch_gram<T, 8, 32>(a, tm, st) : launch_gram<T, 8, 64>(a, tm, st);
        else return narrow ? launch_gram<T, 7, 32>(a, tm, st) : launch_gram<T, 7, 64>(a, tm, st);
    }
}
template int digit_gram<double>(const double *, int64_t, int, const double *, int64_t, int, int64_t, double, double *,
                                int64_t, int *, cudaStream_t, int *);
template int digit_gram<float>(const float *, int64_t, int, const float *, int64_t, int, int64_t, double, double *,
                               int64_t, int *, cudaStream_t, int *);

template <typename T> int column_keys(const T *X, int64_t ldx, int n, int64_t npts, int *keys, cudaStream_t st) {
    RS_CUDA(cudaMemsetAsync(keys, 0, sizeof(int) * (size_t)n, st));
    const int gx = (n + 31) / 32;
    const int rows = (int)std::max<int64_t>(1, std::min<int64_t>((npts + 63) / 64, 152 * 8 / gx));
    k_digit_keys<T><<<dim3((unsigned)gx, (unsigned)rows), 256, 0, st>>>(X, ldx, n, X, ldx, 0, npts, gx, keys);
    RS_LAUNCH_CHECK();
    return RS_OK;
}
template int column_keys<double>(const double *, int64_t, int, int64_t, int *, cudaStream_t);
template int column_keys<float>(const float *, int64_t, int, int64_t, int *, cudaStream_t);

// ----------------------------------------------------------- rotation ---

namespace {

template <typename T> struct RotArgs {
    const T *X;
    const double *C;
    T *Y;
    const int *xk;       // keys of X's columns (their sizes), or nullptr: columns of one size
    int64_t ldx, ldc, ldy, npts;
    int n, m;
    int vec, yvec;       // X, Y rows on 16-byte boundaries
    int cluster;         // Y is X: the CTAs of a row tile form a cluster and write together
    int spin, *err;      // as in GramArgs
    double alpha, beta;
};

// (H 2^32 + L) 2^(64 + e) rounded once to FP64 (NS = 8; |H|, |L| < 2^51): H and L
// added to the mantissas of 1.5 2^52 at their scales give two FP64 numbers by
// one integer addition each, whose offsets cancel in two FP64 additions, the
// first of them exact.  (Normalising the 128-bit sum in integers took ten times
// the instructions and a third of a rotation of 48 columns.)
// ex: (1023 + 52 + 96 + e) << 20
__device__ __forceinline__ double dg_value(int64_t H, int64_t L, int ex) {
    const double a = __hiloint2double((int)(H >> 32) + ex + 0x80000, (int)(uint32_t)H);
    const double b = __hiloint2double((int)(L >> 32) + ex + 0x80000 - (32 << 20), (int)(uint32_t)L);
    const double ab = __hiloint2double(ex + 0x80000, 0x180000);   // both offsets: 1.5 (1 + 2^-32)
    return __dadd_rn(__dsub_rn(a, ab), b);
}

struct RotBars {
    uint64_t keyfull[2], keyfree[2], rd, sums;
    int plain[2][4];   // per half and key warp: a row beyond the digits' range
};

// One CTA per SM, NBLK column blocks of C per CTA, row tiles dealt round robin:
// the key warps find the exponents of the next tile's rows (and bring the
// rows into L2) while the converters work on this one, and the readout and
// the stores of a tile overlap the products of the next.
// Column sizes: an entry of X is resolved relative to the largest of its row, so a
// small column would lose its digits beside large ones, though its row of C may
// be as much larger (Psi U^-1 of columns that are not normalised).  So the columns are brought to
// the size of the largest one by powers of two, 2^-a_k, and the rows of C
// taken the other way, which changes no product: in FP64 as an addend of the
// exponents' distance, in FP32 by a multiplication, which is exact (the factor is at
// least 1) and on a pipe with nothing to do.  sh[k]: a_k at bit 20 (FP64), 2^-a_k
// (FP32).  Columns more than 2^span apart: plain sums.
// ONE: at most 256 states, so that a block is one readout and its sums need no
// registers while the operands are converted (with them the converters spill:
// 5.5 ms instead of 4.7 for 658 416 rows of 256 FP64 states).
template <typename T, int NS, int BN, int NBLK, bool ONE>
__global__ void __launch_bounds__(DG_NT, 1) k_digit_rot(RotArgs<T> a) {
    constexpr int PAD = 32;   // a quarter-warp's four 8-step groups of two rows fall in distinct banks
    constexpr int KW = 3;     // key warps
    using C = DgCfg<NS, BN, PAD>;
    extern __shared__ __align__(128) unsigned char dgsm[];
    __shared__ DgBars b;
    __shared__ RotBars rb;
    __shared__ int ea[2][DG_M], eb[NBLK * BN], etop, zeros;
    int *sh = reinterpret_cast<int *>(dgsm + DG_STAGES * C::STAGE);   // [kst * DG_K]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nb0 = blockIdx.x * NBLK;          // first column block
    const int kst = (a.n + DG_K - 1) / DG_K;    // stages per column block
    const int ntiles = (int)((a.npts + DG_M - 1) / DG_M);
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            dg_bar_init(&rb.keyfull[i], KW * 32);
            dg_bar_init(&rb.keyfree[i], DG_CT + 1);   // the converters and the MMA warp's first lane
        }
        dg_bar_init(&rb.rd, DG_CT * (a.cluster ? gridDim.x : 1));
        dg_bar_init(&rb.sums, DG_CT);
        etop = 0;
        zeros = a.xk != nullptr;
    }
    for (int i = tid; i < NBLK * BN; i += DG_NT) eb[i] = INT_MIN;
    dg_setup<NS>(b, C::TMEM, a.spin);
    if (a.cluster) asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
    // sizes of the columns of X; 0: a column of zeros, or one with entries beyond the
    // digits' range, whose rows take plain sums: left as it is
    auto size_of = [&](int k) {
        const int key = a.xk && k < a.n ? __ldg(a.xk + k) : 0, e = max(key >> ExpOf<T>::mant, 1);
        return key && e <= ExpOf<T>::hi ? e : 0;
    };
    for (int k = tid; k < a.n; k += DG_NT) {
        const int e = size_of(k);
        if (e) atomicMax(&etop, e);
        if (a.xk && a.xk[k]) zeros = 0;   // (all columns are zero: the eigensolver's first directions)
    }
    __syncthreads();
    for (int k = tid; k < kst * DG_K; k += DG_NT) {
        const int e = size_of(k);
        int d = e ? e - etop : 0;
        if (d < -ExpOf<T>::span) {
            b.plain = 1;
            d = 0;
        }
        sh[k] = sizeof(T) == 8 ? d * (1 << 20) : (127 - d) << 23;
    }
    __syncthreads();
    // what is added to the exponent (at bit 20) of row k of C
    auto c_shift = [&](int v) { return sizeof(T) == 8 ? v : (127 << 20) - (v >> 3); };
    // exponents of the columns of C
    for (int blk = 0; blk < NBLK; ++blk)
        for (int w = warp; w < BN / 32 * 12; w += DG_NT / 32) {
            const int cl = (w / 12) * 32 + lane, c = (nb0 + blk) * BN + cl;
            int k = INT_MIN;
            bool pl = false;
            if (c < a.m) {
#pragma unroll 8
                for (int q = w % 12; q < a.n; q += 12) {
                    const int key = abs_key(__ldg(a.C + (int64_t)q * a.ldc + c)), e = key >> 20;
                    if (key) k = max(k, e + (c_shift(sh[q]) >> 20));
                    pl = pl || e > ExpOf<double>::hi;
                }
            }
            if (pl) b.plain = 1;
            if (k != INT_MIN) atomicMax(&eb[blk * BN + cl], k);
        }
    __syncthreads();
    for (int i = tid; i < NBLK * BN; i += DG_NT) {
        const int e = eb[i] == INT_MIN ? ExpOf<double>::bias : eb[i];
        if (e < ExpOf<double>::lo || e > ExpOf<double>::hi) b.plain = 1;
        eb[i] = e;
    }
    __syncthreads();
    const bool cplain = b.plain != 0;

    if (warp > DG_CW) {
        // key warps: eight rows at a time, four lanes to a row
        asm volatile("setmaxnreg.dec.sync.aligned.u32 72;\n");
        int j = 0;
        for (int tile = blockIdx.y; tile < ntiles; tile += gridDim.y, ++j) {
            const int h = j & 1;
            if (j >= 2 && !dg_wait(&rb.keyfree[h], (j / 2 - 1) & 1, &b.give, 50 * kst)) break;
            const int64_t r0 = (int64_t)tile * DG_M;
            const int rows = (int)min((int64_t)DG_M, a.npts - r0);
            bool pl = false;
            for (int g = warp - DG_CW - 1; g < DG_M / 8; g += KW) {
                const int r = g * 8 + (lane >> 2);
                const T *x = a.X + (r0 + min(r, rows - 1)) * a.ldx;
                // largest scaled entry: as a key (FP32), with an addend to the exponent
                // (FP64; of a zero, that stays below any exponent that is taken)
                int k = INT_MIN;
                auto take = [&](T v, int f) {
                    if constexpr (sizeof(T) == 8) k = max(k, (__double2hiint(v) & 0x7fffffff) - f);
                    else k = max(k, abs_key(v * __int_as_float(f)));
                };
                if (a.vec) {
                    constexpr int E = 16 / (int)sizeof(T);
                    const uint4 *xv = reinterpret_cast<const uint4 *>(x);
                    const int nv = a.n / E;
                    for (int q0 = lane & 3; q0 < nv; q0 += 32) {
                        uint4 t[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            t[i] = ld_fresh(xv + min(q0 + 4 * i, nv - 1));   // in this order, ahead of the factors' reads:
                        // with two or three in flight the key warps hold the others up (9.5 ms instead of 4.8 for 256 FP64 states)
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const T *tt = reinterpret_cast<const T *>(&t[i]);
#pragma unroll
                            for (int e = 0; e < E; ++e) take(tt[e], sh[min(q0 + 4 * i, nv - 1) * E + e]);
                        }
                    }
                    for (int q = nv * E + (lane & 3); q < a.n; q += 4) take(x[q], sh[q]);
                } else {
#pragma unroll 8
                    for (int q = lane & 3; q < a.n; q += 4) take(x[q], sh[q]);
                }
                k = max(k, __shfl_xor_sync(0xffffffffu, k, 1));
                k = max(k, __shfl_xor_sync(0xffffffffu, k, 2));
                if (sizeof(T) == 8 && (k >> 20) < ExpOf<T>::lo) {
                    // a row of zeros, or one for the plain sums
                    int any = 0;
                    if (!zeros)
                        for (int q = lane & 3; q < a.n; q += 4) any |= abs_key(x[q]);
                    k = any ? max(k, 1) : 0;
                }
                if (sizeof(T) == 8) {
                    // (the four lanes of a row agree: one with an entry speaks for all)
                    const int kk = max(k, __shfl_xor_sync(0xffffffffu, k, 1));
                    k = max(kk, __shfl_xor_sync(0xffffffffu, kk, 2));
                }
                if ((lane & 3) == 0) ea[h][r] = ExpOf<T>::exponent(k);
                pl = pl || ExpOf<T>::plain(k);
            }
            pl = __any_sync(0xffffffffu, pl);
            if (lane == 0) rb.plain[h][warp - DG_CW - 1] = pl;
            __syncwarp();
            dg_arrive(&rb.keyfull[h]);
        }
    } else if (warp == DG_CW) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 72;\n");
        DgIssue<NS, BN, PAD> mma(b, dgsm);
        int j = 0;
        bool ok = true;
        for (int tile = blockIdx.y; tile < ntiles && ok; tile += gridDim.y, ++j) {
            const int h = j & 1;
            ok = __all_sync(0xffffffffu, dg_wait(&rb.keyfull[h], (j / 2) & 1, &b.give));
            const volatile int *f = rb.plain[h];
            const bool pl = cplain || f[0] || f[1] || f[2];
            __syncwarp();
            if (lane == 0) dg_arrive(&rb.keyfree[h]);
            if (!pl && ok) ok = mma.run(b, kst * NBLK, kst);
        }
        mma.finish(b);
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 216;\n");
        // converter warp: rows 16 warp .. + 15 of A (a lane's unit: one row, 8
        // steps; four lanes read 32 consecutive states of a row) and unit
        // `warp` (32 columns, 8 steps) of B
        constexpr int NB = BN / 32 * KQ;
        static_assert(NB <= DG_CW, "one unit of B per warp");
        const int ar = warp * 16 + (lane >> 2), akq = lane & 3;
        unsigned char *adst = dgsm + akq * C::LBO_A + ar * 16;
        const bool hasb = warp < NB;
        // one or two stages a block: a stage's buffer meets the same digits of C in
        // every tile, so they are written once
        const int bstages = NBLK == 1 && kst <= DG_STAGES ? DG_STAGES : INT32_MAX;
        const int bkq = warp % KQ, bcol = warp / KQ * 32 + lane;
        unsigned char *bdst = dgsm + C::A_BYTES + bkq * C::LBO_B + bcol * 16;
        const int col0 = (warp >> 2) * 32, row = (warp & 3) * 32 + lane;
        const bool owns = col0 < BN;
        const int nst = kst * NBLK;
        bool ok = true;
        T va[2][8];
        double vb[8];
        T held[NBLK > 1 ? 32 : 1];   // two blocks: the first one's results until the rows are read
        constexpr int HC = ONE ? 16 : 32;   // columns summed at a time
        int64_t H[ONE ? 1 : HC], L[ONE ? 1 : HC];
#pragma unroll
        for (int i = 0; i < (ONE ? 1 : HC); ++i) H[i] = L[i] = 0;
        auto load = [&](int u, int tile, int it) {   // u = 0, 1: rows of X; 2: C
            const int blk = it >= kst ? 1 : 0, k0 = (it - blk * kst) * DG_K;   // (NBLK <= 2)
            const int64_t r0 = (int64_t)tile * DG_M;
            const int rows = (int)min((int64_t)DG_M, a.npts - r0);
            if (u < 2) {
                const T *x = a.X + (r0 + min(ar + 8 * u, rows - 1)) * a.ldx + k0 + 8 * akq;
                if (a.vec && k0 + 8 * akq + 8 <= a.n) {
                    constexpr int E = 16 / (int)sizeof(T);
#pragma unroll
                    for (int q = 0; q < 8 / E; ++q) {
                        const uint4 t = reinterpret_cast<const uint4 *>(x)[q];
                        const T *tt = reinterpret_cast<const T *>(&t);
#pragma unroll
                        for (int i = 0; i < E; ++i) va[u][q * E + i] = tt[i];
                    }
                } else {
#pragma unroll
                    for (int k = 0; k < 8; ++k) va[u][k] = k0 + 8 * akq + k < a.n ? x[k] : T(0);
                }
            }
            if (u == 2 && hasb) {
                const int c = (nb0 + blk) * BN + bcol;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int kk = k0 + 8 * bkq + k;
                    vb[k] = (c < a.m && kk < a.n) ? __ldg(a.C + (int64_t)kk * a.ldc + c) : 0.0;
                }
            }
        };
        // column factors of the eight steps kq of a stage, and the values of FP32 columns brought to one size
        auto shifts = [&](int stage, int kq, int (&f)[8]) {
            const int4 *p = reinterpret_cast<const int4 *>(sh + stage * DG_K + 8 * kq);
            const int4 u = p[0], v = p[1];
            f[0] = u.x, f[1] = u.y, f[2] = u.z, f[3] = u.w, f[4] = v.x, f[5] = v.y, f[6] = v.z, f[7] = v.w;
        };
        auto scale = [&](T (&v)[8], const int (&f)[8]) {
            if constexpr (sizeof(T) == 4) {
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] *= __int_as_float(f[k]);
            }
        };
        // in place: tell every CTA of the row tile that this thread has read its rows
        auto rows_read = [&]() {
            if (!a.cluster) return;
            for (int r = 0; r < (int)gridDim.x; ++r)
                asm volatile(
                    "{\n .reg .b32 ra;\n mapa.shared::cluster.u32 ra, %0, %1;\n"
                    " mbarrier.arrive.release.cluster.shared::cluster.b64 _, [ra];\n}\n" ::"r"(dg_su32(&rb.rd)),
                    "r"(r)
                    : "memory");
        };
        const T al = (T)a.alpha, be = (T)a.beta;
        constexpr int E = 16 / (int)sizeof(T);
        // G results of row p from column c on; when Y is added, its G values are
        // read at once (one after another they cost a trip to memory each)
        constexpr int G = 8;
        auto old = [&](int64_t p, int c, T (&o)[G]) {
            const T *y = a.Y + p * a.ldy + c;
            if (a.yvec && c + G <= a.m) {
#pragma unroll
                for (int q = 0; q < G / E; ++q) {
                    const uint4 t = reinterpret_cast<const uint4 *>(y)[q];
                    const T *tt = reinterpret_cast<const T *>(&t);
#pragma unroll
                    for (int i = 0; i < E; ++i) o[q * E + i] = tt[i];
                }
            } else {
#pragma unroll
                for (int i = 0; i < G; ++i) o[i] = c + i < a.m ? y[i] : T(0);
            }
        };
        auto put = [&](int64_t p, int c, T (&v)[G]) {
            T *y = a.Y + p * a.ldy + c;
            if (!ok) {
#pragma unroll
                for (int i = 0; i < G; ++i) v[i] = (T)__longlong_as_double(0x7ff8000000000000ll);
            }
            if (a.yvec && c + G <= a.m) {
#pragma unroll
                for (int q = 0; q < G / E; ++q) {
                    uint4 t;
                    T *tt = reinterpret_cast<T *>(&t);
#pragma unroll
                    for (int i = 0; i < E; ++i) tt[i] = v[q * E + i];
                    reinterpret_cast<uint4 *>(y)[q] = t;
                }
            } else {
#pragma unroll
                for (int i = 0; i < G; ++i)
                    if (c + i < a.m) y[i] = v[i];
            }
        };
        // an interval of products whose accumulators are still to be read out:
        // its tile, the exponent of this thread's row in it, its block, and
        // whether it is the block's last
        bool open = false, pend = false;
        int ptile = 0, ptj = 0, pe = 0, pblk = 0, iv = 0;
        // HC finished sums from the thread's column c0 on: scaled and stored
        auto finish = [&](const int64_t (&h)[HC], const int64_t (&l)[HC], int c0, int64_t p, bool on, bool lastb) {
#pragma unroll
            for (int q = 0; q < HC / G; ++q) {
                T v[G], o[G];
                const bool add = a.beta != 0.0 && on;
                if (add) old(p, (nb0 + pblk) * BN + col0 + c0 + q * G, o);
#pragma unroll
                for (int i = 0; i < G; ++i) {
                    const int c = q * G + i, e = eb[pblk * BN + (owns ? col0 : 0) + c0 + c] - 1022 - 2 * (8 * NS - 2);
                    if constexpr (sizeof(T) == 8) {
                        v[i] = (T)dg_value(h[c], l[c], (1023 + 52 + 96 + pe - 1022 + e) << 20);
                    } else {
                        // NS = 5: H 2^8 + L stays below 2^63
                        v[i] = ldexpf(__ll2float_rn(h[c] * (int64_t)(1ll << (8 * (NS - 4))) + l[c]), 8 * NS + pe - 126 + e);
                    }
                    if (a.alpha != 1.0) v[i] *= al;
                    if (add) v[i] += be * o[i];
                    if (NBLK > 1 && !lastb) held[NBLK > 1 ? c0 + c : 0] = v[i];
                }
                if (lastb && on) put(p, (nb0 + pblk) * BN + col0 + c0 + q * G, v);
            }
        };
        auto readout = [&]() {
            open = false;
            if constexpr (!ONE) {
                ok = ok && dg_drain<NS, BN, HC>(b, iv, owns ? col0 : 0, H, L);
                ++iv;
                if (!pend) return;
            }
            // the block's sums are complete
            const bool lastb = pblk == NBLK - 1;
            if (lastb && a.cluster) ok = dg_wait_warp(&rb.rd, ptj & 1, &b.give) && ok;
            const int64_t p = (int64_t)ptile * DG_M + row;
            const bool on = owns && p < a.npts;
            if (NBLK > 1 && lastb && on) {
#pragma unroll
                for (int q = 0; q < 32 / G; ++q) {
                    T v[G];
#pragma unroll
                    for (int i = 0; i < G; ++i) v[i] = held[NBLK > 1 ? q * G + i : 0];
                    put(p, nb0 * BN + col0 + q * G, v);
                }
            }
            if constexpr (ONE) {
#pragma unroll
                for (int c0 = 0; c0 < 32; c0 += HC) {
                    int64_t h[HC], l[HC];
#pragma unroll
                    for (int i = 0; i < HC; ++i) h[i] = l[i] = 0;
                    ok = ok && dg_drain<NS, BN, HC>(b, iv, owns ? col0 + c0 : 0, h, l, c0 + HC == 32);
                    finish(h, l, c0, p, on, lastb);
                }
                ++iv;
            } else {
                finish(H, L, 0, p, on, lastb);
#pragma unroll
                for (int i = 0; i < HC; ++i) H[i] = L[i] = 0;
            }
        };
        // One loop over the stages of all tiles; it == nst: the next tile is due.
        int tile = (int)blockIdx.y - (int)gridDim.y, j = -1, g = 0, it = nst, kb = 0, blk = 0, h = 0;
        int ex0 = 0, ex1 = 0, er = 0, nplain = 0;
        if ((int)blockIdx.y < ntiles) {
#pragma unroll
            for (int u = 0; u < 3; ++u) load(u, blockIdx.y, 0);
        }
        while (ok) {
            bool plain = false, flush = false, end = false, told = false;
            if (it == nst) {
                tile += gridDim.y;
                ++j;
                end = tile >= ntiles;
                if (!end) {
                    h = j & 1;
                    ok = dg_wait_warp(&rb.keyfull[h], (j / 2) & 1, &b.give);
                    ex0 = ea[h][ar], ex1 = ea[h][ar + 8], er = ea[h][row];
                    const volatile int *f = rb.plain[h];
                    plain = cplain || f[0] || f[1] || f[2];
                    dg_arrive(&rb.keyfree[h]);
                    if (!plain) it = kb = blk = 0;
                }
                flush = open && (end || plain);
            }
            if (!end && !plain && ok) {
                const int s = g % DG_STAGES;
                // read ahead of the wait (where there are registers): behind the digits'
                // stores they would wait for those
                int f[8], fb[8];
                if constexpr (ONE) {
                    shifts(kb, akq, f);
                    shifts(kb, bkq, fb);
                }
                if (g >= DG_STAGES) ok = dg_wait_warp(&b.empty[s], (g / DG_STAGES - 1) & 1, &b.give);
                const bool lasts = it + 1 == nst, more = !lasts || tile + (int)gridDim.y < ntiles;
                const int nt = lasts ? tile + gridDim.y : tile, ni = lasts ? 0 : it + 1;
                if (ok) {
                    if constexpr (!ONE) shifts(kb, akq, f);
                    scale(va[0], f);
                    store_digits<T, NS>(va[0], ex0, adst + s * C::STAGE, C::SL_A, f);
                    if (more) load(0, nt, ni);
                    scale(va[1], f);
                    store_digits<T, NS>(va[1], ex1, adst + s * C::STAGE + 128, C::SL_A, f);
                    if (more) load(1, nt, ni);
                    if (hasb && g < bstages) {
                        if constexpr (!ONE) shifts(kb, bkq, fb);
#pragma unroll
                        for (int k = 0; k < 8; ++k) fb[k] = -c_shift(fb[k]);
                        store_digits<double, NS>(vb, eb[blk * BN + bcol], bdst + s * C::STAGE, C::SL_B, fb);
                    }
                    if (more && g + 1 < bstages) load(2, nt, ni);
                    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                    dg_arrive(&b.full[s]);
                }
                told = lasts;
                flush = kb % DG_DRAIN == 0 && open;
            }
            if (flush) readout();
            // behind the readout of the tile before, whose rows_read it waits for: a
            // thread that signalled twice without that wait (a tile of one stage)
            // would stand in for one that has not read its rows yet
            if (told) rows_read();
            if (end) break;
            if (plain) {
                // a row or column beyond the digits' range: plain sums, then the
                // same order as above (rows read by all, then written)
                const int64_t p = min((int64_t)tile * DG_M + row, a.npts - 1);
                T sum[NBLK * 32];
                for (int i = 0; i < NBLK * 32; ++i) {
                    const int c = (nb0 + i / 32) * BN + col0 + i % 32;
                    double t = 0;
                    if (owns && c < a.m)
                        for (int k = 0; k < a.n; ++k)
                            t = fma((double)a.X[p * a.ldx + k], __ldg(a.C + (int64_t)k * a.ldc + c), t);
                    sum[i] = (T)t;
                }
                // every converter of this CTA has read its row (a bounded wait: a warp
                // whose own wait has given up does not come)
                dg_arrive(&rb.sums);
                ok = dg_wait_warp(&rb.sums, nplain++ & 1, &b.give) && ok;
                rows_read();
                if (a.cluster) ok = dg_wait_warp(&rb.rd, j & 1, &b.give) && ok;
                if (owns && (int64_t)tile * DG_M + row < a.npts)
                    for (int i = 0; i < NBLK * 32; ++i) {
                        const int c = (nb0 + i / 32) * BN + col0 + i % 32;
                        if (c < a.m) {
                            T v = sum[i], *y = a.Y + p * a.ldy + c;
                            if (a.alpha != 1.0) v *= al;
                            if (a.beta != 0.0) v += be * *y;
                            *y = ok ? v : (T)__longlong_as_double(0x7ff8000000000000ll);
                        }
                    }
                if (tile + (int)gridDim.y < ntiles) {
#pragma unroll
                    for (int u = 0; u < 3; ++u) load(u, tile + gridDim.y, 0);
                }
            } else {
                if (kb % DG_DRAIN == DG_DRAIN - 1 || kb == kst - 1) {
                    open = true;
                    pend = kb == kst - 1;
                    ptile = tile, ptj = j, pe = er, pblk = blk;
                }
                ++it, ++g;
                if (++kb == kst) kb = 0, ++blk;
            }
        }
        if (!ok) {
            // a wait gave up: NaN in the tile before this one, which may not have been
            // stored, and in all that follow
            for (int t = max((int)blockIdx.y, tile - (int)gridDim.y); t < ntiles; t += gridDim.y) {
                const int64_t p = (int64_t)t * DG_M + row;
                if (!owns || p >= a.npts) continue;
#pragma unroll 1
                for (int i = 0; i < NBLK * 32; ++i) {
                    const int c = (nb0 + i / 32) * BN + col0 + i % 32;
                    if (c < a.m) a.Y[p * a.ldy + c] = (T)__longlong_as_double(0x7ff8000000000000ll);
                }
            }
        }
    }
    DG_FENCE_BEFORE();
    __syncthreads();
    if (tid == 0 && a.err && b.give.bad) atomicExch(a.err, 1);
    if (warp == DG_CW)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(b.tmem), "r"(C::TMEM) : "memory");
    // no CTA leaves while another may still signal it
    if (a.cluster) asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

// Launches a rotation kernel: gx column blocks, as many row workers as are
// resident at once; in place the column blocks of a row tile are a cluster.
template <typename Fn, typename Args>
int launch_rows(Fn fn, Args a, unsigned gx, size_t smem, bool in_place, cudaStream_t st) {
    a.cluster = in_place && gx > 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(gx, 1);
    cfg.blockDim = dim3(DG_NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = a.cluster ? gx : 1;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int workers = 0;
    if (a.cluster) {
        RS_CUDA(cudaOccupancyMaxActiveClusters(&workers, fn, &cfg));
    } else {
        RS_TRY(sm_count(&workers));
        workers /= (int)gx;
    }
    const int64_t tiles = (a.npts + DG_M - 1) / DG_M;
    cfg.gridDim.y = (unsigned)std::max<int64_t>(1, std::min<int64_t>(tiles, workers));
    RS_CUDA(cudaLaunchKernelEx(&cfg, fn, a));
    return RS_OK;
}

template <typename T, int NS, int BN, int NBLK, bool ONE> int launch_rot(RotArgs<T> a, bool in_place, cudaStream_t st) {
    using C = DgCfg<NS, BN, 32>;
    auto fn = k_digit_rot<T, NS, BN, NBLK, ONE>;
    const size_t smem = C::SMEM + sizeof(int) * (size_t)((a.n + DG_K - 1) / DG_K * DG_K);
    RS_TRY(smem_optin((const void *)fn, smem));
    return launch_rows(fn, a, (unsigned)((a.m + BN * NBLK - 1) / (BN * NBLK)), smem, in_place, st);
}

// ------------------------------------- FP32 rotation by BF16 pieces ---
// Y = alpha X C + beta Y to FP32 accuracy, for the eigensolver's inner steps
// and rs_rotate_block: every operand is the exact sum of three BF16 pieces
// (8 + 8 + 8 bits), and the six piece products of weight 2^-16 and up are
// summed in FP32 by the tensor core, the leading one apart from the others.
// The pieces need no exponent pass and a quarter of the digits' instructions.
//
// One CTA per SM, row tiles of 128 dealt round robin, one column block of BN per
// CTA; eight converter warps cut X into pieces, the pieces of C (made once by
// k_piece_c) come by bulk copies, four stages of 32 states ahead; two
// accumulator sets let the products of a tile run while the last one's are
// stored.  In place the CTAs of a row tile are a cluster, as in k_digit_rot.
// What it measured (658 416 rows, 256 -> 256 / 256 -> 64 columns): 685 / 302 us,
// 943 / 564 us for a split pass and a product kernel before.

struct PieceArgs {
    const float *X;
    const uint4 *Cp;     // [block][stage][8-step group][piece][column][8 steps] BF16
    float *Y;
    int64_t ldx, ldy, npts;
    int n, m;
    int vec, yvec, cluster;
    int spin, *err;      // as in GramArgs
    float alpha, beta;
};

constexpr int PC_ST = 4;   // stages

template <int BN> struct PcCfg {
    static constexpr int LBO_A = DG_M * 16 + 32, SL_A = KQ * LBO_A, A_BYTES = 3 * SL_A;
    static constexpr int SL_B = BN * 16, LBO_B = 3 * SL_B, B_BYTES = KQ * LBO_B;
    static constexpr int STAGE = A_BYTES + B_BYTES;
    static constexpr int TMEM = 4 * BN;   // two sets of (leading, other) products
    static constexpr size_t SMEM = (size_t)PC_ST * STAGE + 128;
};

// two values to one word per piece, the first in the low half
__device__ __forceinline__ void bf16_pieces(float x, float y, uint32_t (&p)[3]) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;\n" : "=r"(p[k]) : "f"(y), "f"(x));
        x -= __uint_as_float(p[k] << 16);
        y -= __uint_as_float(p[k] & 0xffff0000u);
    }
}

template <int BN> __global__ void k_piece_c(const double *__restrict__ C, int64_t ldc, int n, int m, int kst, uint4 *__restrict__ P) {
    // one thread per (block, stage, group, column)
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int col = t % BN, g = t / BN, kq = g % KQ, st = g / KQ % kst, blk = g / KQ / kst;
    const int c = blk * BN + col, k0 = st * DG_K + kq * 8;
    if (blk >= (m + BN - 1) / BN) return;
    uint32_t w[4][3];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int k = k0 + 2 * i;
        const float x = c < m && k < n ? (float)__ldg(C + (int64_t)k * ldc + c) : 0.f;
        const float y = c < m && k + 1 < n ? (float)__ldg(C + (int64_t)(k + 1) * ldc + c) : 0.f;
        bf16_pieces(x, y, w[i]);
    }
#pragma unroll
    for (int p = 0; p < 3; ++p) P[((int64_t)g * 3 + p) * BN + col] = make_uint4(w[0][p], w[1][p], w[2][p], w[3][p]);
}

template <int BN> __global__ void __launch_bounds__(DG_NT, 1) k_piece_rot(PieceArgs a) {
    using C = PcCfg<BN>;
    extern __shared__ __align__(128) unsigned char dgsm[];
    __shared__ uint64_t full[PC_ST], empty[PC_ST], accfull[2], accfree[2], rd, done;
    __shared__ uint32_t tmem_s;
    __shared__ DgGive give;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int kst = (a.n + DG_K - 1) / DG_K;
    const int ntiles = (int)((a.npts + DG_M - 1) / DG_M);
    if (tid == 0) {
        for (int i = 0; i < PC_ST; ++i) {
            dg_bar_init(&full[i], DG_CT + 1);
            dg_bar_init(&empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            dg_bar_init(&accfull[i], 1);
            dg_bar_init(&accfree[i], DG_CT);
        }
        dg_bar_init(&rd, DG_CT * (a.cluster ? gridDim.x : 1));
        dg_bar_init(&done, 1);
        give = {0, a.spin};
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == DG_CW) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(dg_su32(&tmem_s)), "r"(C::TMEM)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    DG_FENCE_BEFORE();
    __syncthreads();
    DG_FENCE_AFTER();
    if (a.cluster) asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");

    if (warp == DG_CW + 1) {
        // the pieces of C, stage by stage
        if (lane == 0) {
            int g = 0;
            bool ok = true;
            for (int tile = blockIdx.y; tile < ntiles && ok; tile += gridDim.y)
                for (int it = 0; it < kst; ++it, ++g) {
                    const int s = g % PC_ST;
                    if (g >= PC_ST && !dg_wait(&empty[s], (g / PC_ST - 1) & 1, &give)) {
                        ok = false;
                        break;
                    }
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(dg_su32(&full[s])), "r"(C::B_BYTES)
                                 : "memory");
                    asm volatile(
                        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                            dg_su32(dgsm + s * C::STAGE + C::A_BYTES)),
                        "l"(a.Cp + ((int64_t)blockIdx.x * kst + it) * (C::B_BYTES / 16)), "r"(C::B_BYTES), "r"(dg_su32(&full[s]))
                        : "memory");
                }
            // no copy is in flight when the CTA ends
            for (int q = g < PC_ST ? 0 : g - PC_ST; q < g; ++q)
                for (int i = 0; i < (*(volatile int *)&give.bad ? 64 : DG_SPIN) && !dg_try(&full[q % PC_ST], (q / PC_ST) & 1); ++i) {
                }
        }
    } else if (warp == DG_CW) {
        const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_s, 0), lead = lane == 0;
        const uint64_t da0 = dg_desc(dg_su32(dgsm), C::LBO_A), db0 = dg_desc(dg_su32(dgsm) + C::A_BYTES, C::LBO_B);
        constexpr uint32_t BF = (1u << 7) | (1u << 10);   // both operands BF16
        int g = 0, j = 0;
        bool ok = true;
        for (int tile = blockIdx.y; tile < ntiles && ok; tile += gridDim.y, ++j) {
            const uint32_t acc = tmem + (j & 1) * 2 * BN;
            if (j >= 2) ok = __all_sync(0xffffffffu, dg_wait(&accfree[j & 1], (j / 2 - 1) & 1, &give));
            DG_FENCE_AFTER();
            for (int it = 0; it < kst && ok; ++it, ++g) {
                const int s = g % PC_ST;
                ok = __all_sync(0xffffffffu, dg_wait(&full[s], (g / PC_ST) & 1, &give));
                DG_FENCE_AFTER();
                const uint64_t da = da0 + (uint64_t)(s * (C::STAGE >> 4)), db = db0 + (uint64_t)(s * (C::STAGE >> 4));
                if (ok) {
#pragma unroll
                    for (int k = 0; k < DG_K / 16; ++k) {
                        const uint64_t ka = (uint64_t)(2 * k * C::LBO_A >> 4), kb = (uint64_t)(2 * k * C::LBO_B >> 4);
                        auto A = [&](int i) { return da + ka + (uint64_t)(i * C::SL_A >> 4); };
                        auto B = [&](int i) { return db + kb + (uint64_t)(i * C::SL_B >> 4); };
                        const uint32_t on = it > 0 || k > 0;
                        // leading product and A0 B1 side by side, then the rest onto the latter
                        dg_mma(acc, A(0), B(0), dg_idesc(DG_M, 2 * BN) | BF, on, lead);
                        dg_mma(acc + BN, A(0), B(2), dg_idesc(DG_M, BN) | BF, 1u, lead);
                        dg_mma(acc + BN, A(1), B(0), dg_idesc(DG_M, BN) | BF, 1u, lead);
                        dg_mma(acc + BN, A(1), B(1), dg_idesc(DG_M, BN) | BF, 1u, lead);
                        dg_mma(acc + BN, A(2), B(0), dg_idesc(DG_M, BN) | BF, 1u, lead);
                    }
                }
                dg_commit(&empty[s], lead);
            }
            dg_commit(&accfull[j & 1], lead);
        }
        dg_commit(&done, lead);
        dg_settle(&done, 0);
    } else if (warp < DG_CW) {
        const int ar = warp * 16 + (lane >> 2), akq = lane & 3;
        unsigned char *adst = dgsm + akq * C::LBO_A + ar * 16;
        constexpr int CPT = BN / 2;   // columns per thread in the readout
        const int col0 = (warp >> 2) * CPT, row = (warp & 3) * 32 + lane;
        bool ok = true;
        float va[2][8];
        auto load = [&](int u, int tile, int it) {
            const int64_t r0 = (int64_t)tile * DG_M;
            const int rows = (int)min((int64_t)DG_M, a.npts - r0), k0 = it * DG_K + 8 * akq;
            {
                const float *x = a.X + (r0 + min(ar + 8 * u, rows - 1)) * a.ldx + k0;
                if (a.vec && k0 + 8 <= a.n) {
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const float4 t = reinterpret_cast<const float4 *>(x)[q];
                        va[u][4 * q] = t.x, va[u][4 * q + 1] = t.y, va[u][4 * q + 2] = t.z, va[u][4 * q + 3] = t.w;
                    }
                } else {
#pragma unroll
                    for (int k = 0; k < 8; ++k) va[u][k] = k0 + k < a.n ? x[k] : 0.f;
                }
            }
        };
        auto readout = [&](int tile, int j) {
            ok = ok && dg_wait_warp(&accfull[j & 1], (j / 2) & 1, &give);
            if (a.cluster) ok = dg_wait_warp(&rd, j & 1, &give) && ok;
            DG_FENCE_AFTER();
            const int64_t p = (int64_t)tile * DG_M + row;
            const uint32_t t0 = tmem_s + ((uint32_t)(warp & 3) * 32 << 16) + (j & 1) * 2 * BN + col0;
            const int cb = blockIdx.x * BN + col0;
            float *y = a.Y + p * a.ldy + cb;
#pragma unroll
            for (int c = 0; c < CPT; c += 32) {
                uint32_t r[32];
                float v[32];
                __syncwarp();   // rows beyond the last skipped the stores of the round before
                dg_tmem_ld32(t0 + BN + c, r);
#pragma unroll
                for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
                dg_tmem_ld32(t0 + c, r);
#pragma unroll
                for (int i = 0; i < 32; ++i) v[i] = ok ? a.alpha * (__uint_as_float(r[i]) + v[i]) : __int_as_float(0x7fffffff);
                if (c + 32 >= CPT) {
                    DG_FENCE_BEFORE();
                    dg_arrive(&accfree[j & 1]);
                }
                if (p >= a.npts) continue;
                if (a.yvec && cb + c + 32 <= a.m) {
                    float4 *y4 = reinterpret_cast<float4 *>(y + c);
                    if (a.beta != 0.f) {
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const float4 o = y4[q];
                            v[4 * q] += a.beta * o.x, v[4 * q + 1] += a.beta * o.y, v[4 * q + 2] += a.beta * o.z, v[4 * q + 3] += a.beta * o.w;
                        }
                    }
#pragma unroll
                    for (int q = 0; q < 8; ++q) y4[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                } else {
#pragma unroll
                    for (int i = 0; i < 32; ++i)
                        if (cb + c + i < a.m) y[c + i] = a.beta != 0.f ? v[i] + a.beta * y[c + i] : v[i];
                }
            }
        };
        int j = 0, g = 0, ptile = -1;
        if ((int)blockIdx.y < ntiles) {
            load(0, blockIdx.y, 0);
            load(1, blockIdx.y, 0);
        }
        for (int tile = blockIdx.y; tile < ntiles && ok; tile += gridDim.y, ++j) {
            for (int it = 0; it < kst && ok; ++it, ++g) {
                const int s = g % PC_ST;
                if (g >= PC_ST) ok = dg_wait_warp(&empty[s], (g / PC_ST - 1) & 1, &give);
                if (!ok) break;
                const bool last = it + 1 == kst;
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    uint32_t w[4][3];
#pragma unroll
                    for (int i = 0; i < 4; ++i) bf16_pieces(va[u][2 * i], va[u][2 * i + 1], w[i]);
#pragma unroll
                    for (int p = 0; p < 3; ++p)
                        *reinterpret_cast<uint4 *>(adst + s * C::STAGE + u * 128 + p * C::SL_A) =
                            make_uint4(w[0][p], w[1][p], w[2][p], w[3][p]);
                    if (!last || tile + (int)gridDim.y < ntiles) load(u, last ? tile + gridDim.y : tile, last ? 0 : it + 1);
                }
                asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                dg_arrive(&full[s]);
                // the readout waits for rd of the tile before: ahead of this tile's
                // arrival, or a thread would count twice in one phase (n <= 32: the
                // first stage is the last) and rows be overwritten before a peer reads them
                if (it == 0 && ptile >= 0) readout(ptile, j - 1);
                if (last && a.cluster)
                    for (int r = 0; r < (int)gridDim.x; ++r)
                        asm volatile(
                            "{\n .reg .b32 ra;\n mapa.shared::cluster.u32 ra, %0, %1;\n"
                            " mbarrier.arrive.release.cluster.shared::cluster.b64 _, [ra];\n}\n" ::"r"(dg_su32(&rd)),
                            "r"(r)
                            : "memory");
            }
            ptile = tile;
        }
        if (ptile >= 0) readout(ptile, j - 1);
        if (!ok)   // as in k_digit_rot
            for (int t = max((int)blockIdx.y, ptile - (int)gridDim.y); t < ntiles; t += gridDim.y) {
                const int64_t p = (int64_t)t * DG_M + row;
                const int cb = blockIdx.x * BN + col0;
                if (p >= a.npts) continue;
#pragma unroll 1
                for (int i = 0; i < CPT && cb + i < a.m; ++i) a.Y[p * a.ldy + cb + i] = __int_as_float(0x7fffffff);
            }
    }
    DG_FENCE_BEFORE();
    __syncthreads();
    if (tid == 0 && a.err && give.bad) atomicExch(a.err, 1);
    if (warp == DG_CW)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_s), "r"(C::TMEM) : "memory");
    // no CTA leaves while another may still signal it
    if (a.cluster) asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

template <int BN> int launch_piece(PieceArgs a, const double *C, int64_t ldc, void *work, bool in_place, cudaStream_t st) {
    using P = PcCfg<BN>;
    auto fn = k_piece_rot<BN>;
    RS_TRY(smem_optin((const void *)fn, P::SMEM));
    const int kst = (a.n + DG_K - 1) / DG_K;
    const unsigned gx = (unsigned)((a.m + BN - 1) / BN);
    const int64_t nc = (int64_t)gx * kst * KQ * BN;
    k_piece_c<BN><<<(unsigned)((nc + 127) / 128), 128, 0, st>>>(C, ldc, a.n, a.m, kst, (uint4 *)work);
    RS_LAUNCH_CHECK();
    a.Cp = (const uint4 *)work;
    return launch_rows(fn, a, gx, P::SMEM, in_place, st);
}

// ------------------------------------- FP32 overlap by BF16 pieces ---
// S += dV X^T Y to FP32 accuracy: the six piece products of a chunk of at most
// 2048 points are summed in FP32 by the tensor core, chunks meet in FP64.  The
// converters cut both operands into pieces on the way to shared memory, so that
// an FP32 value is read once per tile and no pieces are written.  Work items (chunk,
// tile), tiles fastest, are dealt round robin to one CTA per SM; the readout of
// an item overlaps the products of the next.
// Measured (658 416 points): 256 x 64 columns 340 us, 256 x 256 790 us; 800 and
// 1382 us with a separate pass that wrote the pieces to memory.

struct PieceGramArgs {
    const float *X, *Y;
    int64_t ldx, ldy, npts, lds;
    int nx, ny;
    double *S;
    double dV;
    int tiles_n, tiles, chunks, kb;   // kb: 64-point stages per chunk
    int spin, *err;                   // as in GramArgs
};

constexpr int PG_K = 64, PG_KQ = PG_K / 8, PG_ST = 2;

template <int BN> struct PgCfg {
    static constexpr int LBO_A = DG_M * 16, SL_A = PG_KQ * LBO_A, A_BYTES = 3 * SL_A;
    static constexpr int LBO_B = BN * 16, SL_B = PG_KQ * LBO_B, STAGE = A_BYTES + 3 * SL_B;
    static constexpr int TMEM = 2 * BN;
    static constexpr size_t SMEM = (size_t)PG_ST * STAGE + 128;
};

template <int BN> __global__ void __launch_bounds__(DG_NT, 1) k_piece_gram(PieceGramArgs a) {
    using C = PgCfg<BN>;
    extern __shared__ __align__(128) unsigned char dgsm[];
    __shared__ uint64_t full[PG_ST], empty[PG_ST], accfull[2], accfree[2], done;
    __shared__ uint32_t tmem_s;
    __shared__ DgGive give;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int items = a.tiles * a.chunks, nkb = (int)((a.npts + PG_K - 1) / PG_K);
    if (tid == 0) {
        for (int i = 0; i < PG_ST; ++i) {
            dg_bar_init(&full[i], DG_CT);
            dg_bar_init(&empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            dg_bar_init(&accfull[i], 1);
            dg_bar_init(&accfree[i], DG_CT);
        }
        dg_bar_init(&done, 1);
        give = {0, a.spin};
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == DG_CW) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(dg_su32(&tmem_s)), "r"(C::TMEM)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    DG_FENCE_BEFORE();
    __syncthreads();
    DG_FENCE_AFTER();
    auto stages_of = [&](int item) { return min(a.kb, nkb - item / a.tiles * a.kb); };

    if (warp == DG_CW) {
        const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_s, 0), lead = lane == 0;
        const uint64_t da0 = dg_desc(dg_su32(dgsm), C::LBO_A), db0 = dg_desc(dg_su32(dgsm) + C::A_BYTES, C::LBO_B);
        constexpr uint32_t idesc = dg_idesc(DG_M, BN) | (1u << 7) | (1u << 10);   // both operands BF16
        int g = 0, j = 0;
        bool ok = true;
        for (int item = blockIdx.x; item < items && ok; item += gridDim.x, ++j) {
            const uint32_t acc = tmem + (j & 1) * BN;
            const int nst = stages_of(item);
            if (j >= 2) ok = dg_wait_warp(&accfree[j & 1], (j / 2 - 1) & 1, &give);
            DG_FENCE_AFTER();
            for (int it = 0; it < nst && ok; ++it, ++g) {
                const int s = g % PG_ST;
                ok = dg_wait_warp(&full[s], (g / PG_ST) & 1, &give);
                DG_FENCE_AFTER();
                const uint64_t da = da0 + (uint64_t)(s * (C::STAGE >> 4)), db = db0 + (uint64_t)(s * (C::STAGE >> 4));
                if (ok) {
                    // pieces (0,0) (0,1) (1,0) (0,2) (1,1) (2,0), each over the stage's four steps of 16
#pragma unroll
                    for (int pr = 0; pr < 6; ++pr) {
                        constexpr int pa[6] = {0, 0, 1, 0, 1, 2}, pb[6] = {0, 1, 0, 2, 1, 0};
#pragma unroll
                        for (int k = 0; k < PG_K / 16; ++k)
                            dg_mma(acc, da + (uint64_t)((pa[pr] * C::SL_A + 2 * k * C::LBO_A) >> 4),
                                   db + (uint64_t)((pb[pr] * C::SL_B + 2 * k * C::LBO_B) >> 4), idesc,
                                   (it > 0 || pr > 0 || k > 0) ? 1u : 0u, lead);
                    }
                }
                dg_commit(&empty[s], lead);
            }
            dg_commit(&accfull[j & 1], lead);
        }
        dg_commit(&done, lead);
        dg_settle(&done, 0);
    } else if (warp < DG_CW) {
        // units (32 columns, 8 points): 4 x 8 of X, BN / 32 x 8 of Y; warp w takes
        // the points 8 w .. of every column group
        constexpr int NA = DG_M / 32, NU = NA + BN / 32;
        float v[NU][8];
        bool ok = true;
        auto column = [&](int tile, int u) {
            const int m0 = tile / a.tiles_n * DG_M, n0 = tile % a.tiles_n * BN;
            return u < NA ? m0 + u * 32 + lane : n0 + (u - NA) * 32 + lane;
        };
        auto load = [&](int item, int it) {
            const int tile = item % a.tiles;
            const int64_t p = ((int64_t)(item / a.tiles) * a.kb + it) * PG_K + 8 * warp;
#pragma unroll
            for (int u = 0; u < NU; ++u) {
                const bool isx = u < NA;
                const int c = column(tile, u);
                const bool in = c < (isx ? a.nx : a.ny);
                const int64_t ld = isx ? a.ldx : a.ldy;
                const float *src = (isx ? a.X : a.Y) + p * ld + c;
                // columns beyond the last are zero
#pragma unroll
                for (int k = 0; k < 8; ++k) v[u][k] = in && p + k < a.npts ? __ldg(src + k * ld) : 0.f;
            }
        };
        constexpr int CPT = BN / 2;
        const int col0 = (warp >> 2) * CPT, row = (warp & 3) * 32 + lane;
        auto readout = [&](int item, int j) {
            ok = ok && dg_wait_warp(&accfull[j & 1], (j / 2) & 1, &give);
            DG_FENCE_AFTER();
            const int tile = item % a.tiles, i = tile / a.tiles_n * DG_M + row, c0 = tile % a.tiles_n * BN + col0;
            const uint32_t t0 = tmem_s + ((uint32_t)(warp & 3) * 32 << 16) + (j & 1) * BN + col0;
            double *srow = a.S + (int64_t)i * a.lds + c0;
#pragma unroll
            for (int c = 0; c < CPT; c += 32) {
                uint32_t r[32];
                __syncwarp();   // rows beyond the last skipped the sums of the round before
                dg_tmem_ld32(t0 + c, r);
                if (c + 32 >= CPT) {
                    DG_FENCE_BEFORE();
                    dg_arrive(&accfree[j & 1]);
                }
                if (i < a.nx) {
#pragma unroll
                    for (int q = 0; q < 32; ++q)
                        if (c0 + c + q < a.ny)
                            atomicAdd(srow + c + q, ok ? a.dV * (double)__uint_as_float(r[q]) : __longlong_as_double(0x7ff8000000000000ll));
                }
            }
        };
        int j = 0, g = 0, pitem = -1;
        if ((int)blockIdx.x < items) load(blockIdx.x, 0);
        for (int item = blockIdx.x; item < items && ok; item += gridDim.x, ++j) {
            const int nst = stages_of(item);
            for (int it = 0; it < nst && ok; ++it, ++g) {
                const int s = g % PG_ST;
                if (g >= PG_ST) ok = dg_wait_warp(&empty[s], (g / PG_ST - 1) & 1, &give);
                if (!ok) break;
                unsigned char *st = dgsm + s * C::STAGE + lane * 16;
#pragma unroll
                for (int u = 0; u < NU; ++u) {
                    uint32_t w[4][3];
#pragma unroll
                    for (int i = 0; i < 4; ++i) bf16_pieces(v[u][2 * i], v[u][2 * i + 1], w[i]);
                    unsigned char *d = u < NA ? st + warp * C::LBO_A + u * 512 : st + C::A_BYTES + warp * C::LBO_B + (u - NA) * 512;
#pragma unroll
                    for (int p = 0; p < 3; ++p)
                        *reinterpret_cast<uint4 *>(d + p * (u < NA ? C::SL_A : C::SL_B)) = make_uint4(w[0][p], w[1][p], w[2][p], w[3][p]);
                }
                asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                dg_arrive(&full[s]);
                const bool last = it + 1 == nst;
                const int ni = last ? item + gridDim.x : item;
                if (ni < items) load(ni, last ? 0 : it + 1);
                if (it == 0 && pitem >= 0) readout(pitem, j - 1);
            }
            pitem = item;
        }
        if (pitem >= 0) readout(pitem, j - 1);
        if (!ok)   // a wait gave up: NaN in the tiles of the item before the last one tried and of all that follow
            for (int item = max((int)blockIdx.x, pitem - (int)gridDim.x); item < items; item += gridDim.x) {
                const int tile = item % a.tiles, i = tile / a.tiles_n * DG_M + row, c0 = tile % a.tiles_n * BN + col0;
                if (i >= a.nx) continue;
#pragma unroll 1
                for (int q = 0; q < CPT && c0 + q < a.ny; ++q)
                    atomicAdd(a.S + (int64_t)i * a.lds + c0 + q, __longlong_as_double(0x7ff8000000000000ll));
            }
    }
    DG_FENCE_BEFORE();
    __syncthreads();
    if (tid == 0 && a.err && give.bad) atomicExch(a.err, 1);
    if (warp == DG_CW)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_s), "r"(C::TMEM) : "memory");
}

template <int BN> int launch_piece_gram(PieceGramArgs a, cudaStream_t st) {
    using C = PgCfg<BN>;
    RS_TRY(smem_optin((const void *)k_piece_gram<BN>, C::SMEM));
    a.tiles_n = (a.ny + BN - 1) / BN;
    a.tiles = (a.nx + DG_M - 1) / DG_M * a.tiles_n;
    // chunks: enough for 148 CTAs, of at most 2048 points.  (148, not this chip's
    // 152: the chunks are the FP32 sums of a result, which stay what they were with the kernel
    // before this one; they bind below 303 104 points divided by the tiles, where 4 SMs idle.)
    const int64_t nkb = (a.npts + PG_K - 1) / PG_K;
    const int64_t want = std::max<int64_t>(1, std::min<int64_t>(nkb, (148 + a.tiles - 1) / a.tiles));
    a.kb = (int)std::min<int64_t>((nkb + want - 1) / want, 2048 / PG_K);
    a.chunks = (int)((nkb + a.kb - 1) / a.kb);
    int nsm = 0;
    RS_TRY(sm_count(&nsm));
    if ((int64_t)a.tiles * a.chunks > INT32_MAX) return fail(RS_EINVAL, "piece_gram: too many tiles");
    k_piece_gram<BN><<<(unsigned)std::min(nsm, a.tiles * a.chunks), DG_NT, C::SMEM, st>>>(a);
    RS_LAUNCH_CHECK();
    return RS_OK;
}

}  // namespace

// In place, the CTAs of a row tile are one cluster of at most 8 (64 columns
// each, or two blocks of 64).  A contraction of more than 1536 states could
// leave the 51 bits that dg_value takes.
bool digit_rot_takes(int n, int m, bool in_place) {
    return n <= 1536 && (!in_place || m <= 1024);
}

template <typename T>
int digit_rot(const T *X, int64_t ldx, int n, const double *C, int64_t ldc, int m, T *Y, int64_t ldy, int64_t npts,
              double alpha, double beta, const int *xkeys, cudaStream_t st, int *err) {
    RotArgs<T> a{};
    a.X = X, a.C = C, a.Y = Y, a.xk = xkeys, a.ldx = ldx, a.ldc = ldc, a.ldy = ldy, a.npts = npts, a.n = n, a.m = m;
    a.alpha = alpha, a.beta = beta, a.spin = t_rot_spin, a.err = err;
    a.vec = aligned16(X) && (ldx * (int64_t)sizeof(T)) % 16 == 0;
    a.yvec = aligned16(Y) && (ldy * (int64_t)sizeof(T)) % 16 == 0;
    constexpr int NS = sizeof(T) == 8 ? 8 : 5;
    const bool in_place = X == Y;
    const bool one = n <= DG_DRAIN * DG_K;
    if (m <= 32) return one ? launch_rot<T, NS, 32, 1, true>(a, false, st) : launch_rot<T, NS, 32, 1, false>(a, false, st);
    if (in_place && m > 512) return launch_rot<T, NS, 64, 2, false>(a, true, st);
    return one ? launch_rot<T, NS, 64, 1, true>(a, in_place, st) : launch_rot<T, NS, 64, 1, false>(a, in_place, st);
}
template int digit_rot<double>(const double *, int64_t, int, const double *, int64_t, int, double *, int64_t, int64_t,
                               double, double, const int *, cudaStream_t, int *);
template int digit_rot<float>(const float *, int64_t, int, const double *, int64_t, int, float *, int64_t, int64_t, double,
                              double, const int *, cudaStream_t, int *);

}  // namespace rs

namespace rs {

int64_t piece_rot_bytes(int n, int m) {
    const int64_t BN = m <= 64 ? 64 : 128;
    return (m + BN - 1) / BN * BN * ((n + DG_K - 1) / DG_K) * DG_K * 6;
}

int piece_gram(const float *X, int64_t ldx, int nx, const float *Y, int64_t ldy, int ny, int64_t npts, double dV, double *S,
               int64_t lds, cudaStream_t st, int *err) {
    k_digit_init<<<(unsigned)std::min<int64_t>(256, ((int64_t)nx * ny + 255) / 256), 256, 0, st>>>(S, lds, nx, ny, nullptr, 0);
    RS_LAUNCH_CHECK();
    PieceGramArgs a{};
    a.X = X, a.Y = Y, a.ldx = ldx, a.ldy = ldy, a.npts = npts, a.lds = lds, a.nx = nx, a.ny = ny, a.S = S, a.dV = dV;
    a.spin = t_gram_spin, a.err = err;
    return ny <= 64 ? launch_piece_gram<64>(a, st) : launch_piece_gram<128>(a, st);
}

int piece_rot(const float *X, int64_t ldx, int n, const double *C, int64_t ldc, int m, float *Y, int64_t ldy, int64_t npts,
              double alpha, double beta, void *work, cudaStream_t st, int *err) {
    PieceArgs a{};
    a.X = X, a.Y = Y, a.ldx = ldx, a.ldy = ldy, a.npts = npts, a.n = n, a.m = m;
    a.vec = aligned16(X) && ldx % 4 == 0;
    a.yvec = aligned16(Y) && ldy % 4 == 0;
    a.alpha = (float)alpha, a.beta = (float)beta, a.spin = t_rot_spin, a.err = err;
    if (m <= 64) return launch_piece<64>(a, C, ldc, work, X == Y, st);
    return launch_piece<128>(a, C, ldc, work, X == Y, st);
}

}  // namespace rs

// ---------------------------------------------------------------- C ABI ---

using namespace rs;

namespace {
int64_t round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

// the pieces of C are stored and copied 16 bytes at a time
int check_work(const void *work) {
    if (!work) return fail(RS_EINVAL, "tensor-core call: null workspace");
    if (!aligned16(work)) return fail(RS_EINVAL, "tensor-core call: workspace not on a 16-byte boundary");
    return RS_OK;
}

// the status word of the call's waits: the last 256 bytes of the workspace
int clear_status(void *work, int64_t bytes, int **err, cudaStream_t st) {
    *err = reinterpret_cast<int *>((char *)work + bytes - 256);
    RS_CUDA(cudaMemsetAsync(*err, 0, sizeof(int), st));
    return RS_OK;
}
int read_status(const int *err, cudaStream_t st) {
    int e = 0;
    RS_CUDA(cudaMemcpyAsync(&e, err, sizeof(int), cudaMemcpyDeviceToHost, st));
    RS_CUDA(cudaStreamSynchronize(st));
    if (e) return fail(RS_ETIMEOUT, "tensor-core call: a pipeline wait timed out");
    return RS_OK;
}
}  // namespace

extern "C" int64_t rs_tc_workspace_bytes(int64_t rows_a, int64_t rows_b, int64_t K) {
    if (rows_a < 1 || rows_b < 1 || K < 1) return -1;
    return 6 * (round_up(rows_a, 128) + round_up(rows_b, 128)) * round_up(K, 64) + 4352;
}

extern "C" int rs_overlap_block_tc(const rs_grid *g, const float *X_dev, int64_t ldx, int nx, const float *Y_dev,
                                   int64_t ldy, int ny, double *S_dev, int64_t lds, void *work_dev, void *stream) {
    if (!g || !X_dev || !Y_dev || !S_dev) return fail(RS_EINVAL, "rs_overlap_block_tc: null argument");
    if (nx < 1 || ny < 1 || ldx < nx || ldy < ny || lds < ny) return fail(RS_EINVAL, "rs_overlap_block_tc: bad sizes");
    RS_TRY(check_work(work_dev));
    cudaStream_t st = (cudaStream_t)stream;
    int *err = nullptr;
    RS_TRY(clear_status(work_dev, rs_tc_workspace_bytes(nx, ny, g->npts), &err, st));
    RS_TRY(piece_gram(X_dev, ldx, nx, Y_dev, ldy, ny, g->npts, g->h * g->h * g->h, S_dev, lds, st, err));
    return read_status(err, st);
}

extern "C" int rs_rotate_block(const float *X_dev, int64_t ldx, int n, const double *C_dev, int64_t ldc, int m,
                               float *Y_dev, int64_t ldy, int64_t npts, void *work_dev, void *stream) {
    if (!X_dev || !C_dev || !Y_dev) return fail(RS_EINVAL, "rs_rotate_block: null argument");
    if (n < 1 || m < 1 || npts < 1 || ldx < n || ldy < m || ldc < m) return fail(RS_EINVAL, "rs_rotate_block: bad sizes");
    RS_TRY(check_work(work_dev));
    cudaStream_t st = (cudaStream_t)stream;
    int *err = nullptr;
    RS_TRY(clear_status(work_dev, rs_tc_workspace_bytes(npts, m, n), &err, st));
    RS_TRY(rotate_any(X_dev, ldx, n, C_dev, ldc, m, Y_dev, ldy, npts, 1.0, 0.0, work_dev, st, err));
    return read_status(err, st);
}

extern "C" int rs_contraction_wait_limit(int overlap_tests, int rotation_tests) {
    t_gram_spin = overlap_tests < 0 ? DG_SPIN : overlap_tests;
    t_rot_spin = rotation_tests < 0 ? DG_SPIN : rotation_tests;
    return RS_OK;
}
