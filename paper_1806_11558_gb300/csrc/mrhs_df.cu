// mrhs_df.cu -- the product of the FP64 master with up to 16 right-hand
// sides (the H-matvec of Sec. 2.3) on the tensor cores, for the FP64 residuals
// of the iterative refinement and hm_matvec_block(HM_F64).
//
// GB300 runs FP64 FMAs at 2 per SM and clock, FP32 FMAs at 128 and 16-bit
// tensor multiply-adds at ~1,000 (mma.sync): 16 FP64 products are bound by the
// FP64 pipe, and compensated sums of float pairs (12 FP32 operations per entry
// and right-hand side) by the FP32 pipe.  Here entries and vectors are cut into
// digits base 256 whose products the tensor cores add without rounding (the
// error-free slicing of Ozaki, Ogita, Oishi and Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication and its applications", Numer. Algorithms 2012):
//   * column k of a panel has the exponent e_k of its largest x_r (each x_r
//     scaled by its own mean exponent first) and x_r 2^-e_k becomes an integer
//     of 62 bits and sign, eight balanced digits d in [-128, 127], as FP16;
//   * a term w 2^e_k of a row becomes an integer of 62 bits or less and sign on
//     the scale of the row's largest term so far, in integer operations on the
//     bits of w: eight digits, the top one signed, the others in [0, 255], as
//     FP16 subnormals (u 2^-24, which are the digit's own bits);
//   * of the 64 products of digits the 36 of order i + j <= 7 are formed by
//     mma.m16n8k16 and summed by order: integers below 2^24 times 2^-24, exact
//     in FP32 over 128 columns (orders 4 to 7, worth 2^-32 and less, may round);
//   * the sums are put together as a float pair, without loss for the orders 0
//     to 4, and added to a running pair (TwoSum): every 128 columns, or where a
//     larger term raises the row's scale.
// The scales of columns and rows are those of the largest of 16 right-hand sides.
// Eight digits leave 15 bits for a right-hand side that is smaller there than
// others and has still what a pair of floats keeps (48 bits of an entry and of an x);
// each sum keeps a record of the right-hand sides that had a term of their own
// of that size (NEAR_X and after), and the clusters where one had none are formed
// again in pairs of floats, where no right-hand side sees another.  Seven digits
// and no record were 12% to 19% faster (64,980 panels 1.73 ms a pass) and lost a unit
// vector's entries 10^7 below another's to 2e-9.
// Against the exact product (16 right-hand sides, 1,280 and 2,880 panels) the
// error is 2e-16 of |H||x| in norm for random, 2.3e-15 for positive x and 1.7e-15
// for unit vectors; float pairs throughout have 2e-15, 1.1e-14 and 2.2e-15.
// Time of a pass with 16 right-hand sides, float pairs -> this (HBM alone), ms:
// 5,120 panels 0.415 -> 0.189, 64,980 panels, leaves of 64 rows, 4.59 -> 1.94 (0.48; row
// pass 1.14, column pass 0.57), 327,680 panels, leaves of 80, 26.8 -> 15.6 (3.4; row 9.4,
// column 5.2).  Vectors whose sizes differ by 1e10 between the halves of the sphere,
// so that most clusters are formed again: 0.43, 6.1 and 34 ms.
// Non-finite x or entries give NaN in the rows they reach.
//
//   scale_x / digits_x    : the scale of each x_r, the digits of x
//   col_fx_kernel         : per leaf column cluster kappa the partials
//                           x_kappa^T W of its column panel
//   col_pairs_kernel      : the partials of the listed clusters, in float pairs
//   tsum_fx_kernel        : t_b = sum of b's partials in increasing cluster
//                           order, and its digits
//   row_fx_kernel         : per leaf row cluster, the near-field panel times
//                           the gathered x and the U panel times the gathered t
//   row_reduce_kernel     : the sums of the rows whose panels were split
//   pairs / row_pairs     : the rows of the listed clusters, in float pairs
#include <cuda_fp16.h>

#include <algorithm>
#include <vector>

#include "hm_internal.cuh"

namespace hm {
namespace fx {

constexpr int MR = 16;              // right-hand sides of a pass
constexpr int NA = 8;               // digits of an entry, and of an x
constexpr int NO = 6;               // sums kept: the orders 0 to 5, and with the last 6 / 2^8 and 7 / 2^16
constexpr int DIG = NA * MR;        // halves per row of digits ([digit, top first][rhs])
constexpr int XSTRIDE = 2 * DIG + 16;  // bytes per staged row: 8 rows hit different banks (ldmatrix)
constexpr int QB = 62;              // bits of an integer x
constexpr int E_ZERO = -900;        // exponent of a column of zeros, and the smallest one
constexpr int E_BIAS = 1000;        // added to the exponents of columns, which makes them positive
constexpr int F_EXP = 884;          // a row's factor 2^(E - 1011) as a float: exponent field E - 884
constexpr int E_NAN = F_EXP + 255;  // biased term exponents from here on: not finite, or beyond FP32
// A sum is taken as it is where one of its terms has an x_r within 2^NEAR_X of the
// column's largest and an entry within 2^NEAR_W of the row's scale, or within 2^FAR_X
// and 2^FAR_W (a column of a panel: RAISED more), or in a row within RAISED more by later
// terms that raised the scale: the 2^-61.5 of the scale that a term may be off is then
// 2^-46.5 of that term or less, which is what pairs of floats make of a product.  The
// first kind finds right-hand sides beside another's peak, whose own terms are
// elsewhere and of full size; the second finds those that are smooth and small in a
// whole cluster.  Within a row the scale is mostly raised by the diagonal, or late in U
// by 2; without RAISED one row cluster in some 1,000 of random vectors was unsure.
constexpr int NEAR_X = 2, NEAR_W = 9, FAR_X = 6, FAR_W = 5, RAISED = 3;

// (s, c) += (s2, c2)
__device__ __forceinline__ void dadd(float &s, float &c, float s2, float c2) {
    const float t = __fadd_rn(s, s2);
    const float bp = __fsub_rn(t, s);
    const float sg = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(s2, bp));
    s = t;
    c = __fadd_rn(c, __fadd_rn(c2, sg));
}

// (s, c) -> (h, l) with h = fl(s + c), h + l = s + c exactly (TwoSum)
__device__ __forceinline__ void norm2(float s, float c, float &h, float &l) {
    h = __fadd_rn(s, c);
    const float bp = __fsub_rn(h, s);
    l = __fadd_rn(__fsub_rn(s, __fsub_rn(h, bp)), __fsub_rn(c, bp));
}

__device__ __forceinline__ uint32_t saddr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
template <int N> __device__ __forceinline__ void cp_async(void *dst, const void *src, bool pred) {
    if (N == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(saddr(dst)), "l"(src), "r"(pred ? 16 : 0)
                     : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(saddr(dst)), "l"(src), "r"(pred ? 8 : 0)
                     : "memory");
}

__device__ __forceinline__ void mma_f16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// ---------------------------------------------------------------------------
// digits of the vectors
// ---------------------------------------------------------------------------
// What the scale of an x_r is taken from: its largest exponent, the sum and the
// number of the exponents of its entries (finite and not zero; the exponent of x is e
// where 2^(e-1) <= |x| < 2^e).  All zero at the start.
struct Scale {
    long long sum;
    unsigned int count;
    unsigned int top;  // largest e + 1100
};

__global__ void __launch_bounds__(256) scale_x_kernel(const double *__restrict__ x, int64_t n, Scale *__restrict__ sc) {
    const double *xr = x + (int64_t)blockIdx.y * n;
    int sum = 0, count = 0;  // 256 CTAs: less than 2^20 entries a thread
    unsigned int top = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int eb = (__double2hiint(xr[i]) >> 20) & 0x7ff;
        if (eb != 0 && eb != 0x7ff) {
            sum += eb - 1022;
            ++count;
            top = max(top, (unsigned int)(eb - 1022 + 1100));
        }
    }
    top = __reduce_max_sync(0xffffffffu, top);
    count = __reduce_add_sync(0xffffffffu, count);
    const int lo = __reduce_add_sync(0xffffffffu, sum & 0xffff), hi = __reduce_add_sync(0xffffffffu, sum >> 16);
    if ((threadIdx.x & 31) == 0 && count) {
        Scale *o = sc + blockIdx.y;
        atomicMax(&o->top, top);
        atomicAdd(&o->count, (unsigned int)count);
        atomicAdd(reinterpret_cast<unsigned long long *>(&o->sum), (unsigned long long)((long long)hi * 65536 + lo));
    }
}

// x_r is scaled by 2^-scale: its mean exponent, so that right-hand sides of like size have
// like digits where one of them has a peak (by the largest entry instead, a
// peak of 4,096 in 40 of 655,220 panels made all clusters unsure), but no peak above 2^30
__device__ __forceinline__ int scale_of(const Scale &sc) {
    if (sc.count == 0) return 0;
    return max((int)(sc.sum / (long long)sc.count), (int)sc.top - 1100 - 30);
}

// the eight digits of q, |q| <= 2^62, as halves at o[0], o[MR], ... (top first)
constexpr unsigned long long DIGIT_BIAS = 0x8080808080808080ull;
__device__ __forceinline__ void store_digits(long long q, __half *o) {
    const unsigned long long u = (unsigned long long)q + DIGIT_BIAS;
#pragma unroll
    for (int j = 0; j < NA; ++j) o[(NA - 1 - j) * MR] = __int2half_rn((int)((u >> (8 * j)) & 0xffu) - 128);
}

// Xd[m] = the digits of x_r 2^-(scale_r + e), Xe[m] = ((e + E_BIAS) 2^20, state of
// the x_r), for position m (x is [nr][n], original order when perm is given);
// zeros for r >= nr.  16 lanes per position.  State: bit r and bit r + 16 of x_r are
// 00 zero, 01 (the upper) small beside the column's largest, 11 within 2^NEAR_X of
// it, 10 not finite; and bit r of the exponent's word: within 2^FAR_X or not finite.
__global__ void __launch_bounds__(256) digits_x_kernel(const double *__restrict__ x, int64_t n, int nr,
                                                       const int32_t *__restrict__ perm,
                                                       const Scale *__restrict__ sc, __half *__restrict__ Xd,
                                                       uint2 *__restrict__ Xe) {
    const int r = threadIdx.x & 15;
    const int S = r < nr ? scale_of(sc[r]) : 0;
    const int64_t n2 = (n + 1) / 2 * 2;  // whole warps (two positions each)
    for (int64_t m = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 4; m < n2;
         m += ((int64_t)gridDim.x * blockDim.x) >> 4) {
        const double v = m < n && r < nr ? x[(int64_t)r * n + (perm ? perm[m] : m)] : 0.0;
        const unsigned long long b = (unsigned long long)__double_as_longlong(v);
        const int eb = (int)(b >> 52) & 0x7ff;
        const bool bad = eb == 0x7ff;
        const int ex = eb == 0 || bad ? E_ZERO : max(eb - 1022 - S, E_ZERO);
        int e = ex;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
        // the mantissa (53 bits) on the column's scale, rounded to nearest
        long long q = 0;
        const int sh = e - ex;
        const unsigned int lo = __ballot_sync(0xffffffffu, bad || (eb != 0 && sh <= NEAR_X));
        const unsigned int lf = __ballot_sync(0xffffffffu, bad || (eb != 0 && sh <= FAR_X));
        const unsigned int up = __ballot_sync(0xffffffffu, !bad && eb != 0);
        if (eb != 0 && !bad && sh < 63) {
            const unsigned long long mant = (b & 0xfffffffffffffull) | 0x10000000000000ull;
            q = (long long)(((mant << (QB - 53)) + ((1ull << sh) >> 1)) >> sh);
            if ((long long)b < 0) q = -q;
        }
        if (m < n) {
            store_digits(q, Xd + m * DIG + r);
            if (r == 0)
                Xe[m] = make_uint2((uint32_t)(e + E_BIAS) << 20 | (lf >> (threadIdx.x & 16) & 0xffffu),
                                   (lo >> (threadIdx.x & 16) & 0xffffu) | (up >> (threadIdx.x & 16)) << 16);
        }
    }
}

// ---------------------------------------------------------------------------
// digits of the entries and the products
// ---------------------------------------------------------------------------
// A row of a tile keeps one exponent E (in the top 12 bits of E20) for the
// terms it is summing: at least that of the largest term so far and HEADROOM
// more when it has to rise, which ends the sums so far (flush).  It starts so
// high that zero and subnormal entries (exponent field 0) are shifted out
// whatever their column's exponent.
constexpr uint32_t HEADROOM = 1u << 20;
constexpr uint32_t E20_START = (uint32_t)(E_BIAS + 320) << 20;

// exponent (biased by 1023 + E_BIAS, times 2^20, plus some fraction bits) of the term w 2^e;
// the states in the lower bits of e20 may make it one more, no less
__device__ __forceinline__ uint32_t term_exp(double w, uint32_t e20) {
    return ((uint32_t)__double2hiint(w) & 0x7fffffffu) + e20;
}

// E20 for terms up to tm where the present one is too small, else the present one
__device__ __forceinline__ uint32_t raise_exp(uint32_t tm, uint32_t E20) {
    return tm < E20 + 0x100000u ? E20 : (tm & 0xfff00000u) + HEADROOM;
}

// w 2^(e - E) as 63-bit fixed point plus 2^63: bytes 7..0 are the digits (the
// top one plus 128); returns E minus the term's exponent.  E20: with its lower 20
// bits set, over what is in those of e20.
__device__ __forceinline__ uint32_t fixed_point(double w, uint32_t E20, uint32_t e20, uint32_t &lo, uint32_t &hi) {
    const int h = __double2hiint(w);
    const uint32_t s = min((E20 - e20 - ((uint32_t)h & 0x7ff00000u)) >> 20, 63u);
    const unsigned long long v =
        ((((unsigned long long)(uint32_t)((h & 0xfffff) | 0x100000) << 32) | (uint32_t)__double2loint(w)) << 10) >> s;
    const uint32_t sg = (uint32_t)(h >> 31);
    lo = (uint32_t)v ^ sg;
    hi = (uint32_t)(v >> 32) ^ sg ^ 0x80000000u;
    return s;
}

// the eight digits of two entries of consecutive k (a's column with e20 = e.x and
// state e.y, b's with e.z and e.w), packed for an A fragment (lower k in the
// low half): o[i][reg], top digit first, as FP16 subnormals.  own: the states
// of the columns whose term is near enough to the row's scale for them (MORE: bits
// beyond NEAR_W and FAR_W).  E20 as in fixed_point.
template <int MORE>
__device__ __forceinline__ void digit_pair(double a, double b, uint32_t E20, const uint4 &e, uint32_t (&o)[NA][4], int reg,
                                           uint32_t &own) {
    uint32_t al, ah, bl, bh;
    const uint32_t sa = fixed_point(a, E20, e.x, al, ah), sb = fixed_point(b, E20, e.z, bl, bh);
    if (sa <= NEAR_W + MORE) own |= e.y;
    if (sa <= FAR_W + MORE) own |= e.x;
    if (sb <= NEAR_W + MORE) own |= e.w;
    if (sb <= FAR_W + MORE) own |= e.z;
    const uint32_t t = __byte_perm(ah, bh, 0x7632);  // a6 a7 b6 b7
    const uint32_t u = __byte_perm(ah, bh, 0x5410);  // a4 a5 b4 b5
    const uint32_t p = __byte_perm(al, bl, 0x7632);  // a2 a3 b2 b3
    const uint32_t q = __byte_perm(al, bl, 0x5410);  // a0 a1 b0 b1
    const uint32_t top = __byte_perm(t, 0, 0x4341);
    const __half2 c = __hsub2(*reinterpret_cast<const __half2 *>(&top), __half2half2(__ushort_as_half(0x80)));
    o[0][reg] = *reinterpret_cast<const uint32_t *>(&c);
    o[1][reg] = t & 0x00ff00ffu;
    o[2][reg] = __byte_perm(u, 0, 0x4341);
    o[3][reg] = u & 0x00ff00ffu;
    o[4][reg] = __byte_perm(p, 0, 0x4341);
    o[5][reg] = p & 0x00ff00ffu;
    o[6][reg] = __byte_perm(q, 0, 0x4341);
    o[7][reg] = q & 0x00ff00ffu;
}

// acc[i + j] += A_i X_j over 16 rows of staged digits (row k at xs + k
// XSTRIDE) for i + j < NO, and acc[NO - 1] += A_i X_j 2^(8 (NO - 1 - i - j)) for
// the orders NO and NO + 1
template <int NT>
__device__ __forceinline__ void mma_orders(float (&acc)[NO][NT][4], const uint32_t (&a)[NA][4], const unsigned char *xs) {
    const int lane = threadIdx.x & 31;
    const uint32_t base = saddr(xs) + (lane & 15) * XSTRIDE + (NT == 2 ? (lane >> 4) * 16 : 0);
#pragma unroll
    for (int j = 0; j < NA; ++j) {
        uint32_t b[4];
        if constexpr (NT == 2)
            asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                         : "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3])
                         : "r"(base + j * 2 * MR));
        else
            asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n"
                         : "=r"(b[0]), "=r"(b[1])
                         : "r"(base + j * 2 * MR));
#pragma unroll
        for (int i = 0; i + j < NO; ++i)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) mma_f16(acc[i + j][nt], a[i], b[2 * nt], b[2 * nt + 1]);
        // orders NO (up to j = NO) and NO + 1 on the scale of the last sum
#pragma unroll
        for (int m = 0; m < 2; ++m) {
#pragma unroll
            for (int k = 0; k < 2 * NT; ++k) {
                const __half2 v = __hmul2(*reinterpret_cast<const __half2 *>(&b[k]), __float2half2_rn(0x1p-8f));
                b[k] = *reinterpret_cast<const uint32_t *>(&v);
            }
            if (j <= NO + m)
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) mma_f16(acc[NO - 1][nt], a[max(NO + m - j, 0)], b[2 * nt], b[2 * nt + 1]);
        }
    }
}

__device__ __forceinline__ int exp_of(uint32_t E20) { return (int)(E20 >> 20) - E_BIAS; }
// 2^(E - 1011), subnormal too
__device__ __forceinline__ float row_factor(uint32_t E20) {
    const int e = exp_of(E20) - F_EXP;
    return e > 0 ? __uint_as_float((uint32_t)min(e, 255) << 23) : e > -23 ? __uint_as_float(1u << (e + 22)) : 0.0f;
}

// (h, l) += x with the rounding of h kept in l
__device__ __forceinline__ void add_exact(float &h, float &l, float x) {
    const float t = __fadd_rn(h, x);
    const float bp = __fsub_rn(t, h);
    l = __fadd_rn(l, __fadd_rn(__fsub_rn(h, __fsub_rn(t, bp)), __fsub_rn(x, bp)));
    h = t;
}

// the running sums += 2^(E - 1011) sum_d acc_d 2^-8d for the rows g (E20 = e0) and g + 8
// (e1) of a fragment; acc_d to zero.  The orders 0 to 4 are added without
// loss (24 bits each, their rounding kept) and the pair is normalised, so that
// a right-hand side whose sums begin in a lower order keeps its 48 bits.
// add(nt, e, h, l): the running pair of sum (nt, e) += (h, l).
template <int NT, class Add>
__device__ __forceinline__ void flush(float (&acc)[NO][NT][4], uint32_t e0, uint32_t e1, const Add &add) {
    const float f0 = row_factor(e0), f1 = row_factor(e1);
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float f = e < 2 ? f0 : f1;
            float h = acc[0][nt][e];
            float l = __fmul_rn(acc[5][nt][e], 0x1p-40f);
            add_exact(h, l, __fmul_rn(acc[1][nt][e], 0x1p-8f));
            add_exact(h, l, __fmul_rn(acc[2][nt][e], 0x1p-16f));
            add_exact(h, l, __fmul_rn(acc[3][nt][e], 0x1p-24f));
            add_exact(h, l, __fmul_rn(acc[4][nt][e], 0x1p-32f));
            norm2(h, l, h, l);
            add(nt, e, __fmul_rn(h, f), __fmul_rn(l, f));
#pragma unroll
            for (int d = 0; d < NO; ++d) acc[d][nt][e] = 0.0f;
        }
}

// bits of the right-hand sides whose sum in a row or column of exponent E20 is not
// sure to be good to 2^-46.5 of its own terms: all of them are small beside others'.
// all: the states of the columns together.  A row that is zero or not finite has none.
__device__ __forceinline__ uint32_t unsure(uint32_t E20, uint32_t all, uint32_t own) {
    return E20 == E20_START || exp_of(E20) >= E_NAN ? 0u : all >> 16 & ~own;
}

// E = the new scale; own is kept while the raises (of this row in the bits from sh
// on of raised) come to RAISED at most
__device__ __forceinline__ void raise_own(uint32_t &E, uint32_t to, uint32_t &own, uint32_t &raised, int sh) {
    uint32_t sum = (raised >> sh & 0xffffu) + ((to - E) >> 20);
    if (sum > RAISED) own = sum = 0;
    raised = (raised & ~(0xffffu << sh)) | sum << sh;
    E = to;
}

// the cluster goes to the list of those to be formed again, once
__device__ __forceinline__ void note_cluster(int32_t *todo, int64_t nl, int64_t cluster) {
    if (atomicExch(todo + 1 + nl + cluster, 1) == 0) todo[1 + atomicAdd(todo, 1)] = (int32_t)cluster;
}

// largest of the four lanes of a quad (one fragment row)
__device__ __forceinline__ uint32_t quad_max(uint32_t v) {
    v = max(v, __shfl_xor_sync(0xffffffffu, v, 1));
    return max(v, __shfl_xor_sync(0xffffffffu, v, 2));
}

__device__ __forceinline__ uint32_t quad_or(uint32_t v) {
    v |= __shfl_xor_sync(0xffffffffu, v, 1);
    return v | __shfl_xor_sync(0xffffffffu, v, 2);
}

// ---------------------------------------------------------------------------
// column pass: P[wp_colptr[kappa] + v][r] = sum_j W_kappa[j][v] x_r[c0 + j]
//
// One warp per 16 panel columns (the rows of its fragments), 32 panel rows at
// a time; x_kappa's digits in shared memory.  A lane holds two columns and the
// panel rows 2t, 2t + 1, 2t + 8, 2t + 9 of a 16-row step, read from HBM by
// 16-byte loads (128 contiguous bytes per panel row, eight in flight per lane).
// ---------------------------------------------------------------------------
constexpr int CW = 4;                    // warps per CTA
constexpr int KC = 32;                   // panel rows (columns in the row pass) per chunk
constexpr int FLUSH = 4;                 // chunks summed at most: 4 * 255 * 128 * (4 KC) < 2^24

template <int NT>
__global__ void __launch_bounds__(32 * CW, 4) col_fx_kernel(int parts, const int32_t *__restrict__ leaf_begin,
                                                         const int64_t *__restrict__ wp_off,
                                                         const int32_t *__restrict__ wp_K,
                                                         const int64_t *__restrict__ wp_colptr,
                                                         const double *__restrict__ wp, const __half *__restrict__ Xd,
                                                         const uint2 *__restrict__ Xe, float2 *__restrict__ P,
                                                         const int32_t *__restrict__ order, int64_t nl,
                                                         int32_t *__restrict__ todo) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int q = blockIdx.x / parts, part = blockIdx.x - q * parts;
    const int64_t kap = order ? order[q] : q;
    const int Kw = wp_K[kap];
    if (part * 16 * CW >= Kw) return;
    const int32_t c0 = leaf_begin[kap], mc = leaf_begin[kap + 1] - c0;
    const int mp = (mc + KC - 1) / KC * KC;
    uint2 *se = reinterpret_cast<uint2 *>(smem);      // [mp]
    unsigned char *xs = smem + 8 * mp;              // [mp][XSTRIDE]
    // the running sums, touched once in 128 rows, which would not fit the registers: [4 NT][threads]
    float2 *ss = reinterpret_cast<float2 *>(xs + mp * XSTRIDE) + threadIdx.x;
    for (int e = threadIdx.x; e < mp * 2; e += 32 * CW) {
        const int j = e >> 1, p = NA * (e & 1);
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            uint4 v = make_uint4(0, 0, 0, 0);
            if (j < mc) v = __ldg(reinterpret_cast<const uint4 *>(Xd + (int64_t)(c0 + j) * DIG) + p + i);
            *reinterpret_cast<uint4 *>(xs + j * XSTRIDE + 16 * (p + i)) = v;
        }
    }
    for (int j = threadIdx.x; j < mp; j += 32 * CW) se[j] = j < mc ? __ldg(Xe + c0 + j) : make_uint2(0, 0);
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    unsigned int bad = 0, all = 0;
    for (int j = lane; j < mp; j += 32) {
        const unsigned int y = se[j].y;
        all |= y;
        bad |= y & ~(y >> 16);
    }
    bad = __reduce_or_sync(0xffffffffu, bad);  // in the lower half
    all = __reduce_or_sync(0xffffffffu, all);
    const double *W = wp + wp_off[kap];
    for (int v0 = 16 * (part * CW + warp); v0 < Kw; v0 += 16 * CW * parts) {
        const int v = v0 + 2 * g;
        const bool ok = v < Kw;  // Kw is even
        const double *col = W + (ok ? v : 0) + (int64_t)(2 * t) * Kw;
        float acc[NO][NT][4];
        auto add = [&](int nt, int e, float h, float l) {
            float2 &v = ss[(4 * nt + e) * 32 * CW];
            dadd(v.x, v.y, h, l);
        };
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                ss[(4 * nt + e) * 32 * CW] = make_float2(0.0f, 0.0f);
#pragma unroll
                for (int d = 0; d < NO; ++d) acc[d][nt][e] = 0.0f;
            }
        uint32_t E0 = E20_START, E1 = E20_START, own0 = 0, own1 = 0;
        int held = 0;
#pragma unroll 1
        for (int k0 = 0; k0 < mc; k0 += KC, col += (int64_t)KC * Kw) {
            double2 w[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int j = 8 * (i >> 1) + (i & 1);  // panel row k0 + 2t + j
                w[i] = make_double2(0.0, 0.0);
                if (ok && k0 + 2 * t + j < mc) w[i] = __ldg(reinterpret_cast<const double2 *>(col + (int64_t)j * Kw));
            }
            uint32_t m0 = 0, m1 = 0;
#pragma unroll
            for (int i = 0; i < 8; i += 2) {
                const uint4 e = *reinterpret_cast<const uint4 *>(se + k0 + 2 * t + 4 * i);
                m0 = max(m0, max(term_exp(w[i].x, e.x), term_exp(w[i + 1].x, e.z)));
                m1 = max(m1, max(term_exp(w[i].y, e.x), term_exp(w[i + 1].y, e.z)));
            }
            const uint32_t n0 = raise_exp(quad_max(m0), E0), n1 = raise_exp(quad_max(m1), E1);
            if (__any_sync(0xffffffffu, n0 != E0 || n1 != E1) || held == FLUSH) {
                if (held) flush<NT>(acc, E0, E1, add);
                held = 0;
                if (n0 != E0) own0 = 0;
                if (n1 != E1) own1 = 0;
                E0 = n0;
                E1 = n1;
            }
            ++held;
#pragma unroll
            for (int kk = 0; kk < KC; kk += 16) {
                if (k0 + kk >= mc) break;
                uint32_t a[NA][4];
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    const uint4 e = *reinterpret_cast<const uint4 *>(se + k0 + kk + 8 * hf + 2 * t);
                    const double2 x = w[kk / 4 + 2 * hf], y = w[kk / 4 + 2 * hf + 1];
                    digit_pair<RAISED>(x.x, y.x, E0 | 0xfffffu, e, a, 2 * hf, own0);
                    digit_pair<RAISED>(x.y, y.y, E1 | 0xfffffu, e, a, 2 * hf + 1, own1);
                }
                mma_orders<NT>(acc, a, xs + (k0 + kk) * XSTRIDE);
            }
        }
        flush<NT>(acc, E0, E1, add);
        const int worst = (exp_of(E0) >= E_NAN ? 1 : 0) | (exp_of(E1) >= E_NAN ? 2 : 0);
        if (__any_sync(0xffffffffu, (unsure(E0, all, quad_or(own0)) | unsure(E1, all, quad_or(own1))) != 0) && lane == 0)
            note_cluster(todo, nl, kap);
        if (!ok) continue;
        const float nan = __uint_as_float(0x7fffffffu);
#pragma unroll
        for (int h = 0; h < 2; ++h) {  // columns v, v + 1
            float4 *o = reinterpret_cast<float4 *>(P + (wp_colptr[kap] + v + h) * MR);
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                const int r = 8 * nt + 2 * t;
                const float2 s0 = ss[(4 * nt + 2 * h) * 32 * CW], s1 = ss[(4 * nt + 2 * h + 1) * 32 * CW];
                float4 w = make_float4(s0.x, s0.y, s1.x, s1.y);
                if ((worst >> h & 1) || (bad >> r & 1)) w.x = nan;
                if ((worst >> h & 1) || (bad >> (r + 1) & 1)) w.z = nan;
                o[r / 2] = w;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// t_b(l) = sum over the column clusters of sigma_b of the partials, in
// increasing cluster order, as digits: one lane per entry of t (all right-hand
// sides), 32 consecutive entries per warp; the entry's block is found from
// b0[c] (the block holding entry 32 c) by a search over the next 32 blocks'
// offsets, or over t_off beyond them.
// ---------------------------------------------------------------------------
// x 2^k to the nearest integer, by integer operations, for finite x with |x| 2^k < 2^62
__device__ __forceinline__ long long scaled_int(float x, int k) {
    const uint32_t b = __float_as_uint(x);
    const int eb = max((int)(b >> 23) & 0xff, 1);
    const long long m = (long long)((b & 0x7fffffu) | (b & 0x7f800000u ? 0x800000u : 0u));  // |x| = m 2^(eb - 150)
    const int sh = eb - 150 + k;
    const int dn = min(-sh, 32);
    const long long v = sh >= 0 ? m << sh : (m + (1ll << (dn - 1))) >> dn;
    return (int)b < 0 ? -v : v;
}

// the block of entry e = 32 ch + lane of t (whole warps; any block where e is past the end)
__device__ __forceinline__ int64_t block_of(int64_t ch, int64_t e, int64_t na, const int32_t *__restrict__ b0tab,
                                            const int64_t *__restrict__ t_off) {
    const unsigned full = 0xffffffffu;
    const int64_t b0 = b0tab[ch];
    const int64_t to = t_off[min(b0 + (threadIdx.x & 31), na)];  // t_off has na + 1 entries
    int j = 0;
#pragma unroll
    for (int st = 16; st > 0; st >>= 1) {
        const int64_t tj = __shfl_sync(full, to, j + st);
        if (tj <= e) j += st;
    }
    const int64_t to31 = __shfl_sync(full, to, 31);
    if (to31 > e || b0 + 31 >= na) return b0 + j;
    int64_t lo = b0 + 31, hi = na;
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (t_off[mid] <= e) lo = mid;
        else hi = mid;
    }
    return lo;
}

// entry l of t_b for 8 NT right-hand sides, as normalised pairs
template <int NT>
__device__ __forceinline__ void sum_partials(int64_t b, int64_t l, const int64_t *__restrict__ bcolptr,
                                             const int64_t *__restrict__ pofs, const float2 *__restrict__ P,
                                             float (&s)[8 * NT], float (&c)[8 * NT]) {
#pragma unroll
    for (int r = 0; r < 8 * NT; ++r) s[r] = c[r] = 0.0f;
    for (int64_t q = bcolptr[b]; q < bcolptr[b + 1]; ++q) {
        const float4 *pp = reinterpret_cast<const float4 *>(P + (pofs[q] + l) * MR);
#pragma unroll
        for (int k = 0; k < 4 * NT; ++k) {
            const float4 v = __ldg(pp + k);
            dadd(s[2 * k], c[2 * k], v.x, v.y);
            dadd(s[2 * k + 1], c[2 * k + 1], v.z, v.w);
        }
    }
#pragma unroll
    for (int r = 0; r < 8 * NT; ++r) norm2(s[r], c[r], s[r], c[r]);
}

template <int NT>
__global__ void __launch_bounds__(256) tsum_fx_kernel(int64_t na, int64_t nt, const int32_t *__restrict__ b0tab,
                                                      const int64_t *__restrict__ t_off,
                                                      const int64_t *__restrict__ bcolptr,
                                                      const int64_t *__restrict__ pofs, const float2 *__restrict__ P,
                                                      __half *__restrict__ Td, uint2 *__restrict__ Te) {
    constexpr int NR = 8 * NT;
    const int64_t w0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t nchunk = (nt + 31) / 32;
    for (int64_t ch = w0; ch < nchunk; ch += nw) {
        const int64_t e = ch * 32 + (threadIdx.x & 31);
        const int64_t b = block_of(ch, e, na, b0tab, t_off);
        if (e >= nt) continue;
        const int64_t l = e - t_off[b];
        float s[NR], c[NR];
        sum_partials<NT>(b, l, bcolptr, pofs, P, s, c);
        // the exponent of the largest, and the states (as of x: digits_x_kernel)
        int ex = E_ZERO;
        unsigned int bad = 0;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const uint32_t hb = __float_as_uint(s[r]) & 0x7fffffffu;
            if (hb >= 0x7f800000u) bad |= 1u << r;
            else if (hb) ex = max(ex, max((int)(hb >> 23), 1) - 126);  // |s| < 2^ex, subnormal s too
        }
        unsigned int state = bad, far = bad;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const uint32_t hb = __float_as_uint(s[r]) & 0x7fffffffu;
            if (hb == 0u || hb >= 0x7f800000u) continue;
            const int below = ex - (max((int)(hb >> 23), 1) - 126);
            state |= (below <= NEAR_X ? 0x10001u : 0x10000u) << r;
            far |= (below <= FAR_X ? 1u : 0u) << r;
        }
        Te[e] = make_uint2((uint32_t)(ex + E_BIAS) << 20 | far, state);
        unsigned long long u[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            long long q = 0;
            if (ex > E_ZERO && !(bad >> r & 1)) q = scaled_int(s[r], QB - ex) + scaled_int(c[r], QB - ex);
            u[r] = (unsigned long long)q + DIGIT_BIAS;
        }
        uint4 *o = reinterpret_cast<uint4 *>(Td + e * DIG);
#pragma unroll
        for (int j2 = 0; j2 < NA; ++j2)
#pragma unroll
            for (int k = 0; k < NT; ++k) {
                uint32_t w[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int sh = 8 * (NA - 1 - j2), r = 8 * k + 2 * i;
                    // 1024 + u as a half, minus 1152
                    const uint32_t d = 0x64006400u | (uint32_t)((u[r] >> sh) & 0xffu) | (uint32_t)((u[r + 1] >> sh) & 0xffu) << 16;
                    const __half2 hd = __hsub2(*reinterpret_cast<const __half2 *>(&d), __float2half2_rn(1152.0f));
                    w[i] = *reinterpret_cast<const uint32_t *>(&hd);
                }
                o[2 * j2 + k] = make_uint4(w[0], w[1], w[2], w[3]);
            }
    }
}

// ---------------------------------------------------------------------------
// row pass: Y[r0 + i][r] = sum_k D[i][k] x_r[colidx k] + sum_k U[i][k] t_r[tidx k]
//
// One CTA per 16 MT rows of a leaf row cluster, one warp per 16 rows.  The
// panels are walked in chunks of 32 columns through two shared-memory buffers
// filled by cp.async: the FP64 rows of the chunk, and the digits and exponents
// of the gathered rows of x or t.  A warp takes the largest term of each of its
// rows in the chunk, forms the digits of its entries (each entry by one lane)
// and multiplies.  Per 16 x 16 entries: 72 products of 16 x 8 x 16 (~160 cycles of an
// SM), ~28 integer operations per entry (~100 cycles of the ALU pipe), 2 KB from
// HBM (~95 cycles).
// ---------------------------------------------------------------------------
constexpr int AST = KC * 8;               // bytes per staged panel row; odd rows have their 64-byte halves swapped (banks)
template <int MT> struct RowCfg {
    static constexpr int THREADS = 32 * MT;
    static constexpr int A_BYTES = 16 * MT * AST;
    static constexpr int STAGE = A_BYTES + KC * XSTRIDE + KC * 8;
    static constexpr int SMEM = 2 * STAGE + 2 * KC * 4;
    static constexpr int CTAS = MT <= 2 ? 6 : MT == 3 ? 5 : MT == 4 ? 4 : 3;  // per SM: 128 registers, shared memory
};

template <int MT, int NT>
__global__ void __launch_bounds__(32 * MT, RowCfg<MT>::CTAS) row_fx_kernel(
    int parts, const int32_t *__restrict__ leaf_begin, const int64_t *__restrict__ rho_off,
    const int32_t *__restrict__ rho_K, const int64_t *__restrict__ rho_colptr, const int32_t *__restrict__ colidx,
    const double *__restrict__ dense, const int64_t *__restrict__ up_off, const int32_t *__restrict__ up_K,
    const int64_t *__restrict__ up_colptr, const int32_t *__restrict__ tidx, const double *__restrict__ up,
    const __half *__restrict__ Xd, const uint2 *__restrict__ Xe, const __half *__restrict__ Td,
    const uint2 *__restrict__ Te, const Scale *__restrict__ sc, double *__restrict__ Y,
    const int4 *__restrict__ items, float2 *__restrict__ Ypart, uint2 *__restrict__ part_state, int prow,
    int64_t nl, int32_t *__restrict__ todo) {
    using C = RowCfg<MT>;
    extern __shared__ __align__(16) unsigned char smem[];
    int32_t *s_idx = reinterpret_cast<int32_t *>(smem + 2 * C::STAGE);  // [2][KC]
    const int q = blockIdx.x / parts, part = blockIdx.x - q * parts;
    const int4 it = items[q];  // cluster, chunks [y, z), partial slot or -1
    const int rho = it.x, cend = it.z;
    const int32_t r0 = leaf_begin[rho] + part * 16 * MT;
    const int rows = min(16 * MT, leaf_begin[rho + 1] - r0);
    if (rows <= 0) return;
    const int Kd = rho_K[rho], Ku = up_K[rho];
    const int nd = (Kd + KC - 1) / KC;
    const double *Pd = dense + rho_off[rho] + (int64_t)part * 16 * MT * Kd;
    const double *Pu = up + up_off[rho] + (int64_t)part * 16 * MT * Ku;
    const int32_t *ci = colidx + rho_colptr[rho], *ti = tidx + up_colptr[rho];
    const int tid = threadIdx.x;
    // gather indices of chunk c (-1: past the panel)
    auto load_idx = [&](int c) {
        for (int k = tid; k < KC; k += C::THREADS) {
            const bool u = c >= nd;
            const int K = u ? Ku : Kd, col = (u ? c - nd : c) * KC + k;
            s_idx[(c & 1) * KC + k] = c < cend && col < K ? __ldg((u ? ti : ci) + col) : -1;
        }
    };
    // this thread's pieces of a chunk: 16 bytes of the panel rows arow, arow +
    // THREADS / 16, ... and pieces of the digits of a column
    const int arow = tid >> 4, acol = 2 * (tid & 15);
    auto issue = [&](int c) {
        unsigned char *st = smem + (c & 1) * C::STAGE;
        const bool u = c >= nd;
        const int K = u ? Ku : Kd, k0 = (u ? c - nd : c) * KC;
        const double *P = u ? Pu : Pd;
        const bool in = k0 + acol < K;
        const double *src = P + (int64_t)arow * K + k0 + acol;
        unsigned char *dst = st + arow * AST + ((acol * 8) ^ ((arow & 1) << 6));  // the rows below have the same parity
#pragma unroll
        for (int v = 0; v < 8; ++v, src += (C::THREADS / 16) * (int64_t)K) {
            const bool ok = in && arow + (C::THREADS / 16) * v < rows;
            cp_async<16>(dst + (C::THREADS / 16) * v * AST, ok ? src : P, ok);
        }
        const __half *Z = u ? Td : Xd;
        const uint2 *Ze = u ? Te : Xe;
        unsigned char *sb = st + C::A_BYTES;
        const int32_t *ix = s_idx + (c & 1) * KC;
        // two neighbouring threads take 16 bytes each of a column in turn
#pragma unroll
        for (int e0 = 0; e0 < KC * 2; e0 += C::THREADS) {
            const int e = e0 + tid, k = e >> 1, p = e & 1;
            if (e0 + C::THREADS <= KC * 2 || e < KC * 2) {
                const int z = ix[k];
                const __half *zs = Z + (int64_t)max(z, 0) * DIG + 8 * p;
                unsigned char *zd = sb + k * XSTRIDE + 16 * p;
#pragma unroll
                for (int i = 0; i < NA; ++i) cp_async<16>(zd + 32 * i, zs + 16 * i, z >= 0);
                if (p == 0) cp_async<8>(sb + KC * XSTRIDE + 8 * k, Ze + max(z, 0), z >= 0);
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    const int lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    float acc[NO][NT][4], s[NT][4], c[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            s[nt][e] = c[nt][e] = 0.0f;
#pragma unroll
            for (int d = 0; d < NO; ++d) acc[d][nt][e] = 0.0f;
        }
    auto add = [&](int nt, int e, float h, float l) { dadd(s[nt][e], c[nt][e], h, l); };
    unsigned int bad = 0, all = 0;
    uint32_t E0 = E20_START, E1 = E20_START, own0 = 0, own1 = 0, raised = 0;
    int held = 0;
    load_idx(it.y);
    load_idx(it.y + 1);
    __syncthreads();
    if (it.y < cend) issue(it.y);
#pragma unroll 1
    for (int ch = it.y; ch < cend; ++ch) {
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        __syncthreads();  // chunk ch has landed for every thread; every thread is done with chunk ch - 1
        if (ch + 1 < cend) issue(ch + 1);
        const unsigned char *st = smem + (ch & 1) * C::STAGE;
        // columns 8 i + 2 t, + 1 of a row: the i-th 64 bytes, i's lowest bit flipped in odd rows
        const double *a0 = reinterpret_cast<const double *>(st + (16 * warp + g) * AST) + 2 * t;
        const double *a1 = a0 + 8 * KC;
        const int flip = 8 * (g & 1);
        const unsigned char *sb = st + C::A_BYTES;
        const uint2 *se = reinterpret_cast<const uint2 *>(sb + KC * XSTRIDE) + 2 * t;
        uint32_t m0 = 0, m1 = 0;
#pragma unroll
        for (int k = 0; k < KC; k += 8) {
            const double2 w0 = *reinterpret_cast<const double2 *>(a0 + (k ^ flip));
            const double2 w1 = *reinterpret_cast<const double2 *>(a1 + (k ^ flip));
            const uint4 e = *reinterpret_cast<const uint4 *>(se + k);
            all |= e.y | e.w;
            bad |= (e.y & ~(e.y >> 16)) | (e.w & ~(e.w >> 16));
            m0 = max(m0, max(term_exp(w0.x, e.x), term_exp(w0.y, e.z)));
            m1 = max(m1, max(term_exp(w1.x, e.x), term_exp(w1.y, e.z)));
        }
        const uint32_t n0 = raise_exp(quad_max(m0), E0), n1 = raise_exp(quad_max(m1), E1);
        if (__any_sync(0xffffffffu, n0 != E0 || n1 != E1) || held == FLUSH) {
            if (held) flush<NT>(acc, E0, E1, add);
            held = 0;
            raise_own(E0, n0, own0, raised, 0);
            raise_own(E1, n1, own1, raised, 16);
        }
        ++held;
#pragma unroll
        for (int k = 0; k < KC; k += 16) {
            uint32_t a[NA][4];
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                const double2 w0 = *reinterpret_cast<const double2 *>(a0 + ((k + 8 * hf) ^ flip));
                const double2 w1 = *reinterpret_cast<const double2 *>(a1 + ((k + 8 * hf) ^ flip));
                const uint4 e = *reinterpret_cast<const uint4 *>(se + k + 8 * hf);
                digit_pair<0>(w0.x, w0.y, E0 | 0xfffffu, e, a, 2 * hf, own0);
                digit_pair<0>(w1.x, w1.y, E1 | 0xfffffu, e, a, 2 * hf + 1, own1);
            }
            mma_orders<NT>(acc, a, sb + k * XSTRIDE);
        }
        // the indices of chunk ch + 2 (chunk ch's were read by issue(ch), an iteration ago)
        load_idx(ch + 2);
    }
    flush<NT>(acc, E0, E1, add);
    const int worst = (exp_of(E0) >= E_NAN ? 1 : 0) | (exp_of(E1) >= E_NAN ? 2 : 0);
    bad = __reduce_or_sync(0xffffffffu, bad);  // in the lower half
    all = __reduce_or_sync(0xffffffffu, all);
    own0 = quad_or(own0);
    own1 = quad_or(own1);
    if (it.w >= 0) {  // a part of the row: row_reduce_kernel looks at all of them
        if (t == 0) {
            uint2 *o = part_state + (int64_t)it.w * prow + part * 16 * MT + 16 * warp + g;
            if (16 * warp + g < rows) o[0] = make_uint2(E0 | (raised & 0xffffu), (all & 0xffff0000u) | (own0 & 0xffffu));
            if (16 * warp + g + 8 < rows) o[8] = make_uint2(E1 | raised >> 16, (all & 0xffff0000u) | (own1 & 0xffffu));
        }
    } else if (__any_sync(0xffffffffu, (unsure(E0, all, own0) | unsure(E1, all, own1)) != 0) && lane == 0) {
        note_cluster(todo, nl, rho);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int row = 16 * warp + g + 8 * h;
        if (row >= rows) continue;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int r = 8 * nt + 2 * t + e;
                float hi = s[nt][2 * h + e];
                if ((worst >> h & 1) || (bad >> r & 1)) hi = __uint_as_float(0x7fffffffu);  // NaN
                if (it.w >= 0)
                    Ypart[((int64_t)it.w * prow + part * 16 * MT + row) * MR + r] = make_float2(hi, c[nt][2 * h + e]);
                else
                    Y[(int64_t)(r0 + row) * MR + r] =
                        scalbn((double)hi + (double)c[nt][2 * h + e], scale_of(sc[r]));
            }
    }
}

// rows of the clusters whose panels were split: Y = the sum of the partials
// in slot order (red: cluster, first slot, slots).  A part's own terms speak for the
// row where its scale is within RAISED of the row's, raises included.
template <int NT>
__global__ void __launch_bounds__(256) row_reduce_kernel(const int4 *__restrict__ red, const int32_t *__restrict__ leaf_begin,
                                                         const float2 *__restrict__ Ypart, int prow,
                                                         const uint2 *__restrict__ part_state,
                                                         const Scale *__restrict__ sc, double *__restrict__ Y,
                                                         int64_t nl, int32_t *__restrict__ todo) {
    const int4 rd = red[blockIdx.x];
    const int32_t r0 = leaf_begin[rd.x], mr = leaf_begin[rd.x + 1] - r0;
    for (int e = threadIdx.x; e < mr * 8 * NT; e += 256) {
        const int row = e / (8 * NT), r = e - row * (8 * NT);
        float s = 0.0f, c = 0.0f;
#pragma unroll 4
        for (int k = 0; k < rd.z; ++k) {
            const float2 v = Ypart[((int64_t)(rd.y + k) * prow + row) * MR + r];
            dadd(s, c, v.x, v.y);
        }
        Y[(int64_t)(r0 + row) * MR + r] = scalbn((double)s + (double)c, scale_of(sc[r]));
    }
    for (int row = threadIdx.x; row < mr; row += 256) {
        const uint2 *p = part_state + (int64_t)rd.y * prow + row;
        uint32_t E = E20_START, all = 0, own = 0;
        for (int k = 0; k < rd.z; ++k) E = max(E, p[(int64_t)k * prow].x & 0xfff00000u);
        for (int k = 0; k < rd.z; ++k) {
            const uint2 v = p[(int64_t)k * prow];
            all |= v.y;
            if ((E >> 20) - (v.x >> 20) + (v.x & 0xffffu) <= RAISED) own |= v.y;
        }
        if (unsure(E, all, own)) note_cluster(todo, nl, rd.x);
    }
}

// ---------------------------------------------------------------------------
// The clusters where right-hand sides of unlike sizes meet (unsure), formed again
// with pairs of floats: every entry and x_r is split by itself, w = h + l to
// 2^-47 |w|, and each term is added with an error-free product and sum (the
// compensated dot product of Ogita, Rump and Oishi, "Accurate sum and dot product",
// SIAM J. Sci. Comput. 2005, Algorithm 5.3), so no right-hand side sees another.
// Few or no clusters as a rule (none of random or smooth vectors of like size): the
// lists (todo: length, clusters, marks) are walked by a fixed number of CTAs, which
// end at once where they are empty (3 us a kernel).  Bound
// by the FP32 pipe where all clusters are listed, by latency where few are.
// ---------------------------------------------------------------------------
constexpr int PAIR_CTAS = 8;  // per SM

// h: w truncated to 24 bits, l: the rest, from the bits of w where both are normal
// floats; (0, 0) below the floats, NaN above them
__device__ __forceinline__ void split(double w, float &h, float &l) {
    const uint32_t hi32 = (uint32_t)__double2hiint(w), lo32 = (uint32_t)__double2loint(w);
    const uint32_t mag = hi32 & 0x7fffffffu, sgn = hi32 & 0x80000000u;
    if (mag >= 0x3b500000u && mag < 0x47f00000u) {  // biased exponent in [949, 1151)
        h = __uint_as_float(sgn | ((mag - 0x38000000u) << 3) | (lo32 >> 29));
        const float sc = __uint_as_float((uint32_t)((int)(mag >> 20) - 948) << 23);  // 2^(exponent - 52)
        l = __uint_as_float(__float_as_uint(__fmul_rn(__uint2float_rn(lo32 & 0x1fffffffu), sc)) | sgn);
    } else if (mag >= 0x47f00000u) {
        h = l = __uint_as_float(0x7fffffffu);
    } else {
        h = __double2float_rz(w);
        l = __double2float_rn(w - (double)h);
    }
}

// (s, c) += (ah + al)(xh + xl)
__device__ __forceinline__ void dfma(float &s, float &c, float ah, float al, float xh, float xl) {
    const float p = __fmul_rn(ah, xh);
    const float e = __fmaf_rn(ah, xh, -p);
    const float t = __fadd_rn(s, p);
    const float bp = __fsub_rn(t, s);
    const float sg = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(p, bp));
    s = t;
    c = __fadd_rn(c, __fmaf_rn(al, xh, __fmaf_rn(ah, xl, __fadd_rn(e, sg))));
}

// (s, c)_r += w z_r for the pairs of z at z[r], z[MR + r]
template <int NT>
__device__ __forceinline__ void pair_step(double w, const float4 *z, float (&s)[8 * NT], float (&c)[8 * NT]) {
    float ah, al;
    split(w, ah, al);
#pragma unroll
    for (int q = 0; q < 2 * NT; ++q) {
        const float4 xh = z[q], xl = z[MR / 4 + q];
        dfma(s[4 * q], c[4 * q], ah, al, xh.x, xl.x);
        dfma(s[4 * q + 1], c[4 * q + 1], ah, al, xh.y, xl.y);
        dfma(s[4 * q + 2], c[4 * q + 2], ah, al, xh.z, xl.z);
        dfma(s[4 * q + 3], c[4 * q + 3], ah, al, xh.w, xl.w);
    }
}

// x_r at position m on its own scale, as a pair
__device__ __forceinline__ void x_pair(const double *__restrict__ x, int64_t n, int nr, const int32_t *__restrict__ perm,
                                       const Scale *__restrict__ sc, int64_t m, int r, float &h, float &l) {
    const double v = r < nr ? scalbn(x[(int64_t)r * n + (perm ? perm[m] : m)], -scale_of(sc[r])) : 0.0;
    h = __double2float_rn(v);
    l = __double2float_rn(v - (double)h);
}

// the partials of the listed column clusters; one thread per panel column
constexpr int CP_THREADS = 128;
template <int NT>
__global__ void __launch_bounds__(CP_THREADS) col_pairs_kernel(
    int parts, const int32_t *__restrict__ todo, const int32_t *__restrict__ leaf_begin,
    const int64_t *__restrict__ wp_off, const int32_t *__restrict__ wp_K, const int64_t *__restrict__ wp_colptr,
    const double *__restrict__ wp, const double *__restrict__ x, int64_t n, int nr, const int32_t *__restrict__ perm,
    const Scale *__restrict__ sc, float2 *__restrict__ P) {
    __shared__ float4 sx[MAX_LEAF * MR / 2];
    float *sf = reinterpret_cast<float *>(sx);
    const int64_t count = (int64_t)todo[0] * parts;
    for (int64_t q = blockIdx.x; q < count; q += gridDim.x) {
        const int64_t kap = todo[1 + q / parts];
        const int Kw = wp_K[kap], v0 = (int)(q % parts) * CP_THREADS;
        if (v0 >= Kw) continue;
        const int32_t c0 = leaf_begin[kap], mc = leaf_begin[kap + 1] - c0;
        __syncthreads();  // the last cluster's x has been read
        for (int e = threadIdx.x; e < mc * MR; e += CP_THREADS) {
            const int j = e / MR, r = e % MR;
            x_pair(x, n, nr, perm, sc, c0 + j, r, sf[2 * MR * j + r], sf[2 * MR * j + MR + r]);
        }
        __syncthreads();
        const int v = v0 + threadIdx.x;
        if (v >= Kw) continue;
        float s[8 * NT], c[8 * NT];
#pragma unroll
        for (int r = 0; r < 8 * NT; ++r) s[r] = c[r] = 0.0f;
        const double *col = wp + wp_off[kap] + v;
#pragma unroll 4
        for (int j = 0; j < mc; ++j) pair_step<NT>(__ldg(col + (int64_t)j * Kw), sx + j * MR / 2, s, c);
        float4 *o = reinterpret_cast<float4 *>(P + (wp_colptr[kap] + v) * MR);
#pragma unroll
        for (int r = 0; r < 8 * NT; r += 2) o[r / 2] = make_float4(s[r], c[r], s[r + 1], c[r + 1]);
    }
}

// where a row cluster is listed: x and t as pairs ([row][hi 16, lo 16]), in the place of their digits.
// Few listed clusters: only the rows that they read, a warp per entry of t with its lanes over the
// partials (a block of the top levels has thousands, and one lane's chain of them is what the whole
// sum takes: 1,310,720 panels 2.7 ms).  Else all rows, as tsum_fx_kernel forms them.
constexpr int FEW = 64;  // listed clusters of one in so many
template <int NT>
__global__ void __launch_bounds__(256) pairs_kernel(
    const int32_t *__restrict__ todo, int64_t nl, int64_t na, int64_t nt, const int32_t *__restrict__ b0tab,
    const int64_t *__restrict__ t_off, const int64_t *__restrict__ bcolptr, const int64_t *__restrict__ pofs,
    const float2 *__restrict__ P, const int32_t *__restrict__ rho_K, const int64_t *__restrict__ rho_colptr,
    const int32_t *__restrict__ colidx, const int32_t *__restrict__ up_K, const int64_t *__restrict__ up_colptr,
    const int32_t *__restrict__ tidx, const double *__restrict__ x, int64_t n, int nr, const int32_t *__restrict__ perm,
    const Scale *__restrict__ sc, float *__restrict__ Xp, float *__restrict__ Tp) {
    const int count = todo[0];
    if (count == 0) return;
    const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nth = (int64_t)gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    auto x_row = [&](int64_t m, int r) { x_pair(x, n, nr, perm, sc, m, r, Xp[m * 2 * MR + r], Xp[m * 2 * MR + MR + r]); };
    if ((int64_t)count * FEW > nl) {
        for (int64_t e = t0; e < n * MR; e += nth) x_row(e / MR, (int)(e % MR));
        for (int64_t ch = t0 >> 5; ch < (nt + 31) / 32; ch += nth >> 5) {
            const int64_t e = ch * 32 + lane;
            const int64_t b = block_of(ch, e, na, b0tab, t_off);
            if (e >= nt) continue;
            float s[8 * NT], c[8 * NT];
            sum_partials<NT>(b, e - t_off[b], bcolptr, pofs, P, s, c);
            float4 *o = reinterpret_cast<float4 *>(Tp + e * 2 * MR);
#pragma unroll
            for (int k = 0; k < 2 * NT; ++k) {
                o[k] = make_float4(s[4 * k], s[4 * k + 1], s[4 * k + 2], s[4 * k + 3]);
                o[MR / 4 + k] = make_float4(c[4 * k], c[4 * k + 1], c[4 * k + 2], c[4 * k + 3]);
            }
        }
        return;
    }
    for (int i = 0; i < count; ++i) {
        const int64_t rho = todo[1 + i];
        const int32_t *ci = colidx + rho_colptr[rho], *ti = tidx + up_colptr[rho];
        for (int64_t e = t0; e < (int64_t)rho_K[rho] * MR; e += nth) x_row(ci[e / MR], (int)(e % MR));
        for (int64_t v = t0 >> 5; v < up_K[rho]; v += nth >> 5) {
            const int64_t e = ti[v];
            // the block of e: from the one that holds entry 32 (e / 32) to the one that holds the next such entry
            int64_t b = b0tab[e / 32], hi = (e / 32 + 1) * 32 < nt ? b0tab[e / 32 + 1] + 1 : na;
            while (hi - b > 1) {
                const int64_t mid = (b + hi) >> 1;
                if (t_off[mid] <= e) b = mid;
                else hi = mid;
            }
            const int64_t l = e - t_off[b];
            float s[8 * NT], c[8 * NT];
#pragma unroll
            for (int r = 0; r < 8 * NT; ++r) s[r] = c[r] = 0.0f;
            for (int64_t q = bcolptr[b] + lane; q < bcolptr[b + 1]; q += 32) {
                const float4 *pp = reinterpret_cast<const float4 *>(P + (pofs[q] + l) * MR);
#pragma unroll
                for (int k = 0; k < 4 * NT; ++k) {
                    const float4 w = __ldg(pp + k);
                    dadd(s[2 * k], c[2 * k], w.x, w.y);
                    dadd(s[2 * k + 1], c[2 * k + 1], w.z, w.w);
                }
            }
#pragma unroll
            for (int r = 0; r < 8 * NT; ++r) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const float s2 = __shfl_xor_sync(0xffffffffu, s[r], o), c2 = __shfl_xor_sync(0xffffffffu, c[r], o);
                    dadd(s[r], c[r], s2, c2);
                }
                if (lane == r) norm2(s[r], c[r], Tp[e * 2 * MR + r], Tp[e * 2 * MR + MR + r]);
            }
        }
    }
}

// the rows of the listed row clusters, sixteen per CTA and two per warp (a column's pairs, read from
// shared memory once, serve both); the gathered pairs of 64 columns at a time in shared memory, the next
// 64 and their entries on the way meanwhile
constexpr int RP_WARPS = 8, RP_ROWS = 2 * RP_WARPS, RP_COLS = 64;
constexpr int RP_STRIDE = MR / 2 + 1;  // float4 per column: eight lanes hit different banks
template <int NT>
__global__ void __launch_bounds__(32 * RP_WARPS, 2) row_pairs_kernel(
    int parts, const int32_t *__restrict__ todo, const int32_t *__restrict__ leaf_begin,
    const int64_t *__restrict__ rho_off, const int32_t *__restrict__ rho_K, const int64_t *__restrict__ rho_colptr,
    const int32_t *__restrict__ colidx, const double *__restrict__ dense, const int64_t *__restrict__ up_off,
    const int32_t *__restrict__ up_K, const int64_t *__restrict__ up_colptr, const int32_t *__restrict__ tidx,
    const double *__restrict__ up, const float4 *__restrict__ Xp, const float4 *__restrict__ Tp,
    const Scale *__restrict__ sc, double *__restrict__ Y) {
    constexpr int PIECES = RP_COLS * MR / 2 / (32 * RP_WARPS);  // float4 of a chunk per thread
    __shared__ float4 sz[RP_COLS * RP_STRIDE];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t count = (int64_t)todo[0] * parts;
    for (int64_t q = blockIdx.x; q < count; q += gridDim.x) {
        const int64_t rho = todo[1 + q / parts];
        const int32_t r0 = leaf_begin[rho], mr = leaf_begin[rho + 1] - r0;
        const int row = (int)(q % parts) * RP_ROWS + 2 * warp;
        if (row - 2 * warp >= mr) continue;
        float s[2][8 * NT], c[2][8 * NT];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int r = 0; r < 8 * NT; ++r) s[i][r] = c[i][r] = 0.0f;
#pragma unroll 1
        for (int u = 0; u < 2; ++u) {  // the near field, then the U panel
            const int K = u ? up_K[rho] : rho_K[rho];
            const int32_t *idx = u ? tidx + up_colptr[rho] : colidx + rho_colptr[rho];
            const double *p0 = (u ? up + up_off[rho] : dense + rho_off[rho]);
            const double *p[2] = {p0 + (int64_t)min(row, mr - 1) * K, p0 + (int64_t)min(row + 1, mr - 1) * K};
            const float4 *z = u ? Tp : Xp;
            float4 zn[PIECES];
            double wn[2][RP_COLS / 32];
            auto fetch = [&](int k0) {
#pragma unroll
                for (int i = 0; i < PIECES; ++i) {
                    const int e = threadIdx.x + 32 * RP_WARPS * i, k = k0 + e / (MR / 2);
                    if (k < K) zn[i] = __ldg(z + (int64_t)idx[k] * (MR / 2) + e % (MR / 2));
                }
#pragma unroll
                for (int h = 0; h < RP_COLS / 32; ++h)
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const int k = k0 + 32 * h + lane;
                        wn[i][h] = k < K ? __ldg(p[i] + k) : 0.0;
                    }
            };
            fetch(0);
#pragma unroll 1
            for (int k0 = 0; k0 < K; k0 += RP_COLS) {
                __syncthreads();  // the last chunk has been read
                double w[2][RP_COLS / 32];
#pragma unroll
                for (int i = 0; i < PIECES; ++i) {
                    const int e = threadIdx.x + 32 * RP_WARPS * i;
                    sz[e / (MR / 2) * RP_STRIDE + e % (MR / 2)] = zn[i];
                }
#pragma unroll
                for (int h = 0; h < RP_COLS / 32; ++h)
#pragma unroll
                    for (int i = 0; i < 2; ++i) w[i][h] = wn[i][h];
                __syncthreads();
                if (k0 + RP_COLS < K) fetch(k0 + RP_COLS);
#pragma unroll
                for (int h = 0; h < RP_COLS / 32; ++h) {
                    if (k0 + 32 * h + lane >= K) continue;
#pragma unroll
                    for (int i = 0; i < 2; ++i) pair_step<NT>(w[i][h], sz + (32 * h + lane) * RP_STRIDE, s[i], c[i]);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int r = 0; r < 8 * NT; ++r) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const float s2 = __shfl_xor_sync(0xffffffffu, s[i][r], o), c2 = __shfl_xor_sync(0xffffffffu, c[i][r], o);
                    dadd(s[i][r], c[i][r], s2, c2);
                }
                if (lane == r && row + i < mr)
                    Y[(int64_t)(r0 + row + i) * MR + r] = scalbn((double)s[i][r] + (double)c[i][r], scale_of(sc[r]));
            }
    }
}

// y_r[m] (Morton, [nr][n]) or y_r[perm[m]] (original order) = alpha Y[m][r] + beta y
__global__ void scatter_kernel(const double *__restrict__ Y, int64_t n, int nr, const int32_t *__restrict__ perm,
                               double alpha, double beta, double *__restrict__ y) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n * nr; e += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(e / n);
        const int64_t m = e - (int64_t)r * n;
        const int64_t o = (int64_t)r * n + (perm ? perm[m] : m);
        const double v = alpha * Y[m * MR + r];
        y[o] = beta == 0.0 ? v : v + beta * y[o];
    }
}

// blocks of 256 threads for a grid-stride loop over n items
static unsigned grid_for(int64_t n) {
    const int64_t b = (n + 255) / 256;
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(b, 65535LL * 8));
}

// the working arrays of one pass, in this order (each a multiple of 16 bytes)
struct Work {
    __half *Xd, *Td;
    float2 *P, *Ypart;
    uint2 *Xe, *Te, *part_state;
    Scale *sc;
    int32_t *todo_c, *todo_r;  // column and row clusters to be formed again: length, clusters [nl], marks [nl]
};
constexpr int SCALE_FLOATS = MR * (int)(sizeof(Scale) / sizeof(float));
static int64_t todo_ints(int64_t nl) { return (1 + 2 * nl + 3) / 4 * 4; }

template <int NT>
static void block_product(const hm_matrix *A, const double *x, int nr, const int32_t *perm, double *Y, const Work &w,
                          cudaStream_t s) {
    const hm_tree *tr = A->tree;
    const int64_t n = tr->n, nl = tr->n_leaf;
    // (the lists follow the scales)
    HM_CUDA_CHECK(cudaMemsetAsync(w.sc, 0, sizeof(Scale) * MR + sizeof(int32_t) * 2 * todo_ints(nl), s));
    const unsigned pair_grid = (unsigned)(PAIR_CTAS * num_sms());
    const dim3 gs((unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 2047) / 2048, 256)), (unsigned)nr);
    scale_x_kernel<<<gs, 256, 0, s>>>(x, n, w.sc);
    HM_LAUNCH_CHECK();
    digits_x_kernel<<<grid_for(n * MR), 256, 0, s>>>(x, n, nr, perm, w.sc, w.Xd, w.Xe);
    HM_LAUNCH_CHECK();
    const int32_t *ord = A->mv_order.as<int32_t>();
    if (tr->n_adm > 0) {
        {
            const int smem = (tr->max_leaf + KC - 1) / KC * KC * (XSTRIDE + 8) + 4 * NT * 32 * CW * (int)sizeof(float2);
            HM_CUDA_CHECK(cudaFuncSetAttribute(col_fx_kernel<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
            const int parts = ((A->wp_kmax + 16 * CW * 4 - 1) / (16 * CW * 4)) | 1;  // odd: see col_kernel
            Trace trace("col_fx_kernel", s);
            col_fx_kernel<NT><<<(unsigned)(nl * parts), 32 * CW, smem, s>>>(
                parts, tr->leaf_begin.as<int32_t>(), A->wp_off.as<int64_t>(), A->wp_K.as<int32_t>(),
                A->wp_colptr.as<int64_t>(), A->wp.as<double>(), w.Xd, w.Xe, w.P, ord ? ord + nl : nullptr, nl,
                w.todo_c);
            HM_LAUNCH_CHECK();
            col_pairs_kernel<NT><<<pair_grid, CP_THREADS, 0, s>>>(
                (A->wp_kmax + CP_THREADS - 1) / CP_THREADS, w.todo_c, tr->leaf_begin.as<int32_t>(),
                A->wp_off.as<int64_t>(), A->wp_K.as<int32_t>(), A->wp_colptr.as<int64_t>(), A->wp.as<double>(), x, n, nr,
                perm, w.sc, w.P);
            HM_LAUNCH_CHECK();
        }
        Trace trace("tsum_fx_kernel", s);
        tsum_fx_kernel<NT><<<grid_for((A->total_rank + 31) / 32 * 32), 256, 0, s>>>(
            tr->n_adm, A->total_rank, A->tsum_b0.as<int32_t>(), A->t_off.as<int64_t>(), tr->lr_bcolptr.as<int64_t>(),
            A->pofs.as<int64_t>(), w.P, w.Td, w.Te);
        HM_LAUNCH_CHECK();
    }
    const int tiles = (tr->max_leaf + 15) / 16, parts = (tiles + 4) / 5, mt = (tiles + parts - 1) / parts;
    const int prow = 16 * tiles;
    auto launch = [&](auto kern, int threads, int smem) {
        HM_CUDA_CHECK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        Trace trace("row_fx_kernel", s);
        kern<<<(unsigned)(A->fx_nitems * parts), threads, smem, s>>>(
            parts, tr->leaf_begin.as<int32_t>(), tr->rho_off.as<int64_t>(), tr->rho_K.as<int32_t>(),
            tr->rho_colptr.as<int64_t>(), tr->colidx.as<int32_t>(), A->dense.as<double>(), A->up_off.as<int64_t>(),
            A->up_K.as<int32_t>(), A->up_colptr.as<int64_t>(), A->tidx.as<int32_t>(), A->up.as<double>(), w.Xd, w.Xe,
            w.Td, w.Te, w.sc, Y, A->fx_items.as<int4>(), w.Ypart,
            w.part_state, prow, nl, w.todo_r);
        HM_LAUNCH_CHECK();
    };
    switch (mt) {
        case 1: launch(row_fx_kernel<1, NT>, RowCfg<1>::THREADS, RowCfg<1>::SMEM); break;
        case 2: launch(row_fx_kernel<2, NT>, RowCfg<2>::THREADS, RowCfg<2>::SMEM); break;
        case 3: launch(row_fx_kernel<3, NT>, RowCfg<3>::THREADS, RowCfg<3>::SMEM); break;
        case 4: launch(row_fx_kernel<4, NT>, RowCfg<4>::THREADS, RowCfg<4>::SMEM); break;
        default: launch(row_fx_kernel<5, NT>, RowCfg<5>::THREADS, RowCfg<5>::SMEM); break;
    }
    if (A->fx_nred > 0) {
        row_reduce_kernel<NT><<<(unsigned)A->fx_nred, 256, 0, s>>>(A->fx_red.as<int4>(), tr->leaf_begin.as<int32_t>(),
                                                                   w.Ypart, prow, w.part_state, w.sc, Y, nl, w.todo_r);
        HM_LAUNCH_CHECK();
    }
    float *Xp = reinterpret_cast<float *>(w.Xd), *Tp = reinterpret_cast<float *>(w.Td);
    static_assert(DIG * sizeof(__half) >= 2 * MR * sizeof(float), "pairs in the place of digits");
    pairs_kernel<NT><<<pair_grid, 256, 0, s>>>(
        w.todo_r, nl, tr->n_adm, tr->n_adm > 0 ? A->total_rank : 0, A->tsum_b0.as<int32_t>(), A->t_off.as<int64_t>(),
        tr->lr_bcolptr.as<int64_t>(), A->pofs.as<int64_t>(), w.P, tr->rho_K.as<int32_t>(), tr->rho_colptr.as<int64_t>(),
        tr->colidx.as<int32_t>(), A->up_K.as<int32_t>(), A->up_colptr.as<int64_t>(), A->tidx.as<int32_t>(), x, n, nr,
        perm, w.sc, Xp, Tp);
    HM_LAUNCH_CHECK();
    row_pairs_kernel<NT><<<pair_grid, 32 * RP_WARPS, 0, s>>>(
        (tr->max_leaf + RP_ROWS - 1) / RP_ROWS, w.todo_r, tr->leaf_begin.as<int32_t>(), tr->rho_off.as<int64_t>(),
        tr->rho_K.as<int32_t>(), tr->rho_colptr.as<int64_t>(), tr->colidx.as<int32_t>(), A->dense.as<double>(),
        A->up_off.as<int64_t>(), A->up_K.as<int32_t>(), A->up_colptr.as<int64_t>(), A->tidx.as<int32_t>(),
        A->up.as<double>(), reinterpret_cast<float4 *>(Xp), reinterpret_cast<float4 *>(Tp), w.sc, Y);
    HM_LAUNCH_CHECK();
}

}  // namespace fx

// The row pass's work items: the panels of a leaf row cluster in chunks of 32
// columns (near field first, then U), cut where one is long.  A cluster that
// the Morton order tears apart has a near field ten times the mean width, and
// one CTA walking it would be the pass (21,780 panels: mean 93 chunks, widest
// 336): an item gets at most half of what an SM's share of CTAs would do one
// after the other, 24 to 256 chunks.  A pass with 16 right-hand sides, ms: 21,780
// panels 0.687 (the whole share 0.769, a quarter 0.698); 5,120 panels 0.183 (at least 12
// chunks 0.179, 48 0.222); 259,920 panels, leaves of 128, 10.52 (at most 128 10.51, 512
// 10.57).  Items by decreasing work; K: host copies of the panel widths.
void build_fx_items(hm_matrix *A, const std::vector<int32_t> &begin, const std::vector<int32_t> &kd,
                    const std::vector<int32_t> &ku, cudaStream_t s) {
    const int64_t nl = (int64_t)kd.size();
    auto chunks = [&](int64_t r) { return (kd[r] + fx::KC - 1) / fx::KC + (ku[r] + fx::KC - 1) / fx::KC; };
    int64_t total = 0;
    for (int64_t r = 0; r < nl; ++r) total += chunks(r);
    const int lim = (int)std::min<int64_t>(256, std::max<int64_t>(24, total / (2 * 4 * num_sms())));
    std::vector<int4> items, red;
    int slots = 0;
    for (int64_t r = 0; r < nl; ++r) {
        const int nc = chunks(r), parts = std::max(1, (nc + lim - 1) / lim);
        if (parts > 1) red.push_back(make_int4((int)r, slots, parts, 0));
        for (int p = 0; p < parts; ++p)
            items.push_back(make_int4((int)r, (int)((int64_t)nc * p / parts), (int)((int64_t)nc * (p + 1) / parts),
                                      parts > 1 ? slots++ : -1));
    }
    auto work = [&](const int4 &i) { return (int64_t)(i.z - i.y) * (begin[i.x + 1] - begin[i.x]); };
    std::stable_sort(items.begin(), items.end(), [&](const int4 &a, const int4 &b) { return work(a) > work(b); });
    A->fx_nitems = (int64_t)items.size();
    A->fx_nred = (int64_t)red.size();
    A->fx_nslots = slots;
    A->fx_items.alloc(sizeof(int4) * std::max<size_t>(items.size(), 1));
    A->fx_red.alloc(sizeof(int4) * std::max<size_t>(red.size(), 1));
    HM_CUDA_CHECK(cudaMemcpyAsync(A->fx_items.p, items.data(), sizeof(int4) * items.size(), cudaMemcpyHostToDevice, s));
    HM_CUDA_CHECK(cudaMemcpyAsync(A->fx_red.p, red.data(), sizeof(int4) * red.size(), cudaMemcpyHostToDevice, s));
    HM_CUDA_CHECK(cudaStreamSynchronize(s));
}

// floats of the working arrays of one 16-right-hand-side pass: digits of x
// and t (64 each per row), partials of t (32 each), exponents of x and t (2
// each, a multiple of 4 in all), scales (64) and the two lists of clusters,
// partials and states of split rows (32 and 2 per row of a slot, a multiple of 16
// rows), Y (16 doubles per row)
int64_t df_work_floats(const hm_matrix *A) {
    const int64_t n = A->tree->n, K = std::max<int64_t>(A->total_rank, 1), P = std::max<int64_t>(A->n_partials, 1);
    return 64 * n + 32 * P + 64 * K + (2 * n + 3) / 4 * 4 + (2 * K + 3) / 4 * 4 + fx::SCALE_FLOATS +
           2 * fx::todo_ints(A->tree->n_leaf) +
           34 * A->fx_nslots * ((A->tree->max_leaf + 15) / 16 * 16) + 32 * n;
}

// Y (Morton [n][16] FP64) = H_64 x for the nr <= 16 vectors x_r = x[r * n +
// (perm ? perm[m] : m)] (Morton order without perm, original with it); work:
// df_work_floats(A) floats (16-byte aligned).
void matvec_df_block(const hm_matrix *A, const double *x, int nr, const int32_t *perm, double *Y, float *work,
                     cudaStream_t s) {
    using namespace fx;
    const int64_t n = A->tree->n, K = std::max<int64_t>(A->total_rank, 1), P = std::max<int64_t>(A->n_partials, 1);
    Work w;
    float *p = work;
    w.Xd = reinterpret_cast<__half *>(p);
    p += fx::DIG / 2 * n;
    w.P = reinterpret_cast<float2 *>(p);
    p += 32 * P;
    w.Td = reinterpret_cast<__half *>(p);
    p += fx::DIG / 2 * K;
    w.Xe = reinterpret_cast<uint2 *>(p);
    p += (2 * n + 3) / 4 * 4;
    w.Te = reinterpret_cast<uint2 *>(p);
    p += (2 * K + 3) / 4 * 4;
    w.sc = reinterpret_cast<Scale *>(p);
    p += SCALE_FLOATS;
    w.todo_c = reinterpret_cast<int32_t *>(p);
    p += todo_ints(A->tree->n_leaf);
    w.todo_r = reinterpret_cast<int32_t *>(p);
    p += todo_ints(A->tree->n_leaf);
    w.Ypart = reinterpret_cast<float2 *>(p);
    p += 2 * MR * A->fx_nslots * ((A->tree->max_leaf + 15) / 16 * 16);
    w.part_state = reinterpret_cast<uint2 *>(p);
    // at most 8 right-hand sides need one fragment column of the products, not two
    if (nr <= 8) block_product<1>(A, x, nr, perm, Y, w, s);
    else block_product<2>(A, x, nr, perm, Y, w, s);
}

// y = alpha H_64 x + beta y for nrhs right-hand sides [nrhs][n] in the
// original order, 16 at a time (hm_matvec_block with HM_F64)
void matvec_df(const hm_matrix *A, int nrhs, const double *x, double *y, double alpha, double beta, cudaStream_t s) {
    const hm_tree *tr = A->tree;
    const int64_t n = tr->n;
    for (int r0 = 0; r0 < nrhs; r0 += fx::MR) {
        const int nr = std::min(fx::MR, nrhs - r0);
        SBuf buf;
        buf.alloc(sizeof(float) * df_work_floats(A), s);
        float *work = buf.as<float>();
        double *Y = reinterpret_cast<double *>(work + df_work_floats(A) - 32 * n);
        matvec_df_block(A, x + (int64_t)r0 * n, nr, tr->perm.as<int32_t>(), Y, work, s);
        fx::scatter_kernel<<<fx::grid_for(n * nr), 256, 0, s>>>(Y, n, nr, tr->perm.as<int32_t>(), alpha, beta,
                                                            y + (int64_t)r0 * n);
        HM_LAUNCH_CHECK();
    }
}

// yv (Morton [nr][n]) = H_64 xv (Morton [nr][n]) for nr <= 16 vectors
void matvec_df_morton(const hm_matrix *A, const double *xv, int nr, double *yv, float *work, cudaStream_t s) {
    const int64_t n = A->tree->n;
    double *Y = reinterpret_cast<double *>(work + df_work_floats(A) - 32 * n);
    matvec_df_block(A, xv, nr, nullptr, Y, work, s);
    fx::scatter_kernel<<<fx::grid_for(n * nr), 256, 0, s>>>(Y, n, nr, nullptr, 1.0, 0.0, yv);
    HM_LAUNCH_CHECK();
}

}  // namespace hm
