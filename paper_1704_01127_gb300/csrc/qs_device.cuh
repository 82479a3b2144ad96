// Device building blocks shared by the sweeps (qs_apply.cu), the passes
// (qs_pass.cu), the statistics and the draws (qs_api.cu, qs_batch.cu), so that all
// run the same arithmetic.
#pragma once

#include <cuda_runtime.h>
#include <cstdint>

#include "qs_internal.h"

namespace qsd {

template <typename R> struct cplx;
template <> struct cplx<double> { using t = double2; };
template <> struct cplx<float> { using t = float2; };

struct Targets {
    int q[QS_MAX_K];   // ascending
};

// Insert a zero bit at each (ascending) target position: group id -> index of
// the group's x = 0 member (Sec. 3.2: the c bits fill the non-target positions).
template <int K>
__device__ __forceinline__ uint64_t group_base(uint64_t g, const Targets &t)
{
#pragma unroll
    for (int j = 0; j < K; j++) {
        uint64_t lo = g & ((1ULL << t.q[j]) - 1);
        g = ((g ^ lo) << 1) | lo;
    }
    return g;
}

template <int K>
__device__ __forceinline__ uint64_t member_offset(int x, const Targets &t)
{
    uint64_t o = 0;
#pragma unroll
    for (int j = 0; j < K; j++)
        if ((x >> j) & 1) o |= 1ULL << t.q[j];
    return o;
}

// One group of a dense k-qubit cluster (Sec. 3.2): the 2^K amplitudes at
// strides 2^{q_j} are gathered into registers, v <- U v, and scattered back.
// Each complex multiply-accumulate is the pair of real FMA updates of
// Eqs. (2)-(3): acc += (v_R m_R, v_I m_R) then acc += (-v_I m_I, v_R m_I).
template <typename R, int K>
__device__ __forceinline__ void dense_load(const typename cplx<R>::t *p, const Targets &t, typename cplx<R>::t *v)
{
#pragma unroll
    for (int x = 0; x < (1 << K); x++) v[x] = p[member_offset<K>(x, t)];
}

template <typename R, int K>
__device__ __forceinline__ void dense_rows(typename cplx<R>::t *p, const Targets &t, const typename cplx<R>::t *Us,
                                           const typename cplx<R>::t *v)
{
    using C = typename cplx<R>::t;
    constexpr int D = 1 << K;
    // rows of U one at a time (kept rolled so v[] stays in registers)
#pragma unroll 1
    for (int l = 0; l < D; l++) {
        R ar = 0, ai = 0;
        const C *row = Us + l * D;
#pragma unroll
        for (int x = 0; x < D; x++) {
            C m = row[x];
            ar = fma(v[x].x, m.x, ar);
            ai = fma(v[x].y, m.x, ai);
            ar = fma(-v[x].y, m.y, ar);
            ai = fma(v[x].x, m.y, ai);
        }
        C o;
        o.x = ar;
        o.y = ai;
        p[member_offset<K>(l, t)] = o;
    }
}

template <typename R, int K>
__device__ __forceinline__ void dense_group(typename cplx<R>::t *p, const Targets &t,
                                            const typename cplx<R>::t *Us)
{
    typename cplx<R>::t v[1 << K];
    dense_load<R, K>(p, t, v);
    dense_rows<R, K>(p, t, Us, v);
}

// Multiply by e^{i pi m / 4}: an odd m first takes one factor
// e^{i pi/4} = (1 + i)/sqrt(2); the remaining quarter turn i^{m >> 1} only swaps
// and negates, done on the bit patterns (sign-bit flips) so complex128 spends
// no FP64 instruction on it.
__device__ __forceinline__ float flip(float x, bool f) { return __int_as_float(__float_as_int(x) ^ (f ? 0x80000000 : 0)); }
__device__ __forceinline__ double flip(double x, bool f)
{
    return __longlong_as_double(__double_as_longlong(x) ^ (f ? (long long)0x8000000000000000ULL : 0LL));
}

__device__ __forceinline__ float2 eighth_turn(float2 a)   // times e^{i pi / 4}
{
    const float r = 0.70710678118654752440f;
    return make_float2((a.x - a.y) * r, (a.x + a.y) * r);
}
// the FP64 form in volatile statements: the compiler otherwise computes it for
// every amplitude and selects, and the FP64 pipe is the narrow one
__device__ __forceinline__ double2 eighth_turn(double2 a)
{
    double2 b;
    asm volatile("{\n\t.reg .f64 s, d;\n\tsub.rn.f64 d, %2, %3;\n\tadd.rn.f64 s, %2, %3;\n\t"
                 "mul.rn.f64 %0, d, %4;\n\tmul.rn.f64 %1, s, %4;\n\t}"
                 : "=d"(b.x), "=d"(b.y)
                 : "d"(a.x), "d"(a.y), "d"(0.70710678118654752440));
    return b;
}
template <typename C>
__device__ __forceinline__ C quarter_turns(C a, int q)   // times i^q: 0 (x, y), 1 (-y, x), 2 (-x, -y), 3 (y, -x)
{
    q &= 3;
    const bool sw = q & 1;
    C o;
    o.x = flip(sw ? a.y : a.x, q == 1 || q == 2);
    o.y = flip(sw ? a.x : a.y, q >= 2);
    return o;
}
template <typename C, typename R>
__device__ __forceinline__ C rotate8(C a, int m)
{
    if (m & 1) a = eighth_turn(a);
    return quarter_turns<C>(a, m >> 1);
}

// Phase products (Sec. 2, Sec. 3.5): amplitude i gets e^{i pi m(i)/4},
// m(i) = sum_q c_q i_q + 4 sum_a i_a popc(i & P_a) mod 8, with P_a the CZ
// partners b > a of qubit a: the exponent of the bits x alone, both ends of a CZ
// below bit L.
__device__ __forceinline__ uint8_t phase_low(uint64_t x, const uint64_t *cm, const int *act,
                                             const uint64_t *part, int n_act, int L)
{
    const uint64_t lowmask = (1ULL << L) - 1;
    int m = __popcll(x & cm[0]) + 2 * __popcll(x & cm[1]) + 4 * __popcll(x & cm[2]);
    int par = 0;
    for (int t = 0; t < n_act; t++)
        if (act[t] < L && ((x >> act[t]) & 1)) par ^= __popcll(x & part[t] & lowmask);
    return (uint8_t)((m + 4 * (par & 1)) & 7);
}

// fl(x^2) of a double, rounded to nearest even, from integer operations: the
// FP64 unit gives two results a clock per SM, the integer units 64, so a pass
// that also adds in FP64 runs the squares beside it.  x = m 2^(e - 1075), m the
// 53-bit significand; m^2 has 105 or 106 bits (s = 0 or 1) and its top 53 are
// kept: the round bit and the bits below it sit in x (bit 0 set when a dropped
// word is not zero), whose carry out of 2^31 - 1 + lsb is the increment.  Squares
// outside the normal range (and infinities, NaN) take the FP64 unit.
__device__ __forceinline__ double sq_rn(double d)
{
    const uint32_t hi = (uint32_t)__double2hiint(d) & 0x7FFFFFFFu, lo = (uint32_t)__double2loint(d);
    const uint32_t e = hi >> 20;
    if (e - 513u > 1020u) {
        if ((hi | lo) == 0) return 0.0;   // real-valued states: not the FP64 unit for every zero
        double sq;
        asm volatile("mul.rn.f64 %0, %1, %1;" : "=d"(sq) : "d"(d));
        return sq;
    }
    const uint32_t mh = (hi & 0xFFFFFu) | 0x100000u;
    const uint64_t ll = (uint64_t)lo * lo, lh = (uint64_t)lo * mh, hh = (uint64_t)mh * mh;
    uint32_t L1, H0, H1;   // m^2 = H1:H0:L1:L0
    const uint32_t lhl = (uint32_t)lh, lhh = (uint32_t)(lh >> 32);
    asm("add.cc.u32 %0, %3, %4;\n\taddc.cc.u32 %1, %5, %6;\n\taddc.u32 %2, %7, 0;"
        : "=r"(L1), "=r"(H0), "=r"(H1)
        : "r"((uint32_t)(ll >> 32)), "r"(lhl << 1), "r"((uint32_t)hh), "r"(__funnelshift_l(lhl, lhh, 1)),
          "r"((uint32_t)(hh >> 32)));
    const uint32_t s = H1 >> 9, sh = 20u + s;
    const uint32_t ql = __funnelshift_r(L1, H0, sh), qh = __funnelshift_r(H0, H1, sh);
    const uint32_t x = (L1 << (32u - sh)) | ((uint32_t)ll != 0u ? 1u : 0u);
    uint32_t rl, rh;
    asm("{\n\t.reg .u32 t;\n\tadd.cc.u32 t, %2, %3;\n\taddc.cc.u32 %0, %4, 0;\n\taddc.u32 %1, %5, %6;\n\t}"
        : "=r"(rl), "=r"(rh)
        : "r"(x), "r"(0x7FFFFFFFu + (ql & 1u)), "r"(ql), "r"(qh), "r"((2u * e - 1024u + s) << 20));
    return __hiloint2double((int)rh, (int)rl);
}
// p = fl(fl(re^2) + fl(im^2)) in FP64 (no contraction into an FMA).
__device__ __forceinline__ double prob(double2 a)
{
    return __dadd_rn(sq_rn(a.x), sq_rn(a.y));
}
// x^2 of a float as a double, exact: the 24-bit significand squared fits in
// 48 bits, so the product is assembled from integer operations (the same value
// as the FP64 multiplication of x by itself, without the FP64 pipe, which runs
// at 1/64 of the FP32 rate on this part).  |x| = m 2^E; m^2 has its leading
// one at bit t <= 47, so x^2 = 1.f 2^(t + 2E) with f the bits below it; every
// such square, subnormal x included, is a normal double.
__device__ __forceinline__ double sq_exact(float x)
{
    const uint32_t b = __float_as_uint(x) & 0x7fffffffu;
    const uint32_t e = b >> 23;
    if (e == 0xffu) {                                  // inf, nan: the FP64 unit
        const double d = x;
        return __dmul_rn(d, d);
    }
    const uint32_t m = e ? ((b & 0x7fffffu) | 0x800000u) : b;
    if (m == 0) return 0.0;
    const int E = e ? (int)e - 150 : -149;
    const uint64_t q = (uint64_t)m * m;
    const int lz = __clzll((long long)q);             // leading one at bit 63 - lz
    const uint64_t frac = ((q << lz) << 1) >> 12;     // the 52 bits below it
    const uint64_t bexp = (uint64_t)(63 - lz + 2 * E + 1023);
    return __longlong_as_double((long long)((bexp << 52) | frac));
}
static __device__ __noinline__ double prob_rare(float2 v)
{
    if (v.x == 0.f && v.y == 0.f) return 0.0;
    return __dadd_rn(sq_exact(v.x), sq_exact(v.y));
}
// p = fl(x^2 + y^2) with exact squares: fl(fl(x^2) + fl(y^2)) in FP64, in integer
// operations as well, so a pass that adds p in FP64 has that pipe to itself.  With
// a >= b the magnitudes, significands shifted up by 7: A = ma^2 in [2^60, 2^62), and
// mb^2 shifted down by twice the exponents' difference s, its dropped bits joined
// into the lowest one (they lie below the rounding position).  The sum's leading one
// is at bit 60, 61 or 62 and it is rounded to 53 bits, half to even, as in sq_rn.
// Subnormal components, infinities and NaN take the squares one by one.  A zero b
// beside a >= 2^-95 is shifted out altogether (s = 63), and the joined bit is below
// half of a sum whose 14 lowest bits are zero otherwise: p = fl(a^2) without a branch
// of its own.
__device__ __forceinline__ double prob(float2 v)
{
    const uint32_t bx = __float_as_uint(v.x) & 0x7fffffffu, by = __float_as_uint(v.y) & 0x7fffffffu;
    const uint32_t a = max(bx, by), b = min(bx, by);
    if (b < 0x800000u || a >= 0x7f800000u)
        if (b != 0 || a < 0x10000000u || a >= 0x7f800000u) return prob_rare(v);
    const uint32_t ea = a >> 23, ma = (a << 7) & 0x3fffff80u | 0x40000000u, mb = (b << 7) & 0x3fffff80u | 0x40000000u;
    const uint64_t A = (uint64_t)ma * ma, B = (uint64_t)mb * mb;
    const uint32_t s = min(2u * (ea - (b >> 23)), 63u);
    uint64_t r = B >> s;
    if ((r << s) != B) r |= 1u;
    const uint64_t S = A + r;
    const uint32_t lo = (uint32_t)S, hi = (uint32_t)(S >> 32);
    const uint32_t sh = 11u - (uint32_t)__clz((int)hi);   // 8, 9 or 10
    const uint32_t ql = __funnelshift_r(lo, hi, sh), qh = hi >> sh;
    const uint32_t x = lo << (32u - sh);
    uint32_t rl, rh;
    asm("{\n\t.reg .u32 t;\n\tadd.cc.u32 t, %2, %3;\n\taddc.cc.u32 %0, %4, 0;\n\taddc.u32 %1, %5, %6;\n\t}"
        : "=r"(rl), "=r"(rh)
        : "r"(x), "r"(0x7FFFFFFFu + (ql & 1u)), "r"(ql), "r"(qh), "r"((2u * ea + sh + 760u) << 20));
    return __hiloint2double((int)rh, (int)rl);
}

// Natural logarithm of a positive normal double, table-driven (P. T. P. Tang,
// "Table-driven implementation of the logarithm function in IEEE floating-point
// arithmetic", ACM TOMS 16(4), 1990): p = 2^e m, m in [1, 2); c_j is the centre
// of the mantissa interval [1 + j/1024, 1 + (j+1)/1024) picked by the top ten
// mantissa bits, r = m / c_j - 1 (|r| <= 2^-11) and
//   ln p = e ln 2 + ln c_j + ln(1 + r),  ln(1 + r) = r - r^2/2 + r^3/3 - r^4/4,
// truncation error below r^5/5 < 2^-57.  ln c_j and 1/c_j come from the CUDA
// math library once per block (shared-memory table, 16 KB).
constexpr int kLogBits = 10;
struct LogTable {
    double inv[1 << kLogBits], ln[1 << kLogBits];
};

__device__ __forceinline__ void log_table_init(LogTable &t)
{
    for (int j = threadIdx.x; j < (1 << kLogBits); j += blockDim.x) {
        const double c = 1.0 + (j + 0.5) / (double)(1 << kLogBits);
        t.inv[j] = 1.0 / c;
        t.ln[j] = log(c);
    }
}

__device__ __forceinline__ double log_tab(const LogTable &t, double p)
{
    const long long bits = __double_as_longlong(p);
    const int e = (int)(bits >> 52) - 1023;
    const int j = (int)((bits >> (52 - kLogBits)) & ((1 << kLogBits) - 1));
    const double m = __longlong_as_double((bits & 0xFFFFFFFFFFFFFLL) | 0x3FF0000000000000LL);
    const double r = fma(m, t.inv[j], -1.0);
    double q = -0.25;
    q = fma(q, r, 1.0 / 3.0);
    q = fma(q, r, -0.5);
    q = fma(q, r, 1.0);
    return fma((double)e, 0.69314718055994530942, fma(q, r, t.ln[j]));
}

// ---------------------------------------------------------------------------
// Float-float ("double-float") arithmetic: a value is hi + lo with |lo| at most
// half an ulp of hi, about 48 significant bits.  Error-free transforms after
// Knuth (two-sum), Dekker (fast two-sum) and the FMA product error; GB300's
// FP32 pipe is ~64x its FP64 pipe, so 10-20 FP32 operations per emulated
// operation still run far faster than FP64.
struct ff {
    float hi, lo;
};
__device__ __forceinline__ ff ff_two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    return ff{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ ff ff_fast_two_sum(float a, float b)   // |a| >= |b| or a = 0
{
    const float s = __fadd_rn(a, b);
    return ff{s, __fsub_rn(b, __fsub_rn(s, a))};
}
// x^2 exactly as hi + lo (the FMA gives the rounding error of the product)
__device__ __forceinline__ ff ff_sqr_f(float x)
{
    const float p = __fmul_rn(x, x);
    return ff{p, fmaf(x, x, -p)};
}
// x^2 with its low part left unnormalised (the product's rounding error plus
// 2 x.hi x.lo; x.lo^2 is below 2^-48 of the result)
__device__ __forceinline__ ff ff_sqr_loose(ff x)
{
    const float p = __fmul_rn(x.hi, x.hi);
    return ff{p, fmaf(__fadd_rn(x.hi, x.hi), x.lo, fmaf(x.hi, x.hi, -p))};
}
// s += a, the error of the high parts' sum and a's low part collected in s.lo and
// not folded back (Ogita, Rump and Oishi's Sum2, SIAM J. Sci. Comput. 26, 2005): s.lo
// grows with the number of terms, and its roundings with it (of k equal terms they all
// go one way, some k^2 2^-50 of the sum), so a sum takes a few terms and goes into
// another one by ff_add
__device__ __forceinline__ void ff_accumulate(ff &s, ff a)
{
    const ff t = ff_two_sum(s.hi, a.hi);
    s.hi = t.hi;
    s.lo = __fadd_rn(s.lo, __fadd_rn(t.lo, a.lo));
}
__device__ __forceinline__ void ff_accumulate(ff &s, float a)
{
    const ff t = ff_two_sum(s.hi, a);
    s.hi = t.hi;
    s.lo = __fadd_rn(s.lo, t.lo);
}
// a + b, normalised
__device__ __forceinline__ ff ff_add(ff a, ff b)
{
    const ff s = ff_two_sum(a.hi, b.hi);
    return ff_fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
// |d| of a double with |d| in [2^-60, 2^30), its high word h without the sign:
// hi = its top 24 significant bits (the exponent rebased by flipping one bit),
// lo = the other 29, rounded to 24
__device__ __forceinline__ ff ff_abs_double(uint32_t h, uint32_t l)
{
    const uint32_t b = (__funnelshift_l(l, h, 3) ^ 0x40000000u) & 0x7FFFFFFFu;
    const float scale = __uint_as_float((b & 0x7F800000u) - (52u << 23));   // a unit of d's last place
    return ff{__uint_as_float(b), __fmul_rn(__uint2float_rn(l & 0x1FFFFFFFu), scale)};
}
// A double d with |d| in [2^-126, 2^128) by bit manipulation only: hi = its top 24
// significant bits, lo = the other 29 rounded to 24 (0 when they fall below the
// normal float range).  Relative error 2^-48 at most.
__device__ __forceinline__ ff ff_from_double(double d)
{
    const uint32_t hw = (uint32_t)__double2hiint(d), lw = (uint32_t)__double2loint(d);
    const int E = (int)((hw >> 20) & 0x7FFu) - 1023;
    const uint32_t sign = hw & 0x80000000u;
    const float hi = __uint_as_float(sign | ((uint32_t)(E + 127) << 23) | ((hw & 0xFFFFFu) << 3) | (lw >> 29));
    const float scale = __uint_as_float((uint32_t)max(E - 52 + 127, 0) << 23);   // 2^(E-52) or 0
    const float lo = __uint2float_rn(lw & 0x1FFFFFFFu) * scale;
    return ff{hi, sign ? -lo : lo};
}

// p ln p for p in [2^-79, 2^100] in float-float, table-driven after Tang
// (ACM TOMS 16(4), 1990): p = 2^e m, c_j the centre of the mantissa interval
// picked by the top ten bits, r = m / c_j - 1 (|r| < 2^-10), and
//   ln p = e ln 2 + ln c_j + r - r^2/2 + r^3/3 - r^4/4,
// with e ln 2, ln c_j and 1/c_j as float-float table entries.  The error of
// ln p is about 2^-48 of |e ln 2| + |ln c_j| plus 2^-55 (float-float
// rounding), so each term p ln p carries a relative error near 2^-47.
constexpr int kFFLogBits = 10;
struct FFLogTable {
    ff inv[1 << kFFLogBits], ln[1 << kFFLogBits];
    ff eln2[255];   // e ln 2 for e = -127 .. 127
};
__device__ __forceinline__ void ff_log_table_init(FFLogTable &t)
{
    for (int j = threadIdx.x; j < (1 << kFFLogBits); j += blockDim.x) {
        const double c = 1.0 + (j + 0.5) / (double)(1 << kFFLogBits);
        t.inv[j] = ff_from_double(1.0 / c);
        t.ln[j] = ff_from_double(log(c));
    }
    for (int e = threadIdx.x; e < 255; e += blockDim.x)
        t.eln2[e] = e == 127 ? ff{0.0f, 0.0f} : ff_from_double((double)(e - 127) * 0.69314718055994530942);
}
__device__ __forceinline__ ff ff_p_ln_p(const FFLogTable &t, ff p)
{
    const uint32_t b = __float_as_uint(p.hi);
    const int e = (int)((b >> 23) & 0xFFu) - 127;
    const int j = (int)((b >> (23 - kFFLogBits)) & ((1u << kFFLogBits) - 1));
    // m = p 2^-e: the exponent of hi replaced, lo scaled by the same power of two
    const ff m = ff{__uint_as_float((b & 0x807FFFFFu) | (127u << 23)), p.lo * __uint_as_float((uint32_t)(127 - e) << 23)};
    // r = m / c_j - 1: hi - 1 is exact (hi within 2^-10 of 1)
    const ff inv = t.inv[j];
    const float ph = __fmul_rn(m.hi, inv.hi);
    const float pl = fmaf(m.hi, inv.lo, fmaf(m.lo, inv.hi, fmaf(m.hi, inv.hi, -ph)));
    const ff r = ff_fast_two_sum(__fsub_rn(ph, 1.0f), pl);
    // ln(1 + r) = r - r^2/2 + r^3/3 - r^4/4: -x^2/2 (x = r.hi) exactly as
    // float-float, the rest (below 2^-32) in FP32, -x r.lo for the cross term.
    // e ln 2, x and -x^2/2 are summed with their errors; the low parts add up in FP32
    const float x = r.hi;
    const ff sq = ff_sqr_f(x);
    const float tail = fmaf(x * x * x, fmaf(x, -0.25f, 0.33333334f), -x * r.lo);
    const ff el = t.eln2[e + 127], lc = t.ln[j];
    const ff s0 = ff_fast_two_sum(el.hi, lc.hi);        // |e ln 2| >= ln c_j, or e = 0
    const ff s1 = ff_two_sum(s0.hi, x), s2 = ff_two_sum(s1.hi, -0.5f * sq.hi);
    const float lo = ((s0.lo + s1.lo) + (s2.lo + (el.lo + lc.lo))) + (r.lo + fmaf(-0.5f, sq.lo, tail));
    // p ln p, the low part left unnormalised
    const float q = __fmul_rn(p.hi, s2.hi);
    return ff{q, fmaf(p.lo, s2.hi, fmaf(p.hi, lo, fmaf(p.hi, s2.hi, -q)))};
}

}  // namespace qsd
