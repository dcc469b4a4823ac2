// Short-characteristics weights in 64-bit integer arithmetic for the FP64 sweeps.
//
// GB300 executes about 1.7 FP64 operations per clock and SM (2 lanes), against 61
// 32-bit integer multiply-adds, 23 widening ones and 64 logic operations, so
// an FP64 multiply-add takes the time of 14-35 integer instructions, and the
// exponential, reciprocal and differences of one set of weights (16 FP64
// operations) were half the arithmetic of the FP64 sweep.  Here they run on
// the integer pipes instead (about 100 instructions a set) and leave the FP64
// pipe to the intensities: 4.10 -> 1.93 ms for the two-level sweep of 64x64x129
// nodes and 9 frequencies.
//
// The weights of a step with optical path x >= 0 (I = I_up e^-x + w_up S_up +
// w0 S, u = (1 - e^-x)/x, w0 = 1 - u, w_up = u - e^-x) are all in [0, 1].  They
// are formed as 64-bit fractions (units of 2^-64) and rounded once to FP64.
// Operands are (m, e): the value m 2^-64 2^e with the top bit of m set.
//
//   x >= 2^-11: y = x log2 e = n + f; 2^-f = A (1 - W), A = 2^-j1/256 and
//     1 - W = 2^-j2/65536 e^-t from two 256-entry tables and the series of
//     1 - e^-t (t < 2^-16.5), so e^-x has an absolute error below 2^-55.5
//     (FP64: 2^-54); 1 - e^-x is exact from there, u its product with 1/x, and
//     the differences w0 and w_up are exact subtractions of fractions.
//   x < 2^-9 (the caller chooses by the exponent): the Taylor series of w0/x and
//     w_up/x to x^4, as fractions with the product taken on the mantissa of x.
//
// Against 113-bit arithmetic, over 2e5 arguments per octave of x: w0 and w_up
// are within 2^-52 for x < 2^-10 and then within 2^-35 at 2^-10, rising to
// 2^-52 at x = 8 and beyond (the FP64 form: 2^-31 at 2^-11, 2^-33 at 2^-10,
// 2^-52 from x = 8), e^-x within 2^-52.4 everywhere.
#pragma once

#include <cuda_runtime.h>

#include <cmath>

#include "sc_step.cuh"

namespace mg3d {
namespace fx {

typedef unsigned long long u64;

constexpr u64 kLn2 = 0xB17217F7D1CF79ACull;    // ln 2
constexpr u64 kLog2e = 0xB8AA3B295C17F0BCull;  // log2(e) / 2
constexpr int kTab = 256;                      // entries of each table
constexpr int kThinExp = -10;                  // exponents of x up to this take the series
// exponents of dtau and of a profile value for which every product stays in
// the FP64 range; others take the FP64 weights
constexpr int kNodeExp = 700;
constexpr int kSlotExp = 250;

// Host: mantissa and exponent of a positive value.
inline void split(long double v, u64 *m, int *e) {
    int ex = 0;
    const long double f = std::frexp(v, &ex);   // f in [1/2, 1)
    *m = (u64)std::ldexp(f, 64);
    *e = ex;
}

// high 64 bits of a b, up to 2 units below (the low partial product is left out)
__device__ __forceinline__ u64 mulhi(u64 a, u64 b) {
    const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a;
    const unsigned bh = (unsigned)(b >> 32), bl = (unsigned)b;
    return (u64)ah * bh + (((u64)ah * bl) >> 32) + (((u64)al * bh) >> 32);
}
__device__ __forceinline__ u64 shr(u64 a, int s) { return s < 64 ? a >> s : 0; }
__device__ __forceinline__ u64 join(unsigned hi, unsigned lo) { return ((u64)hi << 32) | lo; }

// m 2^-64 2^e (top bit set) as a double, rounded to nearest; a carry out of the
// mantissa runs into the exponent
__device__ __forceinline__ double pack(u64 m, int e) {
    const u64 r = (m >> 11) + ((unsigned)(m >> 10) & 1u);
    return __longlong_as_double((long long)(r + join((unsigned)(e + 1021) << 20, 0u)));
}
// the same for m >= 2^62
__device__ __forceinline__ double pack62(u64 m, int e) {
    const int z = 1 - (int)(m >> 63);
    return pack(m << z, e - z);
}
// the same for m >= 2^32
__device__ __forceinline__ double pack32(u64 m, int e) {
    const int z = __clz((unsigned)(m >> 32));
    return pack(m << z, e - z);
}

// mantissa and exponent of a positive normal double
__device__ __forceinline__ void unpack(double v, u64 *m, int *e) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    *m = join(__funnelshift_l(lo, hi, 11) | 0x80000000u, lo << 11);
    *e = (int)(hi >> 20) - 1022;
}
// sign 0 and |exponent| <= kNodeExp: the integer weights apply
__device__ __forceinline__ bool in_range(double v) {
    return (unsigned)__double2hiint(v) - ((unsigned)(1022 - kNodeExp) << 20) <
           ((unsigned)(2 * kNodeExp) << 20);
}

// 1/(m 2^-64) = r 2^-63 (r = 2^64 - 1 for m = 2^63): a 22-bit start from the FP32
// reciprocal and one step r0 (1 + e + e^2), e = 1 - m r0, whose error is e^3
__device__ __forceinline__ u64 recip(u64 m) {
    const unsigned mh = (unsigned)(m >> 32);
    float f;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"(__uint2float_rz(mh)));
    const unsigned r0 = __float2uint_rz(fminf(f * 9223372036854775808.0f, 4294967040.0f));
    const u64 p = (u64)mh * r0 + (((u64)(unsigned)m * r0) >> 32);       // m r0, 2^-63
    const long long e = (long long)(0x8000000000000000ull - p);         // 2^-63, |e| < 2^43
    const int eh = (int)(e >> 13);                                      // 2^-50
    const unsigned el = (unsigned)e & 0x1fffu;                          // 2^-63
    const long long d1 = (((long long)r0 * eh) >> 18) + (long long)(((u64)r0 * el) >> 31);
    const long long e2 = ((long long)eh * eh) >> 32;                    // e^2, 2^-68
    return join(r0, 0u) + (u64)d1 + (u64)(((long long)r0 * e2) >> 36);
}

// Host: the two tables below, [2][kTab].
inline void build_tables(u64 *t) {
    const long double one = 18446744073709551616.0L;   // 2^64
    for (int j = 0; j < kTab; ++j) {
        t[j] = j == 0 ? ~0ull : (u64)(std::exp2(-(long double)j / 256) * one);
        t[kTab + j] = (u64)(-std::expm1(-(long double)j / 65536 * 0.693147180559945309417232L) * one);
    }
}

// The two tables: A[j] = 2^(-j/256) (A[0] = 2^64 - 1) and V[j] = 1 - 2^(-j/65536).
struct Tables {
    const u64 *A, *V;
};

// 2^-y = E 2^-64 2^-n for y = Y 2^-64 2^e, -12 <= e <= 11; E >= 2^63 - 2^9
__device__ __forceinline__ u64 exp2_neg(u64 Y, int e, const Tables t, int *n) {
    const unsigned yh = (unsigned)(Y >> 32), yl = (unsigned)Y;
    const int s = e + 12;   // y 2^12 = w2.w1w0
    const unsigned w2 = __funnelshift_l(yh, 0u, s), w1 = __funnelshift_l(yl, yh, s);
    const unsigned w0 = yl << s;
    *n = (int)(w2 >> 12);
    const unsigned fh = __funnelshift_r(w1, w2, 12), fl = __funnelshift_r(w0, w1, 12);
    const unsigned gh = __funnelshift_l(fl, fh, 16), gl = fl << 16;   // f below 2^-16
    constexpr unsigned lh = (unsigned)(kLn2 >> 32), ll = (unsigned)kLn2;
    const u64 tq = (u64)gh * lh + (((u64)gh * ll) >> 32) + (((u64)gl * lh) >> 32);  // 2^-80
    const unsigned th = (unsigned)(tq >> 32);                      // t, 2^-48
    const unsigned t2 = __umulhi(th, th);                          // t^2, 2^-64
    const unsigned t3 = __umulhi(t2, th);                          // t^3, 2^-80
    const u64 v = (tq >> 16) - (t2 >> 1) + (t3 >> 16) / 6u;        // 1 - e^-t
    const u64 v2 = t.V[(fh >> 16) & 255u];
    const u64 W = v2 + v - (((v2 >> 24) * (u64)(unsigned)((v + 0x8000u) >> 16)) >> 24);
    const u64 A = t.A[fh >> 24];
    return A - mulhi(A, W);
}

// e^-x and 1 - e^-x for x >= 0: e^-x = E 2^-64 2^-n (0 below 2^-1015), and
// 1 - e^-x = D 2^-64; false for x outside 2^-11 .. 2^700 (E, D not set).
__device__ __forceinline__ bool exp_parts(double x, const Tables t, u64 *E, int *n, u64 *D) {
    u64 m;
    int e;
    unpack(x, &m, &e);
    if (!in_range(x) || e <= kThinExp) return false;
    *E = exp2_neg(mulhi(m, kLog2e), min(e + 1, 11), t, n);
    if (e + 1 > 11 || *n > 1015) *E = 0;
    const u64 Eq = shr(*E, *n);
    *D = Eq ? 0ull - Eq : ~0ull;
    return true;
}
// e^-x in FP64 for x >= 0 (absolute error below 2^-55.5, then one rounding)
__device__ __forceinline__ double exp_neg_fx(double x, const Tables t) {
    u64 E, D;
    int n;
    if (exp_parts(x, t, &E, &n, &D)) return E ? pack62(E, -n) : 0.0;
    // below 2^-11: the Taylor series to x^4
    if (x < 1.0) return fma(x, fma(x, fma(x, fma(x, 1.0 / 24.0, -1.0 / 6.0), 0.5), -1.0), 1.0);
    return exp(-x);
}
struct Weights {
    u64 E;           // e^-x = E 2^-64 2^-n (0: below 2^-1015)
    int n;
    u64 D;           // 1 - e^-x, 2^-64 (closed form)
    u64 u;           // u, 2^-64
    u64 um;          // u = um 2^-64 2^ue without the loss of bits for large x (closed form)
    int ue;
    double w0, wup;
};

// x >= 2^-11: y = x log2 e = (Y, ey), 1/x = V 2^-64 2^ve
__device__ __forceinline__ Weights closed(u64 Y, int ey, u64 V, int ve, const Tables t) {
    Weights w;
    w.E = exp2_neg(Y, min(ey, 11), t, &w.n);
    if (ey > 11 || w.n > 1015) w.E = 0;
    const u64 Eq = shr(w.E, w.n);
    w.D = Eq ? 0ull - Eq : ~0ull;
    w.um = mulhi(w.D, V);
    w.ue = ve;
    w.u = ve >= 0 ? w.um << ve : shr(w.um, -ve);
    w.w0 = pack32(w.u ? 0ull - w.u : ~0ull, 0);   // x > 2^64: u rounds to 0
    // where e^-x is below 2^-64, w_up = u
    w.wup = Eq ? pack32(w.u - Eq, 0) : pack32(w.um, ve);
    return w;
}

// x = (P, ex), ex <= kThinExp; P >= 2^62
__device__ __forceinline__ Weights thin(u64 P, int ex) {
    Weights w;
    const u64 X = shr(P, -ex);                               // x, 2^-64
    const unsigned xh = (unsigned)(X >> 22);                 // 2^-42
    const u64 a = mulhi(X, 0x2AAAAAAAAAAAAAABull);           // x/6
    const unsigned x2 = __umulhi(xh, xh);                    // x^2, 2^-52
    const u64 b = ((u64)x2 * 0xAAAAAAABu) >> 24;             // x^2/24
    const unsigned x3 = __umulhi(x2, xh);                    // x^3, 2^-62
    const unsigned c = __umulhi(x3, 0x08888889u);            // x^3/120
    const unsigned d = __umulhi(__umulhi(x3, xh), 23302u);   // x^4/720
    const u64 half = 0x8000000000000000ull;
    const u64 m0 = mulhi(P, half - a + b - c + d);
    const u64 m1 = mulhi(P, half - 2 * a + 3 * b - 4ull * c + 5ull * d);
    w.w0 = pack32(m0, ex);
    w.wup = pack32(m1, ex);
    const u64 q0 = shr(m0, -ex), q = q0 + shr(m1, -ex);
    w.E = q ? 0ull - q : ~0ull;
    w.n = 0;
    w.u = q0 ? 0ull - q0 : ~0ull;
    w.D = 0;
    w.um = w.u;
    w.ue = 0;
    return w;
}

}  // namespace fx
}  // namespace mg3d
