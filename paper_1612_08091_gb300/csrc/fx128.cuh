// fx128.cuh -- complex128 gate arithmetic in shared-exponent integers.
//
// An SM of this part does 1.9 FP64 FMAs a cycle but 56 integer multiply-adds
// 32 x 32 + 64 -> 64 (mad.wide; both measured), so a dense gate on complex128
// amplitudes, 8 FMAs an amplitude, is bound by FP64 at a third of the HBM
// bandwidth while its integer form is not.  The amplitudes of a group (the
// 2^k that one gate mixes) are brought to one exponent E, the largest of
// theirs, as 59-bit integers v = x 2^(1081 - E), split v = hi 2^28 + lo with
// 0 <= lo < 2^28; a matrix element is w = m 2^S in the same form, at most 57
// bits.  A product is hi hi' 2^56 + (hi lo' + lo hi') 2^28, three
// multiply-adds into two 64-bit sums that are exact (lo lo', below 2^-60 of
// the largest term, is left out).  The result keeps 2^-60 of the group's
// scale and is rounded to double once.
//
// Error.  Every input and matrix element is off by at most 2^-58 of the
// group's (matrix's) largest component, so a result is off by some 2^-57
// sum |m| max |x| plus its one rounding.  FP64 arithmetic rounds each product
// to 2^-53 of itself.  Where every |m| is at least 2^-kFxMinLog of the
// largest, a product with the group's largest amplitude is in every result,
// so FP64's own error of the result, as a complex number, is of at least the
// same size: that is the condition under which the FP64 gates take this path
// (make_fx).  Measured against 128-bit sums on 300,000 random U3 gates: 4.7e-17
// of the result's norm, FP64 7.3e-17, whatever the spread of the inputs'
// exponents.
// A result's real and imaginary parts each have this error: with general
// complex elements the smaller of the two is known to 2^-57 of the group, not
// of itself.  Matrices whose elements are each real or imaginary (H, RX, RY and
// their products with Paulis) do not mix all four components, and FP64 keeps
// the two sets that they do mix apart: there each set has an exponent of its
// own (Apart), so that a result's component is as exact, against the components
// it comes from, as in FP64, and zeros of either sign are exact.
//
// Groups whose exponent is near the ends of the range, and infinities and
// NaN, are left to FP64 (fx_range).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <complex>

#include "common.cuh"

namespace qsim_fx {

constexpr int kFxMinLog = 4;

struct Fx {  // hi 2^28 + lo, 0 <= lo < 2^28
    int hi, lo;
};

// exponent word of a double (sign cleared): its biased exponent is this >> 20
__device__ __forceinline__ uint32_t mag(double x) { return (uint32_t)__double2hiint(x) & 0x7FFFFFFFu; }
__device__ __forceinline__ uint32_t mag(double2 z) { return max(mag(z.x), mag(z.y)); }
// the exponents this arithmetic takes (amplitudes of 2^-894 to 2^961): with
// matrices between 2^-64 and kFxMatrixTop all intermediate and result
// exponents are those of normal numbers (a result is below 2^961 2^59)
__device__ __forceinline__ bool fx_range(int E) { return E > 128 && E < 0x7C0; }
constexpr double kFxMatrixLow = 0x1p-64, kFxMatrixTop = 0x1p56;

// arithmetic right shift, by more than 63 too
__device__ __forceinline__ long long shr_s64(long long v, uint32_t s) {
#ifdef __CUDA_ARCH__
    asm("shr.s64 %0, %0, %1;" : "+l"(v) : "r"(s));
    return v;
#else
    return v >> (s < 63 ? s : 63);
#endif
}

// floor(x 2^(1081 - E)) (one less for some exact negative values and -0.0);
// E >= the biased exponent of x
__device__ __forceinline__ Fx to_fx(double x, int E) {
    const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
    const unsigned long long m = (((unsigned long long)((h & 0xFFFFFu) | 0x100000u) << 32) | l) << 6;
    const uint32_t sg = (uint32_t)((int)h >> 31);
    long long v = (long long)(m ^ (((unsigned long long)sg << 32) | sg));
    v = shr_s64(v, (uint32_t)(E - (int)((h >> 20) & 0x7FFu)));
    return Fx{(int)(v >> 28), (int)((uint32_t)v & 0xFFFFFFFu)};
}
// the same rounded towards zero (E > 64): exact zeros and negative values
// (with it a gate that mixes all components takes 3.5 % longer)
__device__ __forceinline__ Fx to_fx_exact(double x, int E) {
    const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
    const unsigned long long m = (((unsigned long long)((h & 0xFFFFFu) | 0x100000u) << 32) | l) << 6;
    const long long sg = (int)h >> 31;
    const long long v = (shr_s64((long long)m, (uint32_t)(E - (int)((h >> 20) & 0x7FFu))) ^ sg) - sg;
    return Fx{(int)(v >> 28), (int)((uint32_t)v & 0xFFFFFFFu)};
}

// sum of products: a 2^56 + b 2^28
struct Acc {
    long long a, b;
};
// s + a b.  Written out: from (long long)a * b with a factor it knows not to
// be negative the compiler makes several mixed-sign instructions (3.5 in
// place of one in a block gate).
__device__ __forceinline__ long long mad_wide(int a, int b, long long s) {
#ifdef __CUDA_ARCH__
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(s) : "r"(a), "r"(b));
    return s;
#else
    return s + (long long)a * b;
#endif
}
__device__ __forceinline__ void mac(Acc &s, Fx m, Fx x) {
    s.a = mad_wide(m.hi, x.hi, s.a);
    s.b = mad_wide(m.hi, x.lo, s.b);
    s.b = mad_wide(m.lo, x.hi, s.b);
}

// The sum as a double: units of 2^(E - 1081 - S); eadd = (E - 1025 - S) 2^20.
// The conversion runs on the FP64 units (two a cycle), which have nothing else
// to do here; the same steps in 32-bit integers (leading zeros, shift, round)
// took twice the whole gate's other integer work.
__device__ __forceinline__ double to_double(const Acc &s, int eadd) {
    const double d = (double)(s.a + (s.b >> 28));  // units of 2^56; |.| <= 2^62 + 2^34
    const int h = __double2hiint(d);
    return __hiloint2double(h ? h + eadd : 0, __double2loint(d));
}

// ---------------------------------------------------------------------------
// gates on several qubits: 55 bits, the cross sums in FP32
// ---------------------------------------------------------------------------
// For the handles that allow double-float accuracy.  v = x 2^(1077 - E) = hi
// 2^25 + lo with 30 bits and a sign in hi, lo rounded to nearest (-2^24..2^24);
// a matrix element w = m 2^S in the same form, scaled so that its largest row
// sum of |re| + |im| is below 2^55.  The sum of hi hi' is exact in 64 bits (one
// multiply-add a product, four cycles of a pipe that plain FP32 does not
// need); the cross terms, 2^-30 of it, go to two FP32 sums.  Error of a result,
// in units of U, the largest row sum times the group's largest component, each
// rounded up to a power of two (random unitaries on 2 to 4 qubits): at most
// 2^-50.6 with 16 amplitudes that are not 0, 2^-51.3 with 8, 2^-52 with 4, 2^-52.6
// with 2, 2^-53.3 with one; standard deviations 2^-53.7 to 2^-55.7.
struct FxF {  // an amplitude's component
    int hi;
    float fhi, flo;  // hi and lo, hi rounded
};
__device__ __forceinline__ FxF to_fxf(double x, int E) {
    const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
    const unsigned long long m = (((unsigned long long)((h & 0xFFFFFu) | 0x100000u) << 32) | l) << 2;
    const uint32_t sg = (uint32_t)((int)h >> 31);
    const long long v = shr_s64((long long)(m ^ (((unsigned long long)sg << 32) | sg)),
                                (uint32_t)(E - (int)((h >> 20) & 0x7FFu)));
    FxF r;
    r.hi = (int)((v + (1 << 24)) >> 25);
    r.fhi = (float)r.hi;
    r.flo = (float)(int)((uint32_t)v - ((uint32_t)r.hi << 25));
    return r;
}
// a 2^50 + c 2^25 as a double: units of 2^(E - 1077 - S); eadd = (E - 1027 - S)
// 2^20.  |c| <= 2^54 + 2^59: sum |w.hi| <= 2^30 times |lo| <= 2^24, and up to 32
// terms of |w.lo| <= 2^24 times |hi| <= 2^30; it is rounded to 2^4 units of a,
// 2^-56 of the largest a.
__device__ __forceinline__ double to_double_f(long long a, float c, int eadd) {
    const double d = (double)mad_wide(__float2int_rn(c * 0x1p-29f), 16, a);
    const int h = __double2hiint(d);
    return __hiloint2double(h ? h + eadd : 0, __double2loint(d));
}

// A 2x2 matrix in this form.  Element e of an Apart matrix is real or (bit e of
// `imag`) imaginary; its re and im are then the factors of the results' real
// and imaginary parts.
struct MatFx {
    Fx re[4], im[4], nim[4];  // m 2^S; nim = -im
    int shift, apart, imag;   // shift: -1025 - S
    int pad;
    double2 m[4];             // the matrix itself, for groups outside the range
};

// row r of M times (a, b)
__device__ __forceinline__ double2 row(const MatFx &M, int r, Fx ar, Fx ai, Fx br, Fx bi, int E) {
    Acc x{0, 0}, y{0, 0};
    mac(x, M.re[2 * r], ar);
    mac(x, M.nim[2 * r], ai);
    mac(x, M.re[2 * r + 1], br);
    mac(x, M.nim[2 * r + 1], bi);
    mac(y, M.re[2 * r], ai);
    mac(y, M.im[2 * r], ar);
    mac(y, M.re[2 * r + 1], bi);
    mac(y, M.im[2 * r + 1], br);
    const int eadd = (E + M.shift) << 20;
    return make_double2(to_double(x, eadd), to_double(y, eadd));
}
// the same in FP64, outside the range (zeros stay zeros)
__device__ __forceinline__ double2 row_fp64(const MatFx &M, int r, double2 a, double2 b) {
    if (a.x == 0.0 && a.y == 0.0 && b.x == 0.0 && b.y == 0.0) return make_double2(0.0, 0.0);
    return qsim_dev::cfma(M.m[2 * r + 1], b, qsim_dev::cmul(M.m[2 * r], a));
}

// Two components that an Apart matrix mixes, with their exponent; E = 0 for
// two zeros, -1 outside the range.
struct Side {
    Fx a, b;
    int E;
};
__device__ __forceinline__ Side side(double a, double b) {
    const int E = (int)(max(mag(a), mag(b)) >> 20);
    if (fx_range(E)) return Side{to_fx_exact(a, E), to_fx_exact(b, E), E};
    return Side{Fx{0, 0}, Fx{0, 0}, a == 0.0 && b == 0.0 ? 0 : -1};
}
__device__ __forceinline__ double side_sum(const MatFx &M, Fx wa, Fx wb, const Side &s) {
    Acc t{0, 0};
    mac(t, wa, s.a);
    mac(t, wb, s.b);
    return to_double(t, (s.E + M.shift) << 20);
}
// row r of an Apart M: p and q are the components that row 0 takes its real and
// its imaginary part from
__device__ __forceinline__ double2 apart_row(const MatFx &M, int r, const Side &p, const Side &q) {
    const bool crossed = r && ((M.imag ^ (M.imag >> 2)) & 1);
    return make_double2(side_sum(M, M.re[2 * r], M.re[2 * r + 1], crossed ? q : p),
                        side_sum(M, M.im[2 * r], M.im[2 * r + 1], crossed ? p : q));
}
__device__ __forceinline__ bool apart_sides(const MatFx &M, double2 a, double2 b, Side &p, Side &q) {
    const bool ia = M.imag & 1, ib = M.imag & 2;
    p = side(ia ? a.y : a.x, ib ? b.y : b.x);
    q = side(ia ? a.x : a.y, ib ? b.x : b.y);
    return p.E >= 0 && q.E >= 0;
}

// (na, nb) = M (a, b); Apart as M.apart
template <bool Apart>
__device__ __forceinline__ void dense1(const MatFx &M, double2 a, double2 b, double2 &na, double2 &nb) {
    if constexpr (Apart) {
        Side p, q;
        if (apart_sides(M, a, b, p, q)) {
            na = apart_row(M, 0, p, q);
            nb = apart_row(M, 1, p, q);
            return;
        }
    } else {
        const int E = (int)(max(mag(a), mag(b)) >> 20);
        if (fx_range(E)) {
            const Fx ar = to_fx(a.x, E), ai = to_fx(a.y, E), br = to_fx(b.x, E), bi = to_fx(b.y, E);
            na = row(M, 0, ar, ai, br, bi, E);
            nb = row(M, 1, ar, ai, br, bi, E);
            return;
        }
    }
    na = row_fp64(M, 0, a, b);
    nb = row_fp64(M, 1, a, b);
}
// one row of it
__device__ __forceinline__ double2 dense1_row(const MatFx &M, int r, double2 a, double2 b) {
    const int E = (int)(max(mag(a), mag(b)) >> 20);
    Side p, q;
    if (M.apart && apart_sides(M, a, b, p, q)) return apart_row(M, r, p, q);
    if (M.apart || !fx_range(E)) return row_fp64(M, r, a, b);
    return row(M, r, to_fx(a.x, E), to_fx(a.y, E), to_fx(b.x, E), to_fx(b.y, E), E);
}

// Host: m 2^S as hi 2^28 + lo, rounded to nearest (|m| 2^S <= 2^57).
inline Fx host_fx(double m, int S) {
    const long long w = std::llrint(std::ldexp(m, S));
    return Fx{(int)(w >> 28), (int)(w & 0xFFFFFFF)};
}

// Host: the integer form of a 2x2 matrix (row-major); false where it would be
// less exact than FP64 (an element below 2^-kFxMinLog of the largest) or out
// of the exponents it is made for.
inline bool make_fx(const std::complex<double> *m, MatFx &M) {
    double top = 0.0, low = 1e300, comp = 0.0;
    for (int e = 0; e < 4; ++e) {
        top = std::max(top, std::abs(m[e]));
        low = std::min(low, std::abs(m[e]));
        comp = std::max(comp, std::max(std::abs(m[e].real()), std::abs(m[e].imag())));
    }
    if (!(low >= std::ldexp(top, -kFxMinLog)) || !(top > kFxMatrixLow) ||
        !(top < kFxMatrixTop))
        return false;
    int x;
    std::frexp(comp, &x);  // comp < 2^x
    const int S = 57 - x;
    M.apart = 1;
    M.imag = M.pad = 0;
    for (int e = 0; e < 4; ++e) {
        M.apart &= m[e].real() == 0.0 || m[e].imag() == 0.0;
        M.imag |= (m[e].real() == 0.0) << e;
    }
    // two rows that mix the components differently (no unitary does): FP64
    if (M.apart && (__builtin_popcount(M.imag) & 1)) return false;
    for (int e = 0; e < 4; ++e) {
        const bool im = (M.imag >> e) & 1;
        M.re[e] = host_fx(M.apart && im ? -m[e].imag() : m[e].real(), S);
        M.im[e] = host_fx(M.apart && !im ? m[e].real() : m[e].imag(), S);
        M.nim[e] = host_fx(-m[e].imag(), S);
        M.m[e] = make_double2(m[e].real(), m[e].imag());
    }
    M.shift = -1025 - S;
    return true;
}

}  // namespace qsim_fx
