// k_fx.cuh -- complex128 pair updates evaluated in 60-bit fixed point on the integer pipe.
//
// Why: this GPU issues 2 float64 operations per SM and clock (1.25 TFLOP/s), 1/64 of its float32
// and 1/32 of its 32-bit multiply-add rate, so the 16 float64 instructions of a general 2x2
// update (Section III, Eq. 2) take 8 SM clocks per pair while memory delivers a pair in 2.7.
// The update is a 4x4 real matrix times four numbers, and a product of two 60-bit integers needs
// three 32x32 -> 64-bit multiply-adds (below): 48 for the whole pair, on a pipe that is idle.
//
// How: numbers that share a scale, a power of two, become integers X with |X| < 2^60 in two signed
// 30-bit limbs X = xh 2^30 + xl; the matrix entries likewise on the host, A = ah 2^30 + al. Then
//     A X / 2^60 = ah xh + (ah xl + al xh) / 2^30 + al xl / 2^60,
// where the last term is below one unit of the result and is left out; the products of one output
// are summed exactly in 64 bits (at most eight middle terms below 2^60 each, so no overflow), converted to
// float64 with one rounding and scaled back by an integer addition to the exponent.
//
// Error: it must not exceed float64's for any part of any output, whose scale is S, the sum of its four
// real products' magnitudes (not the size of the pair: a phase of 1e-9, or an amplitude's imaginary part
// far below its real one, is to keep its digits). A number with a scale of its own is exact (53 bits);
// one that shares a larger scale is cut at 2^-60 of that.
//   FX_GEN:  one scale for x and y, one for the entries: the cuts, the products al xl and the shift of
//            the middle sum lose at most 9 units of 2^-60 of the two scales' product W. Where every part of the
//            matrix has at least 2^-4 of the largest one's exponent (three in four Haar matrices), the
//            largest part of the pair meets one of those in every output: S >= 2^-6 W, loss <= 2^-50.8 S.
//   FX_GENP: every part of x, y and the matrix has its own scale, and the four products of an output are
//            aligned before the sum: at most 12 units of 2^-58 S. Where three parts of each row are
//            within 2^-2 of the largest, a pair whose outputs all have S >= 2^-6 W takes FX_GEN's arithmetic.
//            [real imag; imag real] (rotations about X): two real updates, as FX_REAL.
//   FX_REAL: as FX_GENP on real numbers; real and imaginary parts never meet.
//   FX_DIAG, FX_SIDE: a complex product per amplitude, with one scale for x and one for an entry whose
//            parts are within 1/8 of each other (S >= 2^-5 W, loss <= 2^-52.7 S), else as a real update of
//            (re x, im x) by [re -im; im re], every part with its own scale.
// Amplitudes whose exponent leaves no room (infinities, NaN, below 2^-767 or above 2^766) and
// matrices outside the rules of make_fx take the float64 form, per pair, in the same kernel;
// pairs of zeros are left as they are.
//
// Measured against extended precision, worst and root mean square of error / S over all parts, this and
// float64: Haar 1.3e-16, 3.1e-17 (3.3e-16, 5.0e-17); amplitudes' parts spread over 2^-20: 1.8e-16, 4.2e-17
// (3.9e-16, 6.5e-17); phases of 1e-9 to 0.1 1.1e-16, 3.2e-17 (2.1e-16, 3.4e-17); RX 1.1e-16 (2.2e-16),
// RY 1.1e-16 (2.2e-16), RZ RY 1.2e-16 (3.8e-16).
//
// Measured, uncontrolled gate at n = 28 on target 14 (8.6 GB moved, a copy of the same bytes 1.35 ms;
// float64 form: general 4.3 ms, diagonal 2.2, one-sided 1.1): FX_GEN 1.41 ms, FX_GENP 1.87, with the
// one-scale test on random amplitudes 1.44, RX 1.46; real 1.36; diagonal 1.43 (own scales 1.43);
// one-sided 0.67 (own scales 0.70). FX_GENP has 16 shifts of 64 bits more than FX_GEN.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "qs_internal.cuh"

namespace qs {

enum FxForm : int { FX_GEN = 0, FX_GENP = 1, FX_REAL = 2, FX_DIAG = 3, FX_SIDE = 4 };

// The matrix of an update in limbs: part i (real or imaginary, row-major) = (h[i], l[i]) * 2^(e[i] - 60).
// span: exponents of amplitudes that take the fixed-point form, 0 = none (float64 form).
struct FxMat {
    int32_t h[8], l[8];
    int32_t e[8];
    int32_t gh[8], gl[8], ge;  // general update: the same at one scale, 2^(ge - 60)
    uint32_t span;
    int32_t form;
    int32_t parts;    // FX_DIAG, FX_SIDE: every part has a scale of its own; FX_GENP: [real imag; imag real]
    int32_t checked;  // FX_GENP: pairs that one scale serves take FX_GEN's arithmetic
};

constexpr int kFxLow = 256;        // smallest biased exponent of a pair's larger number
constexpr int kFxZero = 64;         // smallest scale of the other one: shifts a zero's implicit bit out
constexpr uint32_t kFxSpan = 1534;  // exponents kFxLow .. kFxLow + kFxSpan - 1
constexpr int kFxBelow = 4;         // one scale: binary orders of an output's largest product below the scales' product
constexpr int kFxNone = -4096;      // scale of a part that is zero: below every other

// Form and limbs of `U` (row-major [a b; c d]; one-sided: U[0..1] only) for the operation class
// `op`. span = 0 (the float64 form) where that one is exact or a part is out of range:
//  - a diagonal entry without real or without imaginary part (Z, S, ...): float64 multiplies
//    exactly or once rounded;
//  - a general or real matrix with a zero entry (Y and other permutations with phases): the same;
//  - a part that is not zero outside 2^-48 .. 2^48 (what a scale of kFxZero cuts off is then below
//    2^-96 of the other product).
// The lines between the forms: a line of 2^-4 (kFxBelow) instead of 2^-3 keeps three in four Haar matrices
// on FX_GEN instead of one in four, and its loss, rare and at worst 2^-50.8 S, stays below float64's in the
// mean; third >= 2^-2: with 2^-3, matrices RZ RY of small angles on states with parts of unlike size took both
// forms in turn (n = 20, 8-layer gradient 6.12 ms, with 2^-2 5.93).
inline void fx_limbs(double v, int e, int32_t *h, int32_t *l) {
    const int64_t a = (int64_t)std::nearbyint(std::ldexp(v, 60 - e));
    const int64_t m = a < 0 ? -a : a;
    *h = (int32_t)(m >> 30) * (a < 0 ? -1 : 1);
    *l = (int32_t)(m & ((1 << 30) - 1)) * (a < 0 ? -1 : 1);
}

inline void make_fx(const double *U, int op, FxMat *f) {
    *f = FxMat{};
    if (op == OP_SWAP) return;  // no arithmetic
    f->form = op == OP_REAL ? FX_REAL : op == OP_DIAG ? FX_DIAG : op == OP_SIDE ? FX_SIDE : FX_GEN;
    const int last = op == OP_SIDE ? 1 : 4;
    bool ok = true, alike = true;  // alike: no part below 1/8 of its partner
    double mx = 0.0;
    f->ge = kFxNone;
    for (int q = 0; q < last; ++q) {
        const double re = std::fabs(U[2 * q]), im = std::fabs(U[2 * q + 1]);
        f->e[2 * q] = f->e[2 * q + 1] = kFxNone;
        if (op == OP_DIAG && (q == 1 || q == 2)) continue;
        for (int i = 2 * q; i < 2 * q + 2; ++i) {
            if (U[i] == 0.0) continue;
            std::frexp(U[i], &f->e[i]);
            if (f->e[i] < -48 || f->e[i] > 48) ok = false;
            f->ge = std::max(f->ge, f->e[i]);
        }
        if ((op == OP_DIAG || op == OP_SIDE) && (re == 0.0 || im == 0.0)) ok = false;
        if ((op == OP_GEN || op == OP_REAL) && re == 0.0 && im == 0.0) ok = false;
        if (std::fmin(re, im) * 8.0 < std::fmax(re, im)) alike = false;
        mx = std::fmax(mx, std::fmax(re, im));
    }
    if (!ok) return;
    if (op == OP_GEN) {
        int least = 4096, third = 4096;  // exponents: the smallest part, the third largest of a row
        for (int row = 0; row < 2; ++row) {
            int r[4];
            std::copy(f->e + 4 * row, f->e + 4 * row + 4, r);
            std::sort(r, r + 4);
            least = std::min(least, r[0]);
            third = std::min(third, r[1]);
        }
        if (least < f->ge - kFxBelow) f->form = FX_GENP;
        f->checked = third >= f->ge - 2;
        f->parts = U[1] == 0.0 && U[2] == 0.0 && U[4] == 0.0 && U[7] == 0.0;
    } else if (op == OP_DIAG || op == OP_SIDE) {
        f->parts = !alike;
        if (alike)  // one scale for each entry
            for (int i = 0; i < 2 * last; i += 2) f->e[i] = f->e[i + 1] = std::max(f->e[i], f->e[i + 1]);
    }
    for (int i = 0; i < 2 * last; ++i) {
        if (U[i] == 0.0) continue;
        fx_limbs(U[i], f->e[i], &f->h[i], &f->l[i]);
        if (op == OP_GEN) fx_limbs(U[i], f->ge, &f->gh[i], &f->gl[i]);
    }
    f->span = kFxSpan;
}

// The same for a matrix given in full, its class read from its entries (masked comparator): the
// class plan_gate finds, so that both schedules run the same arithmetic. *side: FX_SIDE's side.
inline void make_fx_full(const double U[8], FxMat *f, int *side) {
    const bool offd = U[2] == 0.0 && U[3] == 0.0 && U[4] == 0.0 && U[5] == 0.0;
    *side = 0;
    if (offd && U[0] == 1.0 && U[1] == 0.0) {
        *side = 1;
        make_fx(U + 6, OP_SIDE, f);
    } else if (offd && U[6] == 1.0 && U[7] == 0.0) {
        make_fx(U, OP_SIDE, f);
    } else if (offd) {
        make_fx(U, OP_DIAG, f);
    } else if (U[1] == 0.0 && U[3] == 0.0 && U[5] == 0.0 && U[7] == 0.0) {
        make_fx(U, OP_REAL, f);
    } else {
        make_fx(U, OP_GEN, f);
    }
}

namespace fx {

__device__ __forceinline__ int abs_hi(double v) { return __double2hiint(v) & 0x7fffffff; }

__device__ __forceinline__ bool nonzero(double v) { return (__double2hiint(v) | __double2loint(v)) != 0; }

// Limbs of v in units of 2^(E - 1082), E the biased exponent of the scale (E >= v's own). The
// implicit bit of a zero or subnormal is shifted out, because E >= kFxZero.
__device__ __forceinline__ void limbs(double v, int E, int &h, int &l) {
    const int hi = __double2hiint(v);
    const int d = E - ((hi & 0x7fffffff) >> 20);
    unsigned long long m = ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(v);
    m <<= 9;  // the leading bit at bit 61: the high word is the high limb, the low word 4 * low limb
    asm("shr.b64 %0, %0, %1;" : "+l"(m) : "r"(d));  // (amounts above 63 give 0)
    const int sg = (hi >> 31) | 1;
    h = (int)(m >> 32) * sg;
    l = (int)((unsigned)m >> 2) * sg;
}

__device__ __forceinline__ long long mad(int a, int b, long long c) { return (long long)a * b + c; }

// s >> d for d >= 0 (amounts above 63 leave the sign).
__device__ __forceinline__ long long sar(long long s, int d) {
    asm("shr.s64 %0, %0, %1;" : "+l"(s) : "r"(d));
    return s;
}

// s * 2^sc as float64, one rounding (s = 0 or the result is a normal number by kFxLow, kFxSpan).
__device__ __forceinline__ double to_f64(long long s, int sc) {
    const double d = __ll2double_rn(s);
    return __hiloint2double(s ? __double2hiint(d) + (sc << 20) : 0, __double2loint(d));
}

// The same on the integer pipe (18 operations; ties away from zero), for forms whose conversions would
// fill the FP64 pipe: a real update of psi and lambda with its derivative product, 2^23 pairs each:
// all by conversion 206 us, half by integers 184, all by integers 207 (160 of memory time).
__device__ __forceinline__ double to_f64_int(long long s, int sc) {
    const long long sg = s >> 63;
    unsigned long long u = (unsigned long long)((s ^ sg) - sg);
    const unsigned uh = (unsigned)(u >> 32);
    const int lz = uh ? __clz((int)uh) : 32 + __clz((int)u);
    asm("shl.b64 %0, %0, %1;" : "+l"(u) : "r"(lz));
    // the leading bit at bit 52, added to the exponent field below. The rounding bit is added after the
    // shift: before it the sum passes 64 bits for results just below a power of two (here it becomes 2^53,
    // whose carry the exponent field takes).
    u = (u >> 11) + ((u >> 10) & 1);
    const unsigned hi = (unsigned)(u >> 32) + ((unsigned)(1023 + 62 - lz + sc) << 20);
    return __hiloint2double(s ? (int)(hi | ((unsigned)sg & 0x80000000u)) : 0, (int)(unsigned)u);
}

// Two-limb products (A X + B Y) / 2^60 and A X / 2^60.
__device__ __forceinline__ long long dot1(int ah, int al, int xh, int xl) {
    return mad(ah, xh, mad(al, xh, (long long)ah * xl) >> 30);
}
__device__ __forceinline__ long long dot2(int ah, int al, int xh, int xl, int bh, int bl, int yh, int yl) {
    long long m = (long long)ah * xl;
    m = mad(al, xh, m);
    m = mad(bh, yl, m);
    m = mad(bl, yh, m);
    return mad(bh, yh, mad(ah, xh, m >> 30));
}
__device__ __forceinline__ long long dot4(const int *h, const int *l, int i, int j, int sgn_j, const int *xh,
                                          const int *xl) {
    // entries i, i + 2 times parts 0, 2 plus entries j, j + 2 (times sgn_j) times parts 1, 3
    long long m = (long long)h[i] * xl[0];
    m = mad(l[i], xh[0], m);
    m = mad(sgn_j * h[j], xl[1], m);
    m = mad(sgn_j * l[j], xh[1], m);
    m = mad(h[i + 2], xl[2], m);
    m = mad(l[i + 2], xh[2], m);
    m = mad(sgn_j * h[j + 2], xl[3], m);
    m = mad(sgn_j * l[j + 2], xh[3], m);
    long long s = m >> 30;
    s = mad(h[i], xh[0], s);
    s = mad(sgn_j * h[j], xh[1], s);
    s = mad(h[i + 2], xh[2], s);
    return mad(sgn_j * h[j + 2], xh[3], s);
}

__device__ __forceinline__ bool in_range(int E, const FxMat &f) { return (unsigned)(E - kFxLow) < f.span; }

// General update, one scale for x and y and one for the matrix. False: out of range (x, y kept).
__device__ __forceinline__ bool gen(double2 &x, double2 &y, const FxMat &f) {
    const int E = max(max(abs_hi(x.x), abs_hi(x.y)), max(abs_hi(y.x), abs_hi(y.y))) >> 20;
    if (!in_range(E, f)) return false;
    int vh[4], vl[4];
    limbs(x.x, E, vh[0], vl[0]);
    limbs(x.y, E, vh[1], vl[1]);
    limbs(y.x, E, vh[2], vl[2]);
    limbs(y.y, E, vh[3], vl[3]);
    const int sc = E - 1082 + f.ge;
    x.x = to_f64(dot4(f.gh, f.gl, 0, 1, -1, vh, vl), sc);
    x.y = to_f64(dot4(f.gh, f.gl, 1, 0, 1, vh, vl), sc);
    y.x = to_f64(dot4(f.gh, f.gl, 4, 5, -1, vh, vl), sc);
    y.y = to_f64(dot4(f.gh, f.gl, 5, 4, 1, vh, vl), sc);
    return true;
}

// Which part of the matrix meets part i of (x, y) in output r (re x', im x', re y', im y').
__device__ __forceinline__ constexpr int part_at(int r, int i) { return 4 * (r >> 1) + 2 * (i >> 1) + ((r ^ i) & 1); }

// Whether one scale serves the pair: every output has a product within 2^kFxBelow of the scales' product.
__device__ __forceinline__ bool one_scale(const double2 &x, const double2 &y, const FxMat &f) {
    const int ex[4] = {abs_hi(x.x) >> 20, abs_hi(x.y) >> 20, abs_hi(y.x) >> 20, abs_hi(y.y) >> 20};
    int least = 0x7fffffff;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        int m = f.e[part_at(r, 0)] + ex[0];
#pragma unroll
        for (int i = 1; i < 4; ++i) m = __viaddmax_s32(f.e[part_at(r, i)], ex[i], m);
        least = min(least, m);
    }
    return least >= f.ge + max(max(ex[0], ex[1]), max(ex[2], ex[3])) - kFxBelow;
}

// Real 2x2 [A B; C D] (parts i0 .. i3 of the matrix, B negated where NEG) on two real numbers; INT: one
// of the two conversions on the integer pipe.
template <bool NEG, bool INT>
__device__ __forceinline__ bool real2(double &x, double &y, const FxMat &f, int i0, int i1, int i2, int i3) {
    int ex = abs_hi(x) >> 20, ey = abs_hi(y) >> 20;
    if (!in_range(max(ex, ey), f)) return false;
    ex = max(ex, kFxZero);
    ey = max(ey, kFxZero);
    int xh, xl, yh, yl;
    limbs(x, ex, xh, xl);
    limbs(y, ey, yh, yl);
    double o[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int i = r ? i2 : i0, j = r ? i3 : i1;
        const bool neg = NEG && r == 0;
        const int e1 = ex + f.e[i], e2 = ey + f.e[j], F = max(e1, e2);
        const long long p = sar(dot1(f.h[i], f.l[i], xh, xl), F - e1), q = sar(dot1(f.h[j], f.l[j], yh, yl), F - e2);
        const long long s = neg ? p - q : p + q;
        o[r] = INT && r == 0 ? to_f64_int(s, F - 1082) : to_f64(s, F - 1082);
    }
    x = o[0];
    y = o[1];
    return true;
}

// General update, own scales of all parts of x, y and the entries. A part of x or y that is neither zero
// nor in range sends the pair to float64: with a zero part in the matrix no larger product covers it.
// [real imag; imag real] is two real updates, of (re x, im y) and (re y, im x).
__device__ __forceinline__ bool genp(double2 &x, double2 &y, const FxMat &f) {
    if (f.parts) {
        double2 p = make_double2(x.x, y.y), q = make_double2(y.x, x.y);
        const bool zp = !(nonzero(p.x) || nonzero(p.y)), zq = !(nonzero(q.x) || nonzero(q.y));
        if (!(zp || real2<true, true>(p.x, p.y, f, 0, 3, 5, 6)) || !(zq || real2<true, true>(q.x, q.y, f, 6, 5, 3, 0)))
            return false;
        x = make_double2(p.x, q.y);
        y = make_double2(q.x, p.y);
        return true;
    }
    if (f.checked && one_scale(x, y, f)) return gen(x, y, f);
    const double v[4] = {x.x, x.y, y.x, y.y};
    int ex[4], vh[4], vl[4], top = 0;
    unsigned low = 0xffffffffu;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int hi = abs_hi(v[i]);
        top = max(top, hi);
        low = min(low, (unsigned)hi - (__double2loint(v[i]) == 0));  // (a zero: the largest)
        ex[i] = max(hi >> 20, kFxZero);
    }
    if (!in_range(top >> 20, f) || low < (unsigned)kFxLow << 20) return false;
#pragma unroll
    for (int i = 0; i < 4; ++i) limbs(v[i], ex[i], vh[i], vl[i]);
    double o[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {  // re x', im x', re y', im y'
        int F = f.e[part_at(r, 0)] + ex[0];
#pragma unroll
        for (int i = 1; i < 4; ++i) F = __viaddmax_s32(f.e[part_at(r, i)], ex[i], F);
        long long s = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int q = part_at(r, i);
            const long long p = sar(dot1(f.h[q], f.l[q], vh[i], vl[i]), F - f.e[q] - ex[i]);
            s = !(r & 1) && (i & 1) ? s - p : s + p;  // - im im
        }
        o[r] = to_f64(s, F - 1082);
    }
    x.x = o[0];
    x.y = o[1];
    y.x = o[2];
    y.y = o[3];
    return true;
}

// Real 2x2 on one real number of each side.
__device__ __forceinline__ bool real(double &x, double &y, const FxMat &f) { return real2<false, true>(x, y, f, 0, 2, 4, 6); }

// Entry Q times x: one scale for the parts of each, or own scales (re -im; im re on the two parts of x).
template <int Q, bool INT = false>
__device__ __forceinline__ bool mul(double2 &x, const FxMat &f) {
    if (f.parts) return real2<true, INT>(x.x, x.y, f, 2 * Q, 2 * Q + 1, 2 * Q + 1, 2 * Q);
    const int E = max(abs_hi(x.x), abs_hi(x.y)) >> 20;
    if (!in_range(E, f)) return false;
    int rh, rl, ih, il;
    limbs(x.x, E, rh, rl);
    limbs(x.y, E, ih, il);
    const int sc = E - 1082 + f.e[2 * Q];
    x.x = to_f64(dot2(f.h[2 * Q], f.l[2 * Q], rh, rl, -f.h[2 * Q + 1], -f.l[2 * Q + 1], ih, il), sc);
    x.y = to_f64(dot2(f.h[2 * Q + 1], f.l[2 * Q + 1], rh, rl, f.h[2 * Q], f.l[2 * Q], ih, il), sc);
    return true;
}

// Keeps the float64 form behind its branch (the compiler may otherwise compute a short one for every
// pair and select).
__device__ __forceinline__ void rare(double &v) { asm volatile("" : "+d"(v)); }

}  // namespace fx
}  // namespace qs
