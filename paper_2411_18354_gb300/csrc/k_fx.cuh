// k_fx.cuh -- complex128 pair updates evaluated in 60-bit fixed point on the integer pipe.
//
// Why: this GPU issues 2 float64 operations per SM and clock (1.25 TFLOP/s), 1/64 of its float32
// and 1/32 of its 32-bit multiply-add rate, so the 16 float64 instructions of a general 2x2
// update (Section III, Eq. 2) take 8 SM clocks per pair while memory delivers a pair in 2.7.
// The update is a 4x4 real matrix times four numbers, and a product of two 60-bit integers needs
// three 32x32 -> 64-bit multiply-adds (below): 48 for the whole pair, on a pipe that is idle.
//
// How: a complex number (or, for a real matrix, each real number) is scaled by its own power of
// two to an integer X with |X| < 2^60 and split into two signed 30-bit limbs X = xh 2^30 + xl; the
// matrix entries likewise on the host, A = ah 2^30 + al. Then
//     A X / 2^60 = ah xh + (ah xl + al xh) / 2^30 + al xl / 2^60,
// where the last term is below one unit of the result and is left out; the products of one output
// are summed exactly in 64 bits (at most eight middle terms below 2^60 each, so no overflow), converted to
// float64 with one rounding and scaled back by an integer addition to the exponent.
//
// Error: cutting X and A to integers, the product al xl and the shift of the middle sum lose at
// most 7 units of 2^-58 |a||x| (a, x: the largest real or imaginary parts of what shares a scale),
// and the conversion rounds once (2^-53 of the result); the float64 form rounds four times. Measured
// against exact arithmetic, random amplitudes, one Haar gate: 2-norm error 4.7e-17 (float64 form
// 7.1e-17), worst output 3.2e-16 of its modulus (8.9e-15).
//   FX_GEN:  x and y share one scale, as do the four entries. Its error is relative to the larger
//            of |x|, |y| and the largest entry, so it is used where every entry is at least 1/8 of
//            the largest (97 % of Haar matrices): |a||x| + |b||y| is then at least 1/8 of that
//            product, and the worst case, 2^-51.9 of it, no larger than four float64 roundings.
//   FX_GENW: x, y and each entry have their own scale and the two products of an output are
//            aligned before the sum: the bound holds for any entries (7 % slower at n = 27).
//   FX_REAL: as FX_GENW on real numbers; real and imaginary parts never meet.
//   FX_DIAG, FX_SIDE: one complex product per amplitude.
// Amplitudes whose exponent leaves no room (infinities, NaN, below 2^-767 or above 2^766) and
// matrices outside the rules of make_fx take the float64 form, per pair, in the same kernel;
// pairs of zeros are left as they are.
//
// Measured, uncontrolled gate at n = 27 (4.3 GB moved), float64 form -> this: general 2152 -> 677 us
// (a copy of the same bytes: 675), real 1090 -> 703, diagonal 1085 -> 712, one-sided 548 -> 365.
#pragma once

#include <cmath>
#include <cstdint>

#include "qs_internal.cuh"

namespace qs {

enum FxForm : int { FX_GEN = 0, FX_GENW = 1, FX_REAL = 2, FX_DIAG = 3, FX_SIDE = 4 };

// The matrix of an update in limbs: entry q (a, b, c, d) = (limb pairs 2q, 2q + 1) * 2^(e[q] - 60).
// span: exponents of amplitudes that take the fixed-point form, 0 = none (float64 form).
struct FxMat {
    int32_t h[8], l[8];
    int32_t e[4];
    uint32_t span;
    int32_t form;
};

constexpr int kFxLow = 256;        // smallest biased exponent of a pair's larger number
constexpr int kFxZero = 64;         // smallest scale of the other one: shifts a zero's implicit bit out
constexpr uint32_t kFxSpan = 1534;  // exponents kFxLow .. kFxLow + kFxSpan - 1

// Form and limbs of `U` (row-major [a b; c d]; one-sided: U[0..1] only) for the operation class
// `op`. span = 0 (the float64 form) where that one is exact or an entry is out of range:
//  - a diagonal entry without real or without imaginary part (Z, S, ...): float64 multiplies
//    exactly or once rounded, while a common scale would cut a much smaller part;
//  - a general or real matrix with a zero entry (Y and other permutations with phases): the same;
//  - an entry outside 2^-48 .. 2^48 (what a scale of kFxZero cuts off is then below 2^-96 of the
//    other product).
inline void make_fx(const double *U, int op, FxMat *f) {
    *f = FxMat{};
    if (op == OP_SWAP) return;  // no arithmetic
    f->form = op == OP_REAL ? FX_REAL : op == OP_DIAG ? FX_DIAG : op == OP_SIDE ? FX_SIDE : FX_GEN;
    const int first = 0, last = op == OP_SIDE ? 1 : 4;
    int e[4];
    bool ok = true;
    double mx = 0.0, mn = INFINITY;
    for (int q = first; q < last; ++q) {
        const double re = std::fabs(U[2 * q]), im = std::fabs(U[2 * q + 1]), w = std::fmax(re, im);
        e[q] = 0;
        if (w > 0.0) std::frexp(w, &e[q]);
        const bool used = !(op == OP_DIAG && (q == 1 || q == 2));
        if (!used) continue;
        if (w > 0.0 && (e[q] < -48 || e[q] > 48)) ok = false;
        if ((op == OP_DIAG || op == OP_SIDE) && (re == 0.0 || im == 0.0)) ok = false;
        if ((op == OP_GEN || op == OP_REAL) && w == 0.0) ok = false;
        mx = std::fmax(mx, std::hypot(re, im));
        mn = std::fmin(mn, std::hypot(re, im));
    }
    if (!ok) return;
    if (op == OP_GEN) {
        if (mn * 8.0 >= mx) {  // balanced: one scale for the whole matrix
            int em = e[0];
            for (int q = 1; q < 4; ++q) em = e[q] > em ? e[q] : em;
            for (int q = 0; q < 4; ++q) e[q] = em;
        } else {
            f->form = FX_GENW;
        }
    }
    for (int q = first; q < last; ++q) {
        f->e[q] = e[q];
        if (op == OP_DIAG && (q == 1 || q == 2)) continue;
        for (int i = 2 * q; i < 2 * q + 2; ++i) {
            const int64_t a = (int64_t)std::nearbyint(std::ldexp(U[i], 60 - e[q]));
            const int64_t m = a < 0 ? -a : a;
            f->h[i] = (int32_t)(m >> 30) * (a < 0 ? -1 : 1);
            f->l[i] = (int32_t)(m & ((1 << 30) - 1)) * (a < 0 ? -1 : 1);
        }
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
    const int sc = E - 1082 + f.e[0];
    x.x = to_f64(dot4(f.h, f.l, 0, 1, -1, vh, vl), sc);
    x.y = to_f64(dot4(f.h, f.l, 1, 0, 1, vh, vl), sc);
    y.x = to_f64(dot4(f.h, f.l, 4, 5, -1, vh, vl), sc);
    y.y = to_f64(dot4(f.h, f.l, 5, 4, 1, vh, vl), sc);
    return true;
}

// General update, own scales of x, y and the entries.
__device__ __forceinline__ bool genw(double2 &x, double2 &y, const FxMat &f) {
    int ex = max(abs_hi(x.x), abs_hi(x.y)) >> 20, ey = max(abs_hi(y.x), abs_hi(y.y)) >> 20;
    if (!in_range(max(ex, ey), f)) return false;
    ex = max(ex, kFxZero);
    ey = max(ey, kFxZero);
    int xh[2], xl[2], yh[2], yl[2];
    limbs(x.x, ex, xh[0], xl[0]);
    limbs(x.y, ex, xh[1], xl[1]);
    limbs(y.x, ey, yh[0], yl[0]);
    limbs(y.y, ey, yh[1], yl[1]);
    double2 o[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int q = 4 * r;
        const int e1 = ex + f.e[2 * r], e2 = ey + f.e[2 * r + 1], F = max(e1, e2);
        const long long re = sar(dot2(f.h[q], f.l[q], xh[0], xl[0], -f.h[q + 1], -f.l[q + 1], xh[1], xl[1]), F - e1) +
                             sar(dot2(f.h[q + 2], f.l[q + 2], yh[0], yl[0], -f.h[q + 3], -f.l[q + 3], yh[1], yl[1]), F - e2);
        const long long im = sar(dot2(f.h[q + 1], f.l[q + 1], xh[0], xl[0], f.h[q], f.l[q], xh[1], xl[1]), F - e1) +
                             sar(dot2(f.h[q + 3], f.l[q + 3], yh[0], yl[0], f.h[q + 2], f.l[q + 2], yh[1], yl[1]), F - e2);
        o[r].x = to_f64(re, F - 1082);
        o[r].y = to_f64(im, F - 1082);
    }
    x = o[0];
    y = o[1];
    return true;
}

// Real 2x2 on one real number of each side.
__device__ __forceinline__ bool real(double &x, double &y, const FxMat &f) {
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
        const int e1 = ex + f.e[2 * r], e2 = ey + f.e[2 * r + 1], F = max(e1, e2);
        const long long s = sar(dot1(f.h[4 * r], f.l[4 * r], xh, xl), F - e1) +
                            sar(dot1(f.h[4 * r + 2], f.l[4 * r + 2], yh, yl), F - e2);
        o[r] = r ? to_f64(s, F - 1082) : to_f64_int(s, F - 1082);
    }
    x = o[0];
    y = o[1];
    return true;
}

// Entry Q times x.
template <int Q>
__device__ __forceinline__ bool mul(double2 &x, const FxMat &f) {
    const int E = max(abs_hi(x.x), abs_hi(x.y)) >> 20;
    if (!in_range(E, f)) return false;
    int rh, rl, ih, il;
    limbs(x.x, E, rh, rl);
    limbs(x.y, E, ih, il);
    const int sc = E - 1082 + f.e[Q];
    x.x = to_f64(dot2(f.h[2 * Q], f.l[2 * Q], rh, rl, -f.h[2 * Q + 1], -f.l[2 * Q + 1], ih, il), sc);
    x.y = to_f64(dot2(f.h[2 * Q + 1], f.l[2 * Q + 1], rh, rl, f.h[2 * Q], f.l[2 * Q], ih, il), sc);
    return true;
}

// Keeps the float64 form behind its branch (the compiler may otherwise compute a short one for every
// pair and select).
__device__ __forceinline__ void rare(double &v) { asm volatile("" : "+d"(v)); }

__device__ __forceinline__ bool nonzero(double v) { return (__double2hiint(v) | __double2loint(v)) != 0; }

}  // namespace fx
}  // namespace qs
