// 64-bit block fixed point: the arithmetic of the FP64 ansatz passes.
//
// GB300 issues one FP64 multiply-add per 64 clocks and warp scheduler, against
// one 32 x 32 + 64-bit integer multiply-add per 4.  A multiply-add of 64-bit
// integers by a constant costs three of those and four cheap instructions: 15
// clocks measured (a stand-alone loop of butterflies, eight to twelve warps per
// scheduler), 4.2 times the rate of DFMA.  So a tile pass turns its tile into
// integers V = x * 2^-E with one exponent E per tile and state, applies the
// gates to the integers and turns the result back into doubles.
//
// Range.  E is chosen from the 2-norm of the tile, which no gate changes:
// |V|_2 <= 2^61 at the start of a pass.  A butterfly without its scale lets
// the norm grow; when the growth since the last shift reaches a factor of two
// (forward; 2^0.75 backward) all values are shifted right by one, and the
// slot's diagonal table carries the power of two back.  So |V|_2 stays below
// 2^62.7 and every component below 2^63, for any input.
//
// Accuracy.  One operation adds an error of about half a unit, and the
// root-mean-square component of a tile of 2^11 amplitudes has 54 bits or more
// above the unit, so the error per operation is below a double's rounding of
// a component of that size (2^-54.3 root mean square); it is relative to the
// tile's norm rather than to the single amplitude.
//
// Spread.  So the integers serve tiles whose amplitudes are of one order, as those
// of a circuit of generic angles are.  Where the angles of a qubit are all small (or
// all near multiples of pi, the same up to exchanges), amplitudes with the qubit
// turned are smaller by about tan of its largest half angle (taken from the nearest
// multiple of pi/2): the product over a tile's qubits is how far the tile's smallest
// amplitudes lie below its largest.  FP64 arithmetic keeps each of those to its own
// precision.  A pass whose tiles spread over more than 2^kFxMaxSpread therefore runs
// in FP64, decided per state at staging.
//
// Error of single amplitudes, relative to each, in FP64 / fixed point (12 qubits,
// medians over three circuits): uniform angles, depth 8 (spread 2^2.5) median 1.0e-15
// / 7.9e-16, 99th percentile 7.9e-15 / 6.7e-15; depth 3 (2^7.6) 7.1e-16 / 7.2e-16 and
// 6.0e-15 / 1.5e-14; depth 2 (2^11) 4.7e-16 / 9.5e-16 and 5.8e-15 / 6.6e-14; normal
// angles of deviation 0.3, depth 4 (2^27) 9.2e-16 / 3.4e-14 and 1.4e-14 / 5.5e-11;
// 0.01 (2^86) 6.4e-16 / 1.8e-5.  The medians meet at about 2^8.
#pragma once

#include <cstddef>
#include <cstdint>

namespace vqe {

// Coefficient of one gated tile bit for the fixed-point passes.  With
// alpha = theta/2,
//     RY(theta) = J^q * 45^o * cos(beta) * [[1, -t], [t, 1]],   t = tan(beta),
// J = [[0, -1], [1, 0]] (a quarter turn), 45^o the turn by pi/4 (o = 0 or 1),
// alpha = q pi/2 + o pi/4 + beta and |beta| <= pi/8, so |t| < 0.4143 fits a
// signed 64-bit fraction T = t 2^64.  A quarter turn exchanges the two
// amplitudes of a pair: an odd q is kept as a flip of the tile bit (the
// amplitude of logical index l sits at l ^ F, F the flips so far), its sign in
// the diagonal table, so that no amplitude moves.  The turn by 45 degrees is
// done as (x - y, x + y), its scale 1/sqrt(2) in the table like cos(beta).
struct RotFx {
    int th, tl;      // T = th 2^32 + tl, both signed
    uint32_t meta;   // FX_* bits
    int wide;        // 0
    double gs;       // 1 / (scale of the buffers when this bit's theta gradient is taken)^2
                     // / 8: the partials have three fraction bits
};

// The same row of a pass that stays in FP64 (see kFxMaxSpread).
struct RotWide {
    double v;        // v, mode and gs as in RotCoef<double>
    int mode;
    int wide = 1;
    double gs;
};
static_assert(sizeof(RotFx) == sizeof(RotWide) && offsetof(RotFx, wide) == offsetof(RotWide, wide),
              "either row tells what it is");

constexpr uint32_t kFxFlip = 1u;      // q is odd
constexpr uint32_t kFx45 = 2u;        // o = 1
constexpr uint32_t kFxBad = 4u;       // an angle of this qubit is not finite
constexpr uint32_t kFxHalf = 8u;      // the slot's table holds d 2^62 (entries of modulus near 1)
constexpr int kFxShiftF = 4;          // bits 4-5: shift after the gate, forward
constexpr int kFxShiftB = 6;          // bits 6-7: shift after the gate, backward
constexpr int kFxSlotShift = 8;       // bits 8-15: the slot's power of two in its table

constexpr int kFxNormBits = 61;       // |V|_2 <= 2^61 when a tile is loaded
constexpr float kFxMaxSpread = 8.f;   // bits between a tile's largest and smallest amplitudes

#ifdef __CUDACC__

__device__ __forceinline__ int fx_lo(long long v) { return (int)v; }
// High half for a signed low half: v = hi 2^32 + lo with lo in [-2^31, 2^31).
__device__ __forceinline__ int fx_hi(long long v) {
    int h;
    asm("{\n"
        ".reg .b32 l, t;\n"
        "mov.b64 {l, %0}, %1;\n"
        "shr.u32 t, l, 31;\n"
        "add.s32 %0, %0, t;\n"
        "}"
        : "=r"(h)
        : "l"(v));
    return h;
}

__device__ __forceinline__ long long fx_madw(int a, int b, long long c) {
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}

__device__ __forceinline__ void fx_acc(long long &c, int a, int b) {
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(c) : "r"(a), "r"(b));
}

// a + T b / 2^64, T = th 2^32 + tl and b = bh 2^32 + bl in signed halves.  The
// two cross products are added exactly (|T| < 2^62.8, |b| < 2^63, so their sum
// fits 64 bits) and cut at 2^32; tl bl (below half a unit) is left out.  A
// rounding constant in the first product costs two more instructions.
__device__ __forceinline__ long long fx_ma(long long a, int th, int tl, int bh, int bl) {
    long long r;
    asm("{\n"
        ".reg .s64 m, x, y;\n"
        ".reg .s32 h, t;\n"
        "mul.wide.s32 m, %1, %4;\n"
        "mad.wide.s32 m, %2, %3, m;\n"
        "mad.wide.s32 x, %1, %3, %5;\n"
        "mov.b64 {t, h}, m;\n"
        "cvt.s64.s32 y, h;\n"
        "add.s64 %0, x, y;\n"
        "}"
        : "=l"(r)
        : "r"(th), "r"(tl), "r"(bh), "r"(bl), "l"(a));
    return r;
}

// (x dr + y di) / 2^63: one component of the product of (x, y) with a table
// entry d 2^-63.  With |(x, y)| <= 2^(61 + A), |d| = 2^(63 - A) and 0 <= A <= 1
// the cross products sum to at most 2^62.9; xl dl is left out.
__device__ __forceinline__ long long fx_dot(int xh, int xl, int drh, int drl, int yh, int yl,
                                            int dih, int dil) {
    long long m = fx_madw(xh, drl, 0ll);
    m = fx_madw(xl, drh, m);
    m = fx_madw(yh, dil, m);
    m = fx_madw(yl, dih, m);
    long long h = fx_madw(xh, drh, 0ll);
    h = fx_madw(yh, dih, h);
    return (h << 1) + (m >> 31);
}

// a b - c d for values of norm at most 2^61, as h 2^64 + m 2^35 (to about one
// unit of 2^35; |m| <= 2^59).
struct FxWide {
    long long h, m;
};
__device__ __forceinline__ FxWide fx_cross(int ah, int al, int bh, int bl, int ch, int cl, int dh,
                                           int dl) {
    const long long m1 = fx_madw(al, bh, fx_madw(ah, bl, (long long)__mulhi(al, bl)));
    const long long m2 = fx_madw(cl, dh, fx_madw(ch, dl, (long long)__mulhi(cl, dl)));
    return FxWide{fx_madw(ah, bh, 0ll) - fx_madw(ch, dh, 0ll), (m1 - m2) >> 3};
}

// Doubles (as bits) to integers x 2^-E and back.  The exponent is moved by
// integer adds; the conversions themselves are two FP64-pipe instructions, a
// pipe that is otherwise idle here (in integer instructions alone a
// conversion takes about 25 of the issue-bound kind each way).  For
// -1020 < E < 0, the largest exponent of the tile being E + 1084 at most.
__device__ __forceinline__ bool fx_plain_exponent(int E) { return E > -960 && E < 0; }
__device__ __forceinline__ long long fx_from_bits(long long bits, int E) {
    // a zero becomes 2^(-E - 1023), far below the unit
    const int hi = (int)(bits >> 32) - E * (1 << 20);
    return __double2ll_rn(__hiloint2double(hi, (int)bits));
}
__device__ __forceinline__ long long fx_to_bits(long long v, int E) {
    const double d = __ll2double_rn(v);
    const int hi = __double2hiint(d);
    return __double_as_longlong(
        __hiloint2double(hi == 0 ? 0 : hi + E * (1 << 20), __double2loint(d)));
}
// Any E (denormal results are rounded twice).
__device__ __forceinline__ long long fx_from_bits_any(long long bits, int E) {
    const double x = __longlong_as_double(bits);
    const int h = -E / 2;
    return __double2ll_rn(ldexp(ldexp(x, h), -E - h));
}
__device__ __forceinline__ long long fx_to_bits_any(long long v, int E) {
    return __double_as_longlong(ldexp((double)v, E));
}

#endif

}  // namespace vqe
