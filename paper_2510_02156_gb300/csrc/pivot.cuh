// pivot.cuh -- the correctly rounded square root of a pivot and quotients by it.
//
// GB300's FP64 square root and division take 611 and 581 cycles where a
// multiply-add takes 64, and every column of a factor waits for one of each.
// Here one approximation of 1 / sqrt(d) serves both, and fused remainders round
// them (P. W. Markstein, IBM J. Res. Dev. 34, 1990): eight operations to the root, five
// more to the quotient.
//
// Bounds (u = 2^-53; relative errors; the hardware's approximation of the
// reciprocal square root is good to 20 bits):
//   y = pivot_recip(d): one third-order step, the first terms of
//     (1 - e)^(-1/2) = 1 + e / 2 + 3 e^2 / 8 + ... for e = 1 - d y0^2.  d y0 is rounded
//     before e is formed, which puts u / 2 on y; with y's own rounding and 5 e^3 / 16
//     it is within 1.6 u of 1 / sqrt(d), up to one unit in the last place.
//   l = pivot_root(d, y): s = d y is within 2.6 u of the root, s + (d - s^2) y / 2 before
//     its rounding within 10 u^2, the rounding of d - s^2 included.  Of the d whose
//     root is that near to the middle between two numbers (finitely many: an odd
//     square within a few units of a multiple of 2^54 or 2^55), every one gives
//     RN(sqrt(d)) with every y inside its bound.
//   rl = reciprocal(l, y): |l y - 1| <= 2.6 u, so one Newton step is within 9 u^2
//     before its rounding: rl lies within (1/2 + 2^-49) units of 1 / l.  (It is not
//     always RN(1 / l): 17 mantissas of l can give its neighbour.)
//   quotients: the remainder r = v - q l of a q within one unit of v / l is exact, and
//     q + r rl differs from v / l by |q - v / l| times the error of rl.  With L the
//     53-bit mantissa of l as an integer, v / l is at least 1 / (2 L) units away from the middle
//     between two numbers and, next to one, q is half a unit away from it; so the rounding of
//     q + r rl is that of v / l while L^2 (1 + 2^-48) < 2^106.  divisor_ok keeps the
//     mantissas closest to all ones, where that fails, out.
//     So q = v rl (pivot_div): within 1.5 units, next to a middle within half.  (v y, which
//     need not wait for l, is up to three units away, and its remainder not exact.  A
//     warp issues an FP64 instruction every 64 cycles whatever depends on what, so
//     the wait costs nothing: 313 against 312 us at order 256, and 329 with a second
//     correction behind v y.)
// root_ok, divisor_ok and the test of v's exponent keep every intermediate
// normal; other operands take sqrt and the division themselves.
#pragma once

namespace rorbk {

// Comparisons with zero on the integer side: an FP64 comparison occupies the FP64
// unit for as long as a multiply-add.  (The halves are taken apart in PTX: with
// the test written on the 64-bit pattern in C++ the trailing update measured
// three times as long.)
__device__ __forceinline__ int2 halves(double v) {
    int2 h;
#ifdef __CUDA_ARCH__
    asm("mov.b64 {%0, %1}, %2;" : "=r"(h.x), "=r"(h.y) : "d"(v));
#else
    __builtin_memcpy(&h, &v, 8);
#endif
    return h;
}
__device__ __forceinline__ bool nonzero(double v) {
    const int2 h = halves(v);
    return ((h.y & 0x7fffffff) | h.x) != 0;
}
__device__ __forceinline__ bool positive(double v) {     // v > 0 (false for NaN)
    const int2 h = halves(v);
    return h.y >= 0 && (h.y | h.x) != 0 && (h.y < 0x7ff00000 || (h.y == 0x7ff00000 && h.x == 0));
}
// g - la lb.  The definition skips a zero factor; adding its zero product
// changes nothing but the sign of a zero.  (A factor that is not finite makes
// its own row's pivot not positive either way.)
__device__ __forceinline__ double sub_prod(double g, double la, double lb) { return __fma_rn(-la, lb, g); }

__device__ __forceinline__ unsigned exponent(double v) { return ((unsigned)halves(v).y >> 20) & 0x7ffu; }
__device__ __forceinline__ bool root_ok(double d) { return exponent(d) - 423u <= 1200u; }
__device__ __forceinline__ double refine_recip(double d, double y0) {
    const double e = __fma_rn(-__dmul_rn(d, y0), y0, 1.0);
    return __fma_rn(__fma_rn(0.375, e, 0.5), __dmul_rn(e, y0), y0);
}
#ifdef __CUDACC__
__device__ __forceinline__ double pivot_recip(double d) {
    double y0;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y0) : "d"(d));
    return refine_recip(d, y0);
}
#endif
__device__ __forceinline__ double pivot_root(double d, double y) {
    const double s = __dmul_rn(d, y);
    const double h = __hiloint2double(halves(y).y - (1 << 20), halves(y).x);   // y / 2 (y is normal)
    return __fma_rn(__fma_rn(-s, s, d), h, s);
}
__device__ __noinline__ double slow_root(double d) { return sqrt(d); }
__device__ __noinline__ double slow_div(double v, double l) { return v / l; }
__device__ __forceinline__ double reciprocal(double l, double y) {
    return __fma_rn(y, __fma_rn(-l, y, 1.0), y);
}
// |exponent| <= 300, and not one of the 32 mantissas up to all ones
__device__ __forceinline__ bool divisor_ok(double l) {
    const int2 h = halves(l);
    return exponent(l) - 723u <= 600u && ((h.y & 0xfffff) != 0xfffff || (unsigned)h.x < 0xffffffe0u);
}
__device__ __forceinline__ bool quotient_ok(double v, bool ok) { return ok & (exponent(v) - 423u <= 1200u || !nonzero(v)); }
// RN(v / l) from a q0 within 1.5 units (within half a unit next to a middle).
__device__ __forceinline__ double quotient_rn(double v, double q0, double l, double rl, bool ok) {
    double q = __fma_rn(__fma_rn(-q0, l, v), rl, q0);
    if (!quotient_ok(v, ok)) q = slow_div(v, l);
    return q;
}

// A pivot d > 0: l = RN(sqrt(d)), rl next to 1 / l, and y ~ 1 / sqrt(d).
struct Pivot {
    double l, rl, y;
    bool ok;
};
__device__ __forceinline__ Pivot pivot_from(double d, double y, bool in) {
    Pivot p;
    p.y = y;
    p.l = in ? pivot_root(d, y) : slow_root(d);
    p.rl = reciprocal(p.l, y);
    p.ok = divisor_ok(p.l);
    return p;
}
#ifdef __CUDACC__
__device__ __forceinline__ Pivot pivot(double d) {
    const bool in = root_ok(d);
    return pivot_from(d, in ? pivot_recip(d) : 1.0 / slow_root(d), in);
}
#endif
__device__ __forceinline__ double pivot_div(double v, const Pivot &p) {      // RN(v / l)
    return quotient_rn(v, __dmul_rn(v, p.rl), p.l, p.rl, p.ok);
}

}  // namespace rorbk
