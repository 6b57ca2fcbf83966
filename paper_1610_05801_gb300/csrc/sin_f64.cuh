// Sines of the FP64 kernels, written for the scarce FP64 pipe of GB300 (2 DFMA per clock per
// SM): on the integer pipe for every phase k z up to ~1e5 (second part of this file), in FP64
// arithmetic beyond and for the sine of a double (sin_f64).
//
// The FP64 form: Cody-Waite argument reduction x = q pi/2 + r (Cody & Waite, "Software Manual
// for the Elementary Functions", 1980), done with fused multiply-adds so a two-part
// pi/2 suffices, then one polynomial on |r| <= pi/4 whose coefficient set (sine or
// cosine) is selected per lane by the quadrant parity:
//     sin r = r + r^3 S(r^2),   cos r = 1 - r^2/2 + r^4 C(r^2),   deg S = deg C = 5,
// fitted by Chebyshev interpolation at 60 digits (gen_sin_coeffs.py; polynomial error
// 2e-17 relative for S, 1.3e-18 for C).  11 FP64 operations per call, no branches and
// no local memory on the path; the quadrant is found in FP32 and the range check on the
// integer pipe.  |x| > 1e5 (far outside any RF bucket) falls back to CUDA's sin().
// Accuracy: a few ulp on |x| <= 1e5 (checked against CUDA's sin and mpmath in the
// tests through phtl_eval_sin).
#pragma once

#include <cuda_runtime.h>

#include "dfloat.cuh"
#include "internal.h"

namespace phtl {
namespace detail {

constexpr double kTwoOverPi = 0.63661977236758134308;
constexpr double kPio2Hi = 1.5707963267948966;      // nearest double to pi/2
constexpr double kPio2Lo = 6.123233995736766e-17;   // pi/2 - kPio2Hi
constexpr float kMagic = 12582912.0f;               // 1.5 * 2^23: rounds to an integer

// sin r = r + r^3 S(r^2), cos r = 1 - r^2/2 + r^4 C(r^2): coefficients of S and C from the
// highest degree down (Chebyshev fits, gen_sin_coeffs.py)
__host__ __device__ constexpr double kS(int i)
{
    return i == 0 ? 1.5918129294866608e-10 : i == 1 ? -2.5051131845003624e-08
         : i == 2 ? 2.755731610255244e-06  : i == 3 ? -0.00019841269836758574
         : i == 4 ? 0.008333333333330948   : -0.16666666666666666;
}
__host__ __device__ constexpr double kC(int i)
{
    return i == 0 ? -1.1382632425521717e-11 : i == 1 ? 2.08761462684032e-09
         : i == 2 ? -2.7557317271729793e-07 : i == 3 ? 2.480158729876569e-05
         : i == 4 ? -0.0013888888888887398  : 0.041666666666666664;
}
constexpr double kTwoPi = 6.283185307179586;

__device__ __forceinline__ double sc_coef(bool odd, double s, double c) { return odd ? c : s; }

// ---- sines on the integer pipe ---------------------------------------------------------
//
// An FP64 instruction takes the FP64 pipe half a clock per lane (2 per clock per SM), as long
// as 64 issue slots of the other pipes, so a kick's sine costs less as ~80 integer
// instructions than as 11 FP64 ones.  The phase is a 64-bit binary fraction (its overflow is
// the reduction modulo 2 pi, and no fold is ever rounded), the sine one unsigned fixed-point
// polynomial
//     sin(pi V) = V p(rho),   rho = (2 V)^2 in [0, 1],   V in [0, 1/2] half turns,
// p of degree 8 (Chebyshev interpolation at 60 digits, gen_sin_coeffs.py --fixed; error 2e-19
// of p): the upper five steps in 64 bits, the three last terms (below 1.2e-7) in 32.  The
// result is normalised and rounded to FP64 once: |error| <= 0.7 2^-53 over the range, where
// the FP64 polynomial has about 1.
//
// The multiplications bound it: a 32 x 32 product, high half or wide, issues at 32 lanes per
// clock per SM (against 64 for shifts and logic, 128 for adds), and there are 26 of them.

// High 64 bits of a 128-bit product, short of it by at most 2 (the low product and the carry
// of the low halves are left out).
__device__ __forceinline__ uint64_t mulhi_trunc(uint64_t a, uint64_t b)
{
    const uint32_t a1 = static_cast<uint32_t>(a >> 32), a0 = static_cast<uint32_t>(a);
    const uint32_t b1 = static_cast<uint32_t>(b >> 32), b0 = static_cast<uint32_t>(b);
    return static_cast<uint64_t>(a1) * b1 + __umulhi(a1, b0) + __umulhi(a0, b1);
}

// The same for a, b < 2^63: the two cross terms add up in 32 bits.
__device__ __forceinline__ uint64_t mulhi_trunc63(uint64_t a, uint64_t b)
{
    const uint32_t a1 = static_cast<uint32_t>(a >> 32), a0 = static_cast<uint32_t>(a);
    const uint32_t b1 = static_cast<uint32_t>(b >> 32), b0 = static_cast<uint32_t>(b);
    return static_cast<uint64_t>(a1) * b1 + (__umulhi(a1, b0) + __umulhi(a0, b1));
}

// 64-bit shifts whose amount saturates (0 for 64 and more), as the hardware's do.
__device__ __forceinline__ uint64_t shr_sat(uint64_t a, uint32_t n)
{
    uint64_t r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(n));
    return r;
}
__device__ __forceinline__ int64_t sar_sat(int64_t a, uint32_t n)  // the sign for 64 and more
{
    int64_t r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(n));
    return r;
}
__device__ __forceinline__ uint64_t shl_sat(uint64_t a, uint32_t n)
{
    uint64_t r;
    asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(n));
    return r;
}

// The significand of a normal double with its leading one at bit 63.
__device__ __forceinline__ uint64_t mantissa64(double x)
{
    const uint32_t hi = static_cast<uint32_t>(__double2hiint(x)), lo = static_cast<uint32_t>(__double2loint(x));
    return (static_cast<uint64_t>(__funnelshift_l(lo, hi, 11) | 0x80000000u) << 32) | (lo << 11);
}

// A phase in half turns (2^-64) folded to [0, 1/2]: sin(pi V) = sin(pi (1 - V)).
__device__ __forceinline__ uint64_t fold_half_turn(uint64_t V)
{
    const uint32_t s = static_cast<uint32_t>(static_cast<int32_t>(V >> 32) >> 31);
    return V ^ (static_cast<uint64_t>(s) << 32 | s);
}

// p(rho) 2^60 of V in [0, 1/2] half turns (2^-64).  rho is kept as 2^62 rho = hi64(V V), so
// each 64-bit Horner step comes down by four in scale: c5 at 2^70, ..., pi at 2^60.
__device__ __forceinline__ uint64_t sin_poly_fixed(uint64_t V)
{
    const uint64_t T = mulhi_trunc63(V, V);
    const uint32_t t = static_cast<uint32_t>(T >> 30);             // rho 2^32
    uint32_t q = 0x02DEF59Bu - __umulhi(t, 0x00067519u);          // c7 and c8 (2^55)
    q = 0xF479B3AFu - __umulhi(t, q);                              // c6
    uint64_t p = 0x001E3074DFAF87AFull - ((static_cast<uint64_t>(t) * q) >> 17);  // c5 (2^70)
    p = 0x015078348551853Bull - mulhi_trunc63(T, p);
    p = 0x09969667313E42F1ull - mulhi_trunc63(T, p);
    p = 0x28CD78CEEB54F91Eull - mulhi_trunc63(T, p);
    p = 0x52AEF39896F94915ull - mulhi_trunc63(T, p);
    return 0x3243F6A8885A308Cull - mulhi_trunc63(T, p);            // pi
}

// S 2^(-60 - x) as a double with the sign bit of `sign`, rounded to nearest (ties up), for
// S >= 2^32.
__device__ __forceinline__ double fixed_to_double(uint64_t S, int x, uint32_t sign)
{
    const int c = __clz(static_cast<int>(S >> 32));
    const uint64_t N = shl_sat(S, static_cast<uint32_t>(c));   // leading one at bit 63
    const uint64_t r = (N >> 11) + ((N >> 10) & 1u);            // the leading one adds 1 to the exponent
    const uint32_t hi = static_cast<uint32_t>(r >> 32) + (static_cast<uint32_t>(1025 - c - x) << 20);
    return __hiloint2double(static_cast<int>(hi | (sign & 0x80000000u)), static_cast<int>(static_cast<uint32_t>(r)));
}

// sin(2 pi U), U in 2^-64 turns, with the sign flipped where bit 31 of `flip` is set: 0 at a zero of
// the sine, fewer significant bits next to one.
__device__ __forceinline__ double sin_turns_any(uint64_t U, uint32_t flip)
{
    const uint64_t V = fold_half_turn(U << 1);
    const uint64_t S = mulhi_trunc63(V, sin_poly_fixed(V));
    const bool low = (S >> 32) == 0u;
    const double r = fixed_to_double(low ? S << 32 : S, low ? 32 : 0, static_cast<uint32_t>(U >> 32) ^ flip);
    return S == 0u ? 0.0 : r;
}

// sin(q pi/2 + r) for |r| <= pi/4 (a hair more when q came out one off), given the low
// bits qi of q.
__device__ __forceinline__ double sin_quadrant(double r, int qi)
{
    const double r2 = r * r;
    const bool odd = (qi & 1) != 0;
    double p = sc_coef(odd, kS(0), kC(0));
#pragma unroll
    for (int i = 1; i < 6; ++i) p = fma(p, r2, sc_coef(odd, kS(i), kC(i)));
    const double m = (odd ? r2 : r) * r2;                 // r^3 or r^4
    const double a = odd ? fma(-0.5, r2, 1.0) : r;        // r or 1 - r^2/2
    const double res = fma(m, p, a);
    // quadrants 2 and 3 flip the sign: an integer XOR of the sign bit, not an FP64 negate
    return __longlong_as_double(__double_as_longlong(res) ^ (static_cast<long long>(qi & 2) << 62));
}

}  // namespace detail

__device__ __forceinline__ double sin_f64(double x)
{
    using namespace detail;
    // |x| >= 1e5 (high word of 1e5 is 0x40f86a00): library sine
    if ((__double2hiint(x) & 0x7fffffff) >= 0x40f86a00) return sin(x);
    // quadrant q = nearest integer to x * 2/pi, found in FP32 from the top 24 bits of x
    // (integer split: no FP64 instruction).  Near a half-integer q may be off by one,
    // which only moves |r| a hair past pi/4, inside the polynomials' accuracy.
    const float xf = split_bits(x).h;
    const float tf = __fmaf_rn(xf, 0.6366197466850281f, kMagic);
    const int qi = __float_as_int(tf);         // q mod 2^22 in the low mantissa bits
    const double q = widen_float_bits(__fsub_rn(tf, kMagic));
    double r = fma(-q, kPio2Hi, x);
    r = fma(-q, kPio2Lo, r);
    return sin_quadrant(r, qi);
}

// The phase k z of up to 2^14 turns (|k z| ~ 1e5) in 2^-64 turns, from the whole product of z's
// significand and k / 2 pi in 127 bits: within 2^-62 turns however many turns there are.  false:
// beyond that, |k z| below 2^-800, or a z that is zero, subnormal, Inf or NaN.
__device__ __forceinline__ bool phase_of_turns(PhaseScale kap, double z, uint64_t& U)
{
    using namespace detail;
    const int e = (__double2hiint(z) >> 20) & 0x7ff;
    const int n = kap.cn - e;
    if (n < -15 || n > 800 || e == 0) return false;
    const uint64_t M = mantissa64(z);
    unsigned __int128 p = static_cast<unsigned __int128>(M) * kap.K;
    p += static_cast<__int128>(__mul64hi(static_cast<long long>(M >> 1), kap.K2)) * 2;
    if (n == -15 && (p >> 126) != 0) return false;
    U = n > 64 ? 0u : static_cast<uint64_t>(p >> (63 + n));
    return true;
}

__device__ __forceinline__ bool is_zero(double z)
{
    return (__double2hiint(z) << 1 | __double2loint(z)) == 0;
}

// sin(k z) where sin_kz_fixed does not cover it.  z = 0 (also the unused lanes of a ragged bunch)
// is returned as it is; up to 2^14 turns (particles that have left the bucket, an unbunched beam)
// the integer form with the longer phase; beyond it, close to zero and for Inf and NaN
// sin_f64(k * z).  Out of line, as sin_phi_rest: none of their instructions may be hoisted into the
// kicks.
static __device__ __noinline__ double sin_kz_rest(double k, PhaseScale kap, double z)
{
    if (is_zero(z)) return z;
    uint64_t U;
    if (!phase_of_turns(kap, z, U)) return sin_f64(k * z);
    return detail::sin_turns_any(U, static_cast<uint32_t>(__double2hiint(z)));
}

// sin(k z + phi) where sin_kz_phi_fixed does not cover it, likewise.  A sum below 2^-7 is left to the
// FP64 product and sine, which are exact relative to it (the phase in turns is exact to 2^-64).
static __device__ __noinline__ double sin_phi_rest(double k, PhaseScale kap, double z, double phi, PhaseOffset o)
{
    const double x = fma(k, z, phi);
    uint64_t U;
    if ((__double2hiint(x) & 0x7fffffff) < 0x3f800000 || !phase_of_turns(kap, z, U)) return sin_f64(x);
    const uint64_t uphi = static_cast<uint64_t>(detail::sar_sat(o.u, static_cast<uint32_t>(o.g)));
    return detail::sin_turns_any(__double2hiint(z) < 0 ? uphi - U : uphi + U, 0u);
}

// Either of the two where phi = 0 (ZERO) or not.  z = 0 with phi = 0 -- a particle at the centre, and the
// lanes beyond the end of a bunch in its last warp, in every turn -- is answered without the call, whose
// time the whole of a small bunch waits for.
template <bool ZERO>
__device__ __forceinline__ double sin_rest(double k, PhaseScale kap, double z, double phi, PhaseOffset o)
{
    if (is_zero(z) && (ZERO || o.u == 0)) return z;
    return ZERO ? sin_kz_rest(k, kap, z) : sin_phi_rest(k, kap, z, phi, o);
}

// The kicks take the integer sine of all their particles first, without a branch in between
// (the particles' chains and the FP64 work beside them overlap), and then mend the few that
// it does not cover: `ok` is cleared for those.

// sin(k z) of a phase below one turn: k / 2 pi = kap.K 2^(959 - kap.cn), so that with the
// significand M and the biased exponent e of z the phase is (M K 2^-64) 2^(-63 - n) turns,
// n = cn - e (n >= 0 for every phase below half a turn, n >= -1 below a whole one).  Below a quarter
// turn (n >= 2) the product keeps all its bits as the last factor, so the result is as exact relative
// to itself as to 1 however small z is.  Not covered: z = 0, n < 0 (a particle that has left the
// bucket; WIDE: n < -1, for the shorter wave of a second RF system, one instruction more), |k z| below
// 2^-800, a phase within 1e-9 of a half turn, Inf and NaN.
template <bool WIDE>
__device__ __forceinline__ double sin_kz_fixed(PhaseScale kap, double z, bool& ok)
{
    using namespace detail;
    const uint32_t hi = static_cast<uint32_t>(__double2hiint(z));
    const int n = kap.cn - static_cast<int>((hi >> 20) & 0x7ffu);
    const uint64_t p = mulhi_trunc(mantissa64(z), kap.K);
    // 2^-63 turns
    const uint64_t W = WIDE ? shr_sat(p, static_cast<uint32_t>(n + 1)) << 1 : shr_sat(p, static_cast<uint32_t>(n));
    const uint64_t V = fold_half_turn(W << 2);
    const bool small = WIDE ? n >= 2 : static_cast<uint32_t>(n) >= 2u;
    const uint64_t S = mulhi_trunc63(small ? p : V, sin_poly_fixed(V));
    ok = static_cast<uint32_t>(WIDE ? n + 1 : n) <= 800u && (S >> 32) != 0u;
    return fixed_to_double(S, small ? n - 2 : 0, hi ^ static_cast<uint32_t>(W >> 31));
}

// sin(k z + phi), phi as a PhaseOffset.  The phases are added as integers in 2^(-64 - t) turns:
// t = 0 adds fractions of a turn modulo 1; where both phases are small, t > 0 scales the sum up until
// its larger term fills the word (k z below 2^-n turns takes t <= n - 3, phi takes t <= g: the sum
// stays below a quarter turn of the scaled word, where the fold is the magnitude).  So the sum is exact
// to 2^-59 of its larger term however small both are, as the FP64 fma(k, z, phi) is to 2^-53; with
// t = 0 throughout it was exact to 2^-62 turns only, which a small k z or phi does not have bits for.
// Not covered: n < -1 (never below one turn of k z), a sum that does not fill the significand (within
// 2^-31 of a half turn, or of cancellation) or lies below 2^-800, Inf and NaN.
__device__ __forceinline__ double sin_kz_phi_fixed(PhaseScale kap, double z, PhaseOffset o, bool& ok)
{
    using namespace detail;
    const uint32_t hi = static_cast<uint32_t>(__double2hiint(z));
    const int n1 = kap.cn + 1 - static_cast<int>((hi >> 20) & 0x7ffu);  // n + 1: from n = -1 on
    const int t = max(min(n1 - 4, o.g), 0);
    const uint64_t U = shr_sat(mulhi_trunc(mantissa64(z), kap.K), static_cast<uint32_t>(n1 - t)) << 2;
    const uint64_t uphi = static_cast<uint64_t>(sar_sat(o.u, static_cast<uint32_t>(o.g - t)));
    const uint64_t W = static_cast<int>(hi) < 0 ? uphi - U : uphi + U;
    const uint64_t V = fold_half_turn(W << 1);
    const uint64_t S = mulhi_trunc63(V, sin_poly_fixed(shr_sat(V, static_cast<uint32_t>(t))));
    ok = n1 >= 0 && t <= 800 && (S >> 32) != 0u;
    return fixed_to_double(S, t, static_cast<uint32_t>(W >> 32));
}

// sin and cos of 2 pi a, a in turns (the chromatic phase advance): the fraction of a as 2^-64
// turns, exact, and two fixed-point sines a quarter turn apart.  |a| >= 2^20 turns, Inf and
// NaN fall back to CUDA's sin and cos.
static __device__ __noinline__ void sincos_turns_wide(double a, double& s, double& c)
{
    s = sin(detail::kTwoPi * a);
    c = cos(detail::kTwoPi * a);
}

__device__ __forceinline__ void sincos_turns(double a, double& s, double& c)
{
    using namespace detail;
    const uint32_t hi = static_cast<uint32_t>(__double2hiint(a));
    const int n = 1022 - static_cast<int>((hi >> 20) & 0x7ffu);  // |a| = M 2^(-64 - n)
    if (n < -20) {
        sincos_turns_wide(a, s, c);
        return;
    }
    const uint64_t M = mantissa64(a);
    const uint64_t U = n >= 0 ? shr_sat(M, static_cast<uint32_t>(n)) : shl_sat(M, static_cast<uint32_t>(-n));
    s = sin_turns_any(U, hi);
    c = sin_turns_any(U + 0x4000000000000000ull, 0u);
}

// The chromatic rotation's sine times beta, sine over beta and cosine of 2 pi (q + xi d):
// the phase as a sum of 2^-64 turns and the products with beta and 1/beta on the fixed-point
// sine, so each is rounded once and no FP64 instruction is used.
static __device__ __noinline__ void chroma_rest(double q, double xi, double beta, double ibeta, double d,
                                                double& sb, double& sib, double& c)
{
    double s;
    sincos_turns(fma(xi, d, q), s, c);
    sb = beta * s;
    sib = s * ibeta;
}

__device__ __forceinline__ void chroma_fixed(const ChromaPlane& w, double d, double& sb, double& sib,
                                             double& c, bool& ok)
{
    using namespace detail;
    const uint32_t hi = static_cast<uint32_t>(__double2hiint(d));
    const uint32_t e = (hi >> 20) & 0x7ffu;
    // |xi d| = hi64(M K) 2^(e + xi.e - 1021) in 2^-64 turns; every |xi d| below half a turn is covered, none
    // from a turn on
    const uint32_t n = static_cast<uint32_t>(1022 - w.xi.e - static_cast<int>(e));
    const uint64_t A = shr_sat(mulhi_trunc(mantissa64(d), w.xi.K), n) << 1;
    ok = n <= 2047u && (e != 0u || (hi << 1 | static_cast<uint32_t>(__double2loint(d))) == 0u);
    const uint64_t U = ((hi >> 31) ^ static_cast<uint32_t>(w.xi.neg)) != 0u ? w.uq - A : w.uq + A;
    const uint64_t V = fold_half_turn(U << 1);
    const uint64_t S = mulhi_trunc63(V, sin_poly_fixed(V));
    const uint32_t sign = static_cast<uint32_t>(U >> 32);
    const uint64_t Sb = mulhi_trunc63(S, w.b.K), Si = mulhi_trunc63(S, w.ib.K);
    ok = ok && (Sb >> 32) != 0u && (Si >> 32) != 0u;
    sb = fixed_to_double(Sb, -1 - w.b.e, sign);  // Sb 2^(b.e - 59)
    sib = fixed_to_double(Si, -1 - w.ib.e, sign);
    c = sin_turns_any(U + 0x4000000000000000ull, 0u);
}

}  // namespace phtl
