// FP64 per-particle operations shared by the FP64 kernels (single bunch and batched).
//
// One thread owns P = 2 particles (1 in small bunches: the functions take their number N from the
// arrays).  The stage order of each scheme follows the readings
// of Sec. 1.1.2 stated in phtl.h; the transverse push is the Sec. 1.1.1 matrix.
#pragma once

#include <cuda_runtime.h>

#include "internal.h"
#include "monitor.cuh"
#include "dfloat.cuh"
#include "sin_f64.cuh"

namespace phtl {
namespace f64 {

// Particles per thread: independent FP64 dependency chains per thread (even).
#ifndef PHTL_F64_PARTICLES_PER_THREAD
#define PHTL_F64_PARTICLES_PER_THREAD 2
#endif
constexpr int P = PHTL_F64_PARTICLES_PER_THREAD;
static_assert(P % 2 == 0, "P must be even (128-bit loads of two doubles)");

// Minimum resident 256-thread blocks per SM asked of the compiler (caps registers at
// 65536 / (256 * this)): the FP64 kernels hide the latency of the FP64 pipe and of the sine's
// integer chain with warps.  3 (80 registers, 24 warps) for all of them: Ruth4 with both planes
// and moments took 11 % longer at 2, Euler-Cromer and leap-frog 3 to 17 % longer at 4 (spills).
#ifndef PHTL_F64_MIN_BLOCKS_256
#define PHTL_F64_MIN_BLOCKS_256 3
#endif
#ifndef PHTL_F64_MIN_BLOCKS_256_RUTH4
#define PHTL_F64_MIN_BLOCKS_256_RUTH4 3
#endif
#ifndef PHTL_F64_BATCHED_MIN_BLOCKS
#define PHTL_F64_BATCHED_MIN_BLOCKS 3  // mixed batch 2 % faster than at 2
#endif
// The general map's batched kernels hold four schemes and spill at 3 (80 registers); at 2 the widened
// map runs 2 to 20 % faster (16 bunches, Ruth4 without planes 1.85 -> 1.57 ms, RK4 3.45 -> 3.06 ms), but
// two sines without a phase or a slippage expansion 2 to 5 % slower (RK4 2.93 -> 3.09 ms).
template <bool GEN, int MODE>
constexpr int batched_min_blocks_256()
{
    return GEN && MODE != kRfPlain ? 2 : PHTL_F64_BATCHED_MIN_BLOCKS;
}
template <int SCHEME>
constexpr int min_blocks_256()
{
    return SCHEME == PHTL_RUTH4 ? PHTL_F64_MIN_BLOCKS_256_RUTH4 : PHTL_F64_MIN_BLOCKS_256;
}

// Weights of the linear map's turn loop (drifts, kicks, shears of the two planes).
struct TurnWeights {
    double dc[4], kw[3], shx[2], shy[2];
};

template <int SCHEME, bool TRANS>
__device__ __forceinline__ TurnWeights turn_weights(const double* dc, const double* kw, const MapConsts& c)
{
    constexpr int kStages = SCHEME == PHTL_RUTH4 ? 3 : 1;  // kicks; drifts: one more but for Euler-Cromer
    TurnWeights w{};
#pragma unroll
    for (int j = 0; j < 3; ++j)
        if (j < kStages) w.kw[j] = in_register(kw[j]);
#pragma unroll
    for (int i = 0; i < 4; ++i)
        if (i < (SCHEME == PHTL_EULER_CROMER ? 1 : kStages + 1)) w.dc[i] = in_register(-dc[i]);
    if (TRANS) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            w.shx[i] = in_register(c.shx[i]);
            w.shy[i] = in_register(c.shy[i]);
        }
    }
    return w;
}

// Work that a turn runs beside the sines of its kick j, in the same stretch of code without a
// branch: the sines occupy the integer pipe and the transverse push the FP64 pipe.
struct NoSideWork {
    __device__ __forceinline__ void operator()(int) const {}
};

// The force of the main RF system per unit weight, sin(phi_s + k z) - sin(phi_s) or lin z in
// rf_linear mode, of the thread's N particles.
template <int MODE, int N, class Side>
__device__ __forceinline__ void rf_force(const MapConsts& c, const double (&z)[N], double (&f)[N],
                                         const Side& side, int j)
{
    if (MODE == kRfLinear) {
#pragma unroll
        for (int p = 0; p < N; ++p) f[p] = c.lin * z[p];
        side(j);
        return;
    }
    bool ok[N], all = true;
#pragma unroll
    for (int p = 0; p < N; ++p) {
        f[p] = MODE != kRfGeneral ? sin_kz_fixed<false>(c.kap, z[p], ok[p])
                                  : sin_kz_phi_fixed(c.kap, z[p], c.ophis, ok[p]);
        all = all && ok[p];
    }
    side(j);
    if (!all) {
#pragma unroll
        for (int p = 0; p < N; ++p)
            if (!ok[p])
                f[p] = sin_rest<MODE != kRfGeneral>(c.k, c.kap, z[p], c.phis, c.ophis);
    }
    if (MODE == kRfGeneral) {
#pragma unroll
        for (int p = 0; p < N; ++p) f[p] -= c.sinphis;
    }
}

// Linear drift, ndc = -w eta C.
template <int N>
__device__ __forceinline__ void drift_neg(double (&z)[N], const double (&d)[N], double ndc)
{
#pragma unroll
    for (int p = 0; p < N; ++p) z[p] = fma(ndc, d[p], z[p]);
}

template <int MODE, int N, class Side>
__device__ __forceinline__ void kick(const double (&z)[N], double (&d)[N], double kw,
                                     const MapConsts& c, const Side& side, int j)
{
    double f[N];
    rf_force<MODE>(c, z, f, side, j);
#pragma unroll
    for (int p = 0; p < N; ++p) d[p] = fma(kw, f[p], d[p]);
}

// One turn of the scheme; stage order as in Sec. 1.1.2's readings (see phtl.h).
// w: the drift (negated) and kick weights of this bunch's scheme, -w_i eta C and w_j A.
// side: work beside the kicks' sines that touches neither z nor delta.
template <int SCHEME, int MODE, int N, class Side>
__device__ __forceinline__ void long_turn(double (&z)[N], double (&d)[N], const MapConsts& c,
                                          const TurnWeights& w, const Side& side)
{
    if (SCHEME == PHTL_EULER_CROMER) {
        kick<MODE>(z, d, w.kw[0], c, side, 0);
        drift_neg(z, d, w.dc[0]);
    } else if (SCHEME == PHTL_LEAPFROG) {
        drift_neg(z, d, w.dc[0]);
        kick<MODE>(z, d, w.kw[0], c, side, 0);
        drift_neg(z, d, w.dc[1]);
    } else {
        drift_neg(z, d, w.dc[0]);
        kick<MODE>(z, d, w.kw[0], c, side, 0);
        drift_neg(z, d, w.dc[1]);
        kick<MODE>(z, d, w.kw[1], c, side, 1);
        drift_neg(z, d, w.dc[2]);
        kick<MODE>(z, d, w.kw[2], c, side, 2);
        drift_neg(z, d, w.dc[3]);
    }
}

// Transverse push of one plane (Sec. 1.1.1 matrix).  With use_shear the rotation is
// applied as three shears (3 DFMA instead of 2 DMUL + 2 DFMA); the same map up to rounding.
template <int N>
__device__ __forceinline__ void rotate(double (&u)[N], double (&v)[N], const double (&m)[4],
                                       const double (&sh)[2], bool use_shear)
{
    if (use_shear) {
#pragma unroll
        for (int p = 0; p < N; ++p) {
            u[p] = fma(sh[0], v[p], u[p]);
            v[p] = fma(sh[1], u[p], v[p]);
            u[p] = fma(sh[0], v[p], u[p]);
        }
        return;
    }
#pragma unroll
    for (int p = 0; p < N; ++p) {
        const double un = fma(m[1], v[p], m[0] * u[p]);
        const double vn = fma(m[3], v[p], m[2] * u[p]);
        u[p] = un;
        v[p] = vn;
    }
}

// The linear map's transverse push as the side work of a turn's kicks: both planes beside the
// only kick, or x beside Ruth4's first and y beside its second.
template <int SCHEME, int N>
struct RotateBeside {
    static constexpr int kYBeside = SCHEME == PHTL_RUTH4 ? 1 : 0;
    double (&x)[N];
    double (&xp)[N];
    double (&y)[N];
    double (&yp)[N];
    bool hx, hy;
    const MapConsts& c;
    const TurnWeights& w;
    __device__ __forceinline__ void operator()(int j) const
    {
        if (j == 0 && hx) rotate(x, xp, c.mx, w.shx, c.shear_x != 0);
        if (j == kYBeside && hy) rotate(y, yp, c.my, w.shy, c.shear_y != 0);
    }
};

// ---- widened map: nonlinear slippage and chromaticity -------------------------------

// Weights of the general turn loop: the drifts and their slippage terms negated (-w_i eta0 C,
// -w_i eta1 C, -w_i eta2 C), the kicks of both RF systems, the shears of planes without
// chromaticity, and the constants with which sums and products are formed as FMAs of registers
// (a + b = fma(a, 1, b) and a b = fma(a, b, -0) exactly; see in_register).
struct GeneralWeights {
    double dc[4], g1[4], g2[4], kw[3], kw2[3], shx[2], shy[2];
    double one, mzero, half, two, sixth;
    int zero;  // see integer_copy
};

// A copy of a double on the integer pipe, zero = 0 in a register the compiler cannot see through:
// it copies a register pair with a DADD otherwise.
__device__ __forceinline__ double integer_copy(double v, int zero)
{
    return __hiloint2double(__double2hiint(v) ^ zero, __double2loint(v) ^ zero);
}

template <int SCHEME>
__device__ __forceinline__ GeneralWeights general_weights(const double* dc, const double* kw,
                                                          const double* kw2, const MapConsts& c)
{
    GeneralWeights w{};
    constexpr int kKicks = SCHEME == PHTL_RUTH4 ? 3 : 1;
    constexpr int kDrifts = SCHEME == PHTL_RUTH4 ? 4 : (SCHEME == PHTL_LEAPFROG ? 2 : 1);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (i < kDrifts) {
            w.dc[i] = in_register(-dc[i]);
            // (also keeps the compiler from forming the products anew in every turn)
            w.g1[i] = in_register(-(drift_weight(SCHEME, i) * c.eta1C));
            w.g2[i] = in_register(-(drift_weight(SCHEME, i) * c.eta2C));
        }
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        if (j < kKicks) {
            w.kw[j] = in_register(kw[j]);
            w.kw2[j] = in_register(kw2[j]);
        }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        w.shx[i] = in_register(c.shx[i]);
        w.shy[i] = in_register(c.shy[i]);
    }
    w.one = in_register(1.0);
    w.mzero = in_register(-0.0);
    w.half = in_register(0.5);
    w.two = in_register(2.0);
    w.sixth = in_register(1.0 / 6.0);
    w.zero = __shfl_sync(kFullMask, 0, 0);
    return w;
}

// Drift with the slippage expansion: z -= (dc + g1 d + g2 d^2) d for this stage's
// w eta(d) C (weights negated, see GeneralWeights).  Without the expansion the linear drift.
template <int MODE, int N>
__device__ __forceinline__ void drift_nl(double (&z)[N], const double (&d)[N], const GeneralWeights& w, int i)
{
    if (MODE == kRfPlain) {
        drift_neg(z, d, w.dc[i]);
        return;
    }
#pragma unroll
    for (int p = 0; p < N; ++p) {
        const double e = fma(fma(w.g2[i], d[p], w.g1[i]), d[p], w.dc[i]);
        z[p] = fma(e, d[p], z[p]);
    }
}

// Forces of both RF systems per unit weight: f of the main one (as rf_force) and, when `dual`, g of
// the second, sin(phi2 + k2 z) - sin(phi2) or cos(phi2) k2 z in rf_linear mode.  The sines of both
// run together, before the particles they do not cover are mended.
// `dual`: a compile-time constant in the single-bunch kernels, which have a variant without the
// second system; the batched kernels pass the ring's flag.
template <int MODE, int N>
__device__ __forceinline__ void rf_forces(const MapConsts& c, const double (&z)[N], double (&f)[N],
                                          double (&g)[N], bool dual)
{
    if (!dual) {
        rf_force<MODE>(c, z, f, NoSideWork{}, 0);
        return;
    }
    if (MODE == kRfLinear) {
#pragma unroll
        for (int p = 0; p < N; ++p) {
            f[p] = c.lin * z[p];
            g[p] = c.lin2 * z[p];
        }
        return;
    }
    bool ok[N], ok2[N], all = true;
#pragma unroll
    for (int p = 0; p < N; ++p) {
        f[p] = MODE != kRfGeneral ? sin_kz_fixed<false>(c.kap, z[p], ok[p])
                                  : sin_kz_phi_fixed(c.kap, z[p], c.ophis, ok[p]);
        g[p] = MODE == kRfPlain ? sin_kz_fixed<true>(c.kap2, z[p], ok2[p])
                                : sin_kz_phi_fixed(c.kap2, z[p], c.ophi2, ok2[p]);
        all = all && ok[p] && ok2[p];
    }
    if (!all) {
#pragma unroll
        for (int p = 0; p < N; ++p) {
            if (!ok[p])
                f[p] = sin_rest<MODE != kRfGeneral>(c.k, c.kap, z[p], c.phis, c.ophis);
            if (!ok2[p]) g[p] = sin_rest<MODE == kRfPlain>(c.k2, c.kap2, z[p], c.phi2, c.ophi2);
        }
    }
#pragma unroll
    for (int p = 0; p < N; ++p) {
        if (MODE == kRfGeneral) f[p] -= c.sinphis;
        if (MODE != kRfPlain) g[p] -= c.sinphi2;
    }
}

// Kick of the widened map: the main RF system, then the second one when `dual` -- kw2: this
// stage's w_j A2.
template <int MODE, int N>
__device__ __forceinline__ void kick_gen(const double (&z)[N], double (&d)[N], double kw, double kw2,
                                         const MapConsts& c, bool dual)
{
    double f[N], g[N];
    rf_forces<MODE>(c, z, f, g, dual);
#pragma unroll
    for (int p = 0; p < N; ++p) {
        d[p] = fma(kw, f[p], d[p]);
        if (dual) d[p] = fma(kw2, g[p], d[p]);
    }
}

// Right-hand side of the smooth motion per turn (classic RK4's derivative):
// dz/dn = -eta(d) C d = -(dc + g1 d + g2 d^2) d and dd/dn = kw F1(z) + kw2 F2(z), with
// dc = eta0 C, g1 = eta1 C, g2 = eta2 C, kw = A, kw2 = A2.
template <int MODE, int N>
__device__ __forceinline__ void rk4_rhs(const double (&z)[N], const double (&d)[N], const MapConsts& c,
                                        const GeneralWeights& w, bool dual, double (&fz)[N],
                                        double (&fd)[N])
{
    // the products are rounded on their own: the stage arguments and the weighted sum reuse
    // them, and an FMA contraction chosen differently where `dual` is a compile-time constant
    // than where it is not would break the bitwise agreement of the single-bunch and batched
    // kernels
    double f[N], g[N];
    rf_forces<MODE>(c, z, f, g, dual);
#pragma unroll
    for (int p = 0; p < N; ++p) {
        const double e = MODE == kRfPlain ? w.dc[0] : fma(fma(w.g2[0], d[p], w.g1[0]), d[p], w.dc[0]);
        fz[p] = __fma_rn(e, d[p], w.mzero);
        fd[p] = __fma_rn(w.kw[0], f[p], w.mzero);
        if (dual) fd[p] = fma(w.kw2[0], g[p], fd[p]);
    }
}

// One classic RK4 step of one turn: k1 at the start, k2 and k3 at the half step from k1
// and k2, k4 at the full step from k3, and the weighted sum (k1 + 2 k2 + 2 k3 + k4) / 6.
// The four stages are a loop that is not unrolled: with the sines of both RF systems in line
// four times the turn's code did not fit the instruction cache (3.5 stalled cycles for
// instructions per issue on the double-RF ring).  rf_linear has no sines: in line, and two FP64
// operations fewer.
template <int MODE, int N>
__device__ __forceinline__ void rk4_turn(double (&z)[N], double (&d)[N], const MapConsts& c,
                                         const GeneralWeights& w, bool dual)
{
    double a[N], b[N], kz[N], kd[N], sz[N], sd[N];
    if constexpr (MODE == kRfLinear) {
        double k1z[N], k1d[N], k2z[N], k2d[N];
        rk4_rhs<MODE>(z, d, c, w, dual, k1z, k1d);
#pragma unroll
        for (int p = 0; p < N; ++p) a[p] = fma(w.half, k1z[p], z[p]), b[p] = fma(w.half, k1d[p], d[p]);
        rk4_rhs<MODE>(a, b, c, w, dual, k2z, k2d);
#pragma unroll
        for (int p = 0; p < N; ++p) a[p] = fma(w.half, k2z[p], z[p]), b[p] = fma(w.half, k2d[p], d[p]);
        rk4_rhs<MODE>(a, b, c, w, dual, kz, kd);
#pragma unroll
        for (int p = 0; p < N; ++p) {
            sz[p] = __fma_rn(k2z[p], w.one, kz[p]);
            sd[p] = __fma_rn(k2d[p], w.one, kd[p]);
            a[p] = __fma_rn(kz[p], w.one, z[p]);
            b[p] = __fma_rn(kd[p], w.one, d[p]);
        }
        rk4_rhs<MODE>(a, b, c, w, dual, kz, kd);
#pragma unroll
        for (int p = 0; p < N; ++p) {
            z[p] = fma(fma(w.two, sz[p], __fma_rn(k1z[p], w.one, kz[p])), w.sixth, z[p]);
            d[p] = fma(fma(w.two, sd[p], __fma_rn(k1d[p], w.one, kd[p])), w.sixth, d[p]);
        }
        return;
    }
#pragma unroll
    for (int p = 0; p < N; ++p) {
        a[p] = integer_copy(z[p], w.zero);
        b[p] = integer_copy(d[p], w.zero);
        sz[p] = sd[p] = 0.0;
    }
#pragma unroll 1
    for (int st = 0;; ++st) {
        rk4_rhs<MODE>(a, b, c, w, dual, kz, kd);
        if (st == 3) break;
        const double cs = st == 0 ? w.one : w.two, step = st == 2 ? w.one : w.half;
#pragma unroll
        for (int p = 0; p < N; ++p) {
            sz[p] = fma(cs, kz[p], sz[p]);
            sd[p] = fma(cs, kd[p], sd[p]);
            a[p] = fma(step, kz[p], z[p]);
            b[p] = fma(step, kd[p], d[p]);
        }
    }
#pragma unroll
    for (int p = 0; p < N; ++p) {
        z[p] = fma(__fma_rn(kz[p], w.one, sz[p]), w.sixth, z[p]);
        d[p] = fma(__fma_rn(kd[p], w.one, sd[p]), w.sixth, d[p]);
    }
}

// One turn of the scheme with the slippage expansion and the second RF system.
template <int SCHEME, int MODE, int N>
__device__ __forceinline__ void long_turn_nl(double (&z)[N], double (&d)[N], const MapConsts& c,
                                             const GeneralWeights& w, bool dual)
{
    if (SCHEME == PHTL_RK4) {
        rk4_turn<MODE>(z, d, c, w, dual);
    } else if (SCHEME == PHTL_EULER_CROMER) {
        kick_gen<MODE>(z, d, w.kw[0], w.kw2[0], c, dual);
        drift_nl<MODE>(z, d, w, 0);
    } else if (SCHEME == PHTL_LEAPFROG) {
        drift_nl<MODE>(z, d, w, 0);
        kick_gen<MODE>(z, d, w.kw[0], w.kw2[0], c, dual);
        drift_nl<MODE>(z, d, w, 1);
    } else {
        drift_nl<MODE>(z, d, w, 0);
        kick_gen<MODE>(z, d, w.kw[0], w.kw2[0], c, dual);
        drift_nl<MODE>(z, d, w, 1);
        kick_gen<MODE>(z, d, w.kw[1], w.kw2[1], c, dual);
        drift_nl<MODE>(z, d, w, 2);
        kick_gen<MODE>(z, d, w.kw[2], w.kw2[2], c, dual);
        drift_nl<MODE>(z, d, w, 3);
    }
}

// Chromatic rotation of one plane: each particle turns by 2 pi (q + xi d) with its own d
// (after the turn's longitudinal step).
template <int N>
__device__ __forceinline__ void rotate_chroma(double (&u)[N], double (&v)[N], const double (&d)[N],
                                              const ChromaPlane& h, double q, double xi, double b,
                                              double ib, double mzero)
{
    double sb[N], sib[N], cs[N];
    bool ok[N], all = h.on != 0;
#pragma unroll
    for (int p = 0; p < N; ++p) {
        chroma_fixed(h, d[p], sb[p], sib[p], cs[p], ok[p]);
        ok[p] = ok[p] && h.on != 0;
        all = all && ok[p];
    }
    if (!all) {
#pragma unroll
        for (int p = 0; p < N; ++p)
            if (!ok[p]) chroma_rest(q, xi, b, ib, d[p], sb[p], sib[p], cs[p]);
    }
#pragma unroll
    for (int p = 0; p < N; ++p) {
        const double un = fma(sb[p], v[p], __fma_rn(cs[p], u[p], mzero));
        const double vn = fma(-sib[p], u[p], __fma_rn(cs[p], v[p], mzero));
        u[p] = un;
        v[p] = vn;
    }
}

// The transverse step of the general loop: chromatic where xi != 0, else the one matrix.
template <int N>
__device__ __forceinline__ void transverse_gen(double (&x)[N], double (&xp)[N], double (&y)[N],
                                               double (&yp)[N], const double (&d)[N], bool hx,
                                               bool hy, const MapConsts& c, const GeneralWeights& w)
{
    if (hx) {
        if (c.chroma_x) rotate_chroma(x, xp, d, c.chx, c.qx, c.xi_x, c.bx, c.ibx, w.mzero);
        else rotate(x, xp, c.mx, w.shx, c.shear_x != 0);
    }
    if (hy) {
        if (c.chroma_y) rotate_chroma(y, yp, d, c.chy, c.qy, c.xi_y, c.by, c.iby, w.mzero);
        else rotate(y, yp, c.my, w.shy, c.shear_y != 0);
    }
}

// ---- moments: exact integer sums per warp ------------------------------------------------
//
// A coordinate's values are brought to the warp's common exponent E (the largest biased
// exponent among its lanes) as 61-bit integers X, a = X 2^(E + kMomentShift - 1086): no bit of a
// value within 2^-8 of the largest is lost.  The thread adds X, X^2 and X Y over its particles,
// the warp the threads' sums as 64-bit integers, and each total is converted to FP64 once.  A
// thread's sum is cut below 2^-56 of the warp's largest magnitude, one of products below 2^-55 of the
// product of its coordinates' largest (up to 2.5 such units), so a warp's totals are within 2^-50.9
// and 2^-48.6 of those.  The squares are products of the magnitudes rounded down, so a single
// particle's variance does not come out positive.
//
// The double-float sums before these took ~590 instructions per particle and record with both
// planes (bit splits, TwoSum and Fast2Sum in every addition); these take ~390.
template <int N>
constexpr int kMomentShift = N <= 2 ? 3 : 4;  // N X below 2^62
constexpr int kSumDrop = 4;                   // the warp adds (sum of X) 2^-4 ...
constexpr int kProductDrop = 65;              // ... and (sum of X Y) 2^-65, below 2^63

struct PlaneExponents {
    int a, b;  // the warp's exponents of the plane's two coordinates
};

// High words without the sign: ordered as the magnitudes are.
template <int N>
__device__ __forceinline__ int warp_exponent(const double (&a)[N])
{
    unsigned m = 0u;
#pragma unroll
    for (int p = 0; p < N; ++p) m = max(m, static_cast<unsigned>(__double2hiint(a[p])) & 0x7fffffffu);
    return static_cast<int>(__reduce_max_sync(kFullMask, m) >> 20);
}

// |a| in units of 2^(E + kMomentShift - 1086), and the sign as a mask.
template <int N>
__device__ __forceinline__ uint64_t moment_magnitude(double a, int E, uint32_t& neg)
{
    const uint32_t hi = static_cast<uint32_t>(__double2hiint(a));
    neg = static_cast<uint32_t>(static_cast<int32_t>(hi) >> 31);
    const uint32_t e = (hi >> 20) & 0x7ffu;  // 0: zero (or subnormal) has no leading one, shift it out
    return detail::shr_sat(detail::mantissa64(a), e != 0u ? static_cast<uint32_t>(E + kMomentShift<N>) - e : 64u);
}

__device__ __forceinline__ int64_t moment_signed(uint64_t X, uint32_t neg)
{
    const uint64_t m = static_cast<uint64_t>(neg) << 32 | neg;
    return static_cast<int64_t>((X ^ m) - m);
}

// Sums of one plane (a, b) over the thread's particles: a, b (in 2^kSumDrop X), a^2, b^2 and ab
// (in 2^kProductDrop X Y).
template <int N>
__device__ __forceinline__ void pair_sums_fixed(const double (&a)[N], const double (&b)[N],
                                                PlaneExponents E, int64_t* f)
{
    uint64_t aa = 0, aac = 0, bb = 0, bbc = 0;
    int64_t ab = 0, abc = 0;
    int64_t sa = 0, sb = 0;
#pragma unroll
    for (int p = 0; p < N; ++p) {
        uint32_t na, nb;
        const uint64_t A = moment_magnitude<N>(a[p], E.a, na), B = moment_magnitude<N>(b[p], E.b, nb);
        const uint32_t a1 = static_cast<uint32_t>(A >> 32), a0 = static_cast<uint32_t>(A);
        const uint32_t b1 = static_cast<uint32_t>(B >> 32), b0 = static_cast<uint32_t>(B);
        aa += static_cast<uint64_t>(a1) * a1;     // A^2 = aa 2^64 + 2 aac 2^32 + (below 2^64)
        aac += static_cast<uint64_t>(a1) * a0;
        bb += static_cast<uint64_t>(b1) * b1;
        bbc += static_cast<uint64_t>(b1) * b0;
        const int64_t As = moment_signed(A, na), Bs = moment_signed(B, nb);
        sa += As;
        sb += Bs;
        const int32_t as1 = static_cast<int32_t>(As >> 32), bs1 = static_cast<int32_t>(Bs >> 32);
        const int32_t ah = static_cast<int32_t>(static_cast<uint32_t>(As) >> 1);
        const int32_t bh = static_cast<int32_t>(static_cast<uint32_t>(Bs) >> 1);
        ab += static_cast<int64_t>(as1) * bs1;    // A B = ab 2^64 + abc 2^33 + ...
        abc += static_cast<int64_t>(as1) * bh;
        abc += static_cast<int64_t>(bs1) * ah;
    }
    f[0] = sa >> kSumDrop;
    f[1] = sb >> kSumDrop;
    f[2] = static_cast<int64_t>((aa >> 1) + (aac >> 32));
    f[3] = static_cast<int64_t>((bb >> 1) + (bbc >> 32));
    f[4] = (ab >> 1) + (abc >> 32);
}

// S 2^x in FP64, rounded to nearest or (nearest = 0, and below the normal range) truncated;
// above the range Inf.  Integer instructions: a conversion to FP64 takes the FP64 pipe.
__device__ __forceinline__ double scaled_to_double(int64_t S, int x, uint32_t nearest)
{
    const uint64_t a = static_cast<uint64_t>(S < 0 ? -S : S);
    const int c = __clzll(static_cast<long long>(a));
    const uint64_t N = detail::shl_sat(a, static_cast<uint32_t>(c));
    const uint64_t r = (N >> 11) + (static_cast<uint32_t>(N >> 10) & nearest);
    const int e = 1085 - c + x;  // biased exponent less the leading one of r
    uint32_t hi = static_cast<uint32_t>(r >> 32) + (static_cast<uint32_t>(e) << 20);
    uint32_t lo = static_cast<uint32_t>(r);
    if (e < 0) {
        const uint64_t sub = detail::shr_sat(N, static_cast<uint32_t>(11 - e));
        hi = static_cast<uint32_t>(sub >> 32);
        lo = static_cast<uint32_t>(sub);
    }
    if (a == 0) hi = lo = 0u;
    if (e > 2045 && a != 0) {
        hi = 0x7ff00000u;
        lo = 0u;
    }
    return __hiloint2double(static_cast<int>(hi | (static_cast<uint32_t>(S >> 32) & 0x80000000u)),
                            static_cast<int>(lo));
}

// Add this block's moment sums of the current turn into monitor row `row`.
// smem: 2 * (blockDim.x / 32) * 16 doubles.
template <bool TRANS, int N>
__device__ __forceinline__ void record(const double (&z)[N], const double (&d)[N],
                                       const double (&x)[N], const double (&xp)[N],
                                       const double (&y)[N], const double (&yp)[N],
                                       float cnt, bool hx, bool hy, double* smem, int parity,
                                       double* rows, int64_t row)
{
    constexpr int NF = TRANS ? 16 : 8;
    constexpr int kShift = TRANS ? 1 : 2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int field = lane >> kShift;  // the field whose total this lane ends up with
    int64_t f[NF];
    f[0] = static_cast<int64_t>(static_cast<int>(cnt));
    PlaneExponents E{warp_exponent(z), warp_exponent(d)};
    PlaneExponents Ef{0, 0};           // of this lane's field; an absent plane's sums are zeros
    if (field < 6) Ef = E;
    int k = field - 1;                 // 0..4: a, b, a^2, b^2, ab of the plane Ef
    pair_sums_fixed(z, d, E, f + 1);
    if constexpr (TRANS) {
        if (hx) {
            E = PlaneExponents{warp_exponent(x), warp_exponent(xp)};
            pair_sums_fixed(x, xp, E, f + 6);
            if (field >= 6 && field < 11) Ef = E;
        } else {
#pragma unroll
            for (int j = 6; j < 11; ++j) f[j] = 0;
        }
        if (hy) {
            E = PlaneExponents{warp_exponent(y), warp_exponent(yp)};
            pair_sums_fixed(y, yp, E, f + 11);
            if (field >= 11) Ef = E;
        } else {
#pragma unroll
            for (int j = 11; j < 16; ++j) f[j] = 0;
        }
        k -= field >= 11 ? 10 : (field >= 6 ? 5 : 0);
    } else {
        f[6] = f[7] = 0;
    }
    const int64_t total = warp_reduce_scatter_int<NF>(f, lane);
    // the unit of X is 2^(E + kMomentShift - 1086); field 0 counts
    const int e1 = k == 1 || k == 3 ? Ef.b : Ef.a;
    const int e2 = k == 3 || k == 4 ? Ef.b : Ef.a;
    const int ex = field == 0 ? 0
                   : k < 2    ? e1 + kMomentShift<N> - 1086 + kSumDrop
                              : e1 + e2 + 2 * (kMomentShift<N> - 1086) + kProductDrop;
    // squares truncated once more: a single particle's variance stays at or below zero
    double v = scaled_to_double(total, ex, k == 2 || k == 3 ? 0u : 1u);
    // Inf or NaN among the warp's values
    if (field != 0 && (e1 == 2047 || (k >= 2 && e2 == 2047))) v = __hiloint2double(0x7ff80000, 0);
    const bool owner = (lane & ((1 << kShift) - 1)) == 0;  // one lane of each field's
    if (nwarps == 1) {
        if (owner && field < (TRANS ? 16 : 6)) atomicAdd(rows + row * PHTL_MON_FIELDS + field, v);
        return;
    }
    double* buf = smem + parity * (nwarps * 16);
    if (owner) buf[warp * 16 + field] = v;
    __syncthreads();
    if (warp == 0 && lane < (TRANS ? 16 : 6)) {
        double s = buf[lane];
        for (int w = 1; w < nwarps; ++w) s += buf[w * 16 + lane];
        atomicAdd(rows + row * PHTL_MON_FIELDS + lane, s);
    }
}

// 128-bit accesses only where the host allowed them (vec) AND the address really is
// 16-byte aligned; anything else takes the scalar path.
__device__ __forceinline__ bool aligned16(const void* p)
{
    return (reinterpret_cast<uintptr_t>(p) & 15) == 0;
}

template <int N>
__device__ __forceinline__ void load2(const double* __restrict__ g, int64_t base, int64_t n,
                                      bool vec, double (&v)[N])
{
    if constexpr (N % 2 == 0) {
        if (vec && base + N <= n && aligned16(g + base)) {
#pragma unroll
            for (int k = 0; k < N; k += 2) {
                const double2 t = __ldcs(reinterpret_cast<const double2*>(g + base + k));
                v[k] = t.x;
                v[k + 1] = t.y;
            }
            return;
        }
    }
#pragma unroll
    for (int p = 0; p < N; ++p) v[p] = (base + p < n) ? g[base + p] : 0.0;
}

template <int N>
__device__ __forceinline__ void store2(double* __restrict__ g, int64_t base, int64_t n,
                                       bool vec, const double (&v)[N])
{
    if constexpr (N % 2 == 0) {
        if (vec && base + N <= n && aligned16(g + base)) {
#pragma unroll
            for (int k = 0; k < N; k += 2)
                __stcs(reinterpret_cast<double2*>(g + base + k), make_double2(v[k], v[k + 1]));
            return;
        }
    }
#pragma unroll
    for (int p = 0; p < N; ++p)
        if (base + p < n) g[base + p] = v[p];
}

}  // namespace f64
}  // namespace phtl
