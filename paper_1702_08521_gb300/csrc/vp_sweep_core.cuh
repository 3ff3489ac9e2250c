// vp_sweep_core.cuh -- per-interface arithmetic of the SL-MPP5/7 sweep and
// the line walker shared by every sweep kernel (strided, contiguous, TMA,
// ensemble).
#pragma once

#include <type_traits>

#include "vp_internal.cuh"

namespace vp_core {

// ---- limiter arithmetic (Appendix A and Sec. 2.1.1) -------------------------

// Every product that meets a sum is written either as fma() or as a
// round-to-nearest multiply (mul_rn), never left to contraction: the walk
// step is compiled in several instances (unrolled and remainder loops, the
// first interface of a segment), and a contraction the compiler takes in one
// instance but not another would make a cell's last bit depend on where the
// tile and segment boundaries fall, i.e. on the autotuner's choice.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// ---- two lines at once ---------------------------------------------------------
//
// P2 holds one value of each of two lines that a thread walks in lockstep.
// Additions, multiplications and fused multiply-adds are the packed FP32
// pair instructions of sm_100+ (one issue slot for both lines, each half
// rounded exactly as the scalar instruction would round it); min, max and
// comparisons are per half.  Every line therefore gets bit for bit the
// result of the one-line walk, whichever of the two walks runs it.
// the scalar overloads stay visible next to the pair overloads below
using ::fma;
using ::fmax;
using ::fmin;

struct P2 {
    float2 v;
    P2() = default;
    __device__ __forceinline__ explicit P2(float s) : v(make_float2(s, s)) {}
    __device__ __forceinline__ P2(float2 x) : v(x) {}
};
__device__ __forceinline__ P2 operator+(P2 a, P2 b) { return P2(__fadd2_rn(a.v, b.v)); }
// a - b as a + (-1) b: the product is exact, so this rounds as the subtraction
__device__ __forceinline__ P2 operator-(P2 a, P2 b) { return P2(__ffma2_rn(b.v, make_float2(-1.f, -1.f), a.v)); }
__device__ __forceinline__ P2 operator-(P2 a) { return P2(make_float2(-a.v.x, -a.v.y)); }
__device__ __forceinline__ P2 operator*(P2 a, P2 b) { return P2(__fmul2_rn(a.v, b.v)); }
__device__ __forceinline__ P2 fma(P2 a, P2 b, P2 c) { return P2(__ffma2_rn(a.v, b.v, c.v)); }
__device__ __forceinline__ P2 fmin(P2 a, P2 b) { return P2(make_float2(fminf(a.v.x, b.v.x), fminf(a.v.y, b.v.y))); }
__device__ __forceinline__ P2 fmax(P2 a, P2 b) { return P2(make_float2(fmaxf(a.v.x, b.v.x), fmaxf(a.v.y, b.v.y))); }
// both lines equal (the flat-stencil test asks it of both lines of a pair)
__device__ __forceinline__ bool operator==(P2 a, P2 b) { return a.v.x == b.v.x && a.v.y == b.v.y; }

// ---- FP64 with integer comparisons -------------------------------------------
//
// A warp's FP64 instruction takes 16 cycles of the SM's two FMA lanes, and
// min, max and comparisons of doubles run there too: ~28 of the ~50 FP64
// instructions of a cell-update.  FD orders doubles by their bits on the
// integer pipe instead (the same minimum or maximum for every pair of finite
// numbers, up to the sign of zero).  Numbers that are not finite, or so large
// that the arithmetic between the comparisons could overflow, are ordered
// differently from fmin / fmax: the walk notes them (FD::kBig) and its caller
// repeats the segment in plain double.
struct FD {
    double v;
    static constexpr int kBig = (1023 + 1000) << 20;  // high word of 2^1000
    FD() = default;
    __device__ __forceinline__ explicit FD(double x) : v(x) {}
};
__device__ __forceinline__ FD operator+(FD a, FD b) { return FD(__dadd_rn(a.v, b.v)); }
__device__ __forceinline__ FD operator-(FD a, FD b) { return FD(__dadd_rn(a.v, -b.v)); }
__device__ __forceinline__ FD operator-(FD a) {
    return FD(__hiloint2double(__double2hiint(a.v) ^ (int)0x80000000, __double2loint(a.v)));
}
__device__ __forceinline__ FD operator*(FD a, FD b) { return FD(__dmul_rn(a.v, b.v)); }
__device__ __forceinline__ FD fma(FD a, FD b, FD c) { return FD(__fma_rn(a.v, b.v, c.v)); }
__device__ __forceinline__ FD mul_rn(FD a, FD b) { return FD(__dmul_rn(a.v, b.v)); }
// equal bits (0 and -0 differ: the flat-stencil test then computes the flux)
__device__ __forceinline__ bool operator==(FD a, FD b) {
    return __double_as_longlong(a.v) == __double_as_longlong(b.v);
}
// a < b for a, b of different bits: two's-complement order, reversed where both are negative
__device__ __forceinline__ bool below(FD a, FD b) {
    const long long x = __double_as_longlong(a.v), y = __double_as_longlong(b.v);
    return (x < y) != ((__double2hiint(a.v) & __double2hiint(b.v)) < 0);
}
__device__ __forceinline__ FD fmin(FD a, FD b) { return below(a, b) ? a : b; }
__device__ __forceinline__ FD fmax(FD a, FD b) { return below(a, b) ? b : a; }

// shift decompositions of a pair of lines walked together (equal n and sigma)
struct LineShiftP2 {
    P2 w[7];
    P2 nu;
    int n;
    int sigma;
};
__device__ __forceinline__ LineShiftP2 pair_shift(const LineShift<float> &a, const LineShift<float> &b) {
    LineShiftP2 s;
#pragma unroll
    for (int k = 0; k < 7; ++k) s.w[k] = P2(make_float2(a.w[k], b.w[k]));
    s.nu = P2(make_float2(a.nu, b.nu));
    s.n = a.n;
    s.sigma = a.sigma;
    return s;
}

// whether the walker tests for warp-wide flat stencils (and then skips the
// interpolant and the bounds); the result is the same either way
template <typename T>
struct FlatSkip {
    static constexpr bool on = true;
};
template <>
struct FlatSkip<P2> {
    static constexpr bool on = true;
};

// 4/3 in the arithmetic's precision
template <typename T>
__device__ __forceinline__ T c43() { return T(4) / T(3); }
template <>
__device__ __forceinline__ P2 c43<P2>() { return P2(4.0f / 3.0f); }
template <>
__device__ __forceinline__ FD c43<FD>() { return FD(4.0 / 3.0); }

// minmod of four: min if all > 0, max if all < 0, else 0 (= max(min,0) + min(max,0))
template <typename T>
__device__ __forceinline__ T mm4(T a, T b, T c, T d) {
    const T mn = fmin(fmin(a, b), fmin(c, d));
    const T mx = fmax(fmax(a, b), fmax(c, d));
    return fmax(mn, T(0)) + fmin(mx, T(0));
}

// min / max of three (the three-input PTX form for FP32; measured here at the
// throughput of two two-input operations)
__device__ __forceinline__ float min3(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ double min3(double a, double b, double c) { return fmin(fmin(a, b), c); }
__device__ __forceinline__ double max3(double a, double b, double c) { return fmax(fmax(a, b), c); }
__device__ __forceinline__ FD min3(FD a, FD b, FD c) { return fmin(fmin(a, b), c); }
__device__ __forceinline__ FD max3(FD a, FD b, FD c) { return fmax(fmax(a, b), c); }
__device__ __forceinline__ P2 min3(P2 a, P2 b, P2 c) {
    return P2(make_float2(min3(a.v.x, b.v.x, c.v.x), min3(a.v.y, b.v.y, c.v.y)));
}
__device__ __forceinline__ P2 max3(P2 a, P2 b, P2 c) {
    return P2(make_float2(max3(a.v.x, b.v.x, c.v.x), max3(a.v.y, b.v.y, c.v.y)));
}

// curvature d_j = u_{j-1} - 2 u_j + u_{j+1} (App. A)
template <typename T>
__device__ __forceinline__ T curv(T um, T u, T up) {
    return fma(T(-2), u, um + up);
}

// d^{M4} between cells with curvatures x and y (App. A):
// minmod(4x - y, 4y - x, x, y).  With m = min(x, y) and M = max(x, y) the
// least of the four is min(m, 4m - M) and the greatest max(M, 4M - m); the
// minmod is the least if it is > 0, the greatest if it is < 0, else 0: the
// clamp of 0 into [least, greatest].
template <typename T>
__device__ __forceinline__ T dm4(T x, T y) {
    const T m = fmin(x, y), M = fmax(x, y);
    const T mn = fmin(m, fma(T(4), m, -M));
    const T mx = fmax(M, fma(T(4), M, -m));
    return fmin(fmax(T(0), mn), mx);
}

// The MP constraint as one clamp.  Steps 4-7 give phi_MP = median(phi, f_min,
// f_max); step 3 keeps phi when it lies strictly between u0 and f^MP, and
// that interval lies inside [f_min, f_max] (f_min <= u0; when the minmod of
// step 2 is positive f_max >= min(u1, f_UL) = f^MP, and the mirror case), so
// there the clamp returns phi as well.  Hence the constraint equals the clamp
// of phi into [f_min, f_max] for every phi.  m4m / m4p are d^{M4} at the
// upwind / downwind face of the upwind cell u0.
template <typename T>
__device__ __forceinline__ void mp_lohi_carried(T um1, T u0, T u1, T alpha, T m4m, T m4p, T &lo, T &hi) {
    const T back = u0 - um1;
    const T ful = fma(alpha, back, u0);
    const T fmd = fma(T(0.5), u0 + u1, T(-0.5) * m4p);
    const T flc = fma(c43<T>(), m4m, fma(T(0.5), back, u0));
    lo = fmax(min3(u0, u1, fmd), min3(u0, ful, flc));
    hi = fmin(max3(u0, u1, fmd), max3(u0, ful, flc));
}
template <typename T>
__device__ __forceinline__ T mp_clamp(T phi, T um1, T u0, T u1, T alpha, T m4m, T m4p) {
    T lo, hi;
    mp_lohi_carried(um1, u0, u1, alpha, m4m, m4p, lo, hi);
    return fmin(fmax(phi, lo), hi);
}

// Steps 4-6 of the MP constraint: the bounds [f_min, f_max].  Both intervals
// of step 6 contain u0, so f_min <= u0 <= f_max exactly.
template <typename T>
__device__ __forceinline__ void mp_lohi(T um2, T um1, T u0, T u1, T u2, T alpha, T &lo, T &hi) {
    const T back = u0 - um1;
    const T dm = um2 + u0 - T(2) * um1;  // curvature at the upwind neighbour
    const T dc = um1 + u1 - T(2) * u0;   // at the upwind cell
    const T dp = u0 + u2 - T(2) * u1;    // at the downwind cell
    const T m4p = mm4(T(4) * dc - dp, T(4) * dp - dc, dc, dp);
    const T m4m = mm4(T(4) * dm - dc, T(4) * dc - dm, dm, dc);
    const T ful = fma(alpha, back, u0);
    const T fmd = fma(T(0.5), u0 + u1, T(-0.5) * m4p);
    const T flc = fma(T(4) / T(3), m4m, fma(T(0.5), back, u0));
    lo = fmax(fmin(fmin(u0, u1), fmd), fmin(fmin(u0, ful), flc));
    hi = fmin(fmax(fmax(u0, u1), fmd), fmax(fmax(u0, ful), flc));
}

// Steps 4-7 (taken only when step 3 rejects phi): the median of step 7 is
// the clamp into [f_min, f_max].
template <typename T>
__device__ __forceinline__ T mp_bounds(T phi, T um2, T um1, T u0, T u1, T u2, T alpha) {
    T lo, hi;
    mp_lohi(um2, um1, u0, u1, u2, alpha, lo, hi);
    return fmin(fmax(phi, lo), hi);
}

// MP constraint of phi at the interface between u0 (upwind) and u1.
// Step 3 accepts phi iff it lies strictly between u0 and f* = u0 + minmod(p, q),
// p = u1 - u0, q = alpha (u0 - u_{-1}); with a = phi - u0 that is: a strictly
// between 0 and p and strictly between 0 and q, i.e. (p - a) a > 0 and
// (q - a) a > 0 -- products on the FMA pipe instead of min/max chains.  A phi
// this test rejects goes to steps 4-7 directly: the interval [u0, f*] lies
// inside [f_min, f_max] (f_min <= u0; f_max >= min(u1, f_UL) >= f* when the
// minmod is positive, and the mirror case), so a phi that step 3 would have
// accepted but whose product underflowed comes back unchanged from the clamp.
template <typename T>
__device__ __forceinline__ T mp_limit(T phi, T um2, T um1, T u0, T u1, T u2, T alpha) {
    const T a = phi - u0;
    const T p = u1 - u0;
    const T q = mul_rn(alpha, u0 - um1);
    if ((p - a) * a > T(0) && (q - a) * a > T(0)) return phi;
    return mp_bounds(phi, um2, um1, u0, u1, u2, alpha);
}

// Half of a cell, rounded towards minus infinity: the most mass one interface
// may take out of a non-negative cell so that two of them leave it >= 0.
__device__ __forceinline__ float half_rd(float u) { return __fmul_rd(u, 0.5f); }
__device__ __forceinline__ double half_rd(double u) { return __dmul_rd(u, 0.5); }
__device__ __forceinline__ FD half_rd(FD u) { return FD(__dmul_rd(u.v, 0.5)); }
__device__ __forceinline__ P2 half_rd(P2 u) { return P2(__fmul2_rd(u.v, make_float2(0.5f, 0.5f))); }
__device__ __forceinline__ P2 mul_rn(P2 a, P2 b) { return P2(__fmul2_rn(a.v, b.v)); }

// PP limiter (Sec. 2.1.1, Eqs. 15-23) on the mass M = nu Phi that an interface
// carries from its upwind cell u0 into u1.  For u0, u1 >= 0 and 0 < nu <= 1/2
// the theta blend returns Phi unless one half of the Euler update goes
// negative; then U+ < 0 gives theta+ (Phi - u0) = (1 - 2 nu) u0 / (2 nu), i.e.
// exactly the flux u0 / (2 nu) that empties the upwind half, and U- < 0 the
// flux -u1 / (2 nu) (both cannot bind at once).  So the limiter is the clamp
// of M into [-u1 / 2, u0 / 2], with h0, h1 the rounded-down halves of u0, u1.
// A cell then loses at most h through each of its two interfaces, and
// (u - M_out) + M_in >= 0 holds after rounding, subnormals included.
template <typename T>
__device__ __forceinline__ T pp_clamp(T M, T h0, T h1) {
    return fmin(fmax(M, -h1), h0);
}

// The PP limiter in its theta form (Eqs. 15-23), as the mass nu Phi^, for an
// interface next to a negative cell, where the clamp above is not the theta
// blend (the unsplit step can leave cells below zero).  A binding theta is
// scaled by (1 - 8 eps) and clamped to [0, 1]; a non-positive denominator
// gives theta = 0, the upwind flux.  Kept out of line so that the rare call
// stays a branch rather than work predicated into every interface.
template <typename T>
__device__ __noinline__ T pp_theta_mass(T phibar, T u0, T u1, T nu) {
    const T tn = T(2) * nu;
    const T up = u0 - tn * phibar, up_up = u0 - tn * u0;
    const T um = u1 + tn * phibar, um_up = u1 + tn * u0;
    T thp = T(1), thm = T(1);
    bool binds = false;
    if (up < T(0)) {
        const T den = up_up - up;
        thp = den > T(0) ? up_up / den : T(0);
        binds = true;
    }
    if (um < T(0)) {
        const T den = um_up - um;
        thm = den > T(0) ? um_up / den : T(0);
        binds = true;
    }
    T th = fmin(thp, thm);
    if (binds) th *= T(1) - T(8) * (sizeof(T) == 4 ? T(5.9604644775390625e-8) : T(1.1102230246251565e-16));
    th = fmin(fmax(th, T(0)), T(1));
    return nu * (th * phibar + (T(1) - th) * u0);
}

// Interface mass on the upwind-ordered stencil (u0 = upwind cell): the CSL
// flux, the MP constraint, times nu, then the PP limiter.  FULL: MP and PP
// both on, so the runtime switches drop out of the loop.
template <typename T, int ORDER, bool FULL>
__device__ __forceinline__ T flux(const LineShift<T> &sh, T um3, T um2, T um1, T u0, T u1, T u2, T u3,
                                  T alpha, int mp, int pp) {
    T phi;
    if ((FULL || mp) && um1 == u0 && u0 == u1) {
        // flat around the interface: every MP bound collapses onto u0, whatever
        // the interpolated value (App. A steps 2-7), so skip computing it
        phi = u0;
    } else {
        if (ORDER == 7) {
            phi = sh.w[0] * um3;
            phi = fma(sh.w[1], um2, phi);
        } else {
            phi = sh.w[1] * um2;
        }
        phi = fma(sh.w[2], um1, phi);
        phi = fma(sh.w[3], u0, phi);
        phi = fma(sh.w[4], u1, phi);
        phi = fma(sh.w[5], u2, phi);
        if (ORDER == 7) phi = fma(sh.w[6], u3, phi);
        if (FULL || mp) phi = mp_limit(phi, um2, um1, u0, u1, u2, alpha);
    }
    T M = mul_rn(sh.nu, phi);
    if (FULL || pp) M = pp_clamp(M, half_rd(u0), half_rd(u1));
    return M;
}

// The CSL interpolant and, for the line walker, the MP constraint as a clamp
// (no branch) with d^{M4} at both faces of u0 passed in.
template <typename T, int ORDER, bool FULL, typename SH>
__device__ __forceinline__ T flux_walk(const SH &sh, T um3, T um2, T um1, T u0, T u1, T u2, T u3,
                                       T alpha, int mp, T m4m, T m4p) {
    T phi;
    if (ORDER == 7) {
        phi = sh.w[0] * um3;
        phi = fma(sh.w[1], um2, phi);
    } else {
        phi = sh.w[1] * um2;
    }
    phi = fma(sh.w[2], um1, phi);
    phi = fma(sh.w[3], u0, phi);
    phi = fma(sh.w[4], u1, phi);
    phi = fma(sh.w[5], u2, phi);
    if (ORDER == 7) phi = fma(sh.w[6], u3, phi);
    if (FULL || mp) phi = mp_clamp(phi, um1, u0, u1, alpha, m4m, m4p);
    return phi;
}

// ---- line walker ---------------------------------------------------------------
//
// Advance cells [r0, r1) of one line staged in shared memory; row r of the
// line is at sm0[r * ss].  Zero-inflow lines have GP >= 1 zero rows on each
// side (rows -GP..-1 and L..L+GP-1); periodic lines wrap.
// The walk goes upwind -> downwind so that each interface mass is computed
// once; the 8-cell stencil window rotates through registers (unrolled by 8).
// The curvature of the upwind cell, d^{M4} at its upwind face and the
// rounded-down half of the cell carry over from one interface to the next, so
// each interface adds one curvature, one d^{M4} and one half.  Where every
// active lane of a warp sits on a flat stencil (u_{-1} = u_0 = u_1) the
// constrained flux is u_0 exactly (all MP bounds collapse onto u_0, d^{M4} at
// the downwind face is 0) and the warp skips the interpolant and the bounds.
// The update is the flux form of Eq. 49 in masses, f' = (u - M_out) + M_in.
// store(i, v) writes the new value of cell i.  NEG: interfaces next to a
// negative cell take the PP limiter's theta form (pp_theta_mass) instead of
// the clamp (scalar T only).  FLAT = false leaves the flat-stencil vote out
// (the same results; for data that is nowhere flat the vote only costs).
// walk_in_place: the store may write the line's own rows (a whole zero-inflow
// line with ghost rows: a row is read before the cell four before it is stored,
// and not again).  walk: what the store writes is not read.

template <typename T, int ORDER, bool PERIODIC, bool FULL, int GP, bool NEG = false, bool FLAT = true,
          typename Store, typename SH>
__device__ __forceinline__ bool walk_in_place(const T *sm0, int ss, int L, const SH &sh,
                                              int r0, int r1, T alpha, int mp, int pp, Store store) {
    if (r0 >= r1) return false;
    // FD: the largest |u| of the segment (high words), for the caller's repeat
    int big = 0;
    auto note = [&](const T &x) {
        if constexpr (std::is_same<T, FD>::value) big = max(big, __double2hiint(x.v) & 0x7fffffff);
    };
    const int sg = sh.sigma;
    const T nu = sh.nu;
    int i = sg > 0 ? r0 : r1 - 1;
    const int cnt = r1 - r0;
    // Source row of load k (k = 0, 1, ...) is p0 + k sg; load k feeds step
    // k - 8 of the walk.
    int p0;
    // Zero-inflow lines read rows outside the staged extent [-GP, L + GP) as
    // the zero row at its edge; periodic lines wrap.  A wrapped row is a line
    // length or two away at most (n is reduced first): additions, where eleven
    // remainders by L cost a short segment as much as its cells.
    auto wrap = [&](int q) {
        while (q < 0) q += L;
        while (q >= L) q -= L;
        return q;
    };
    auto row = [&](int q) -> const T * { return sm0 + min(max(q, -GP), L + GP - 1) * ss; };
    if (PERIODIC) {
        int n = sh.n;
        if (n >= L || n <= -L) n %= L;
        p0 = wrap(i - n - 4 * sg);
    } else {
        p0 = i - sh.n - 4 * sg;
    }
    const T *src = sm0;
    int inc = 0;
    T w[8];
    int pk = p0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        if (PERIODIC) {
            w[k] = sm0[pk * ss];
            pk += sg;
            pk = pk < 0 ? L - 1 : (pk == L ? 0 : pk);
        } else {
            w[k] = *row(p0 + k * sg);
        }
        note(w[k]);
    }
    // incoming mass of the first cell: upwind cell i - sg, stencil w[0..6]
    T dc = T(0), m4m = T(0);  // curvature at the next upwind cell, d^{M4} at its upwind face
    T m4p = T(0);
    if (FULL || mp) {
        const T dm = curv(w[1], w[2], w[3]);
        dc = curv(w[2], w[3], w[4]);
        const T dp = curv(w[3], w[4], w[5]);
        m4m = dm4(dm, dc);
        m4p = dm4(dc, dp);
    }
    // hc: rounded-down half of the cell the walk is on (the upwind cell of its
    // outgoing interface)
    T hc = (FULL || pp) ? half_rd(w[4]) : T(0);
    const T phi0 = flux_walk<T, ORDER, FULL>(sh, w[0], w[1], w[2], w[3], w[4], w[5], w[6], alpha, mp, m4m, m4p);
    T fin = mul_rn(nu, phi0);
    if (FULL || pp) {
        if constexpr (NEG) {
            if (w[3] < T(0) || w[4] < T(0))
                fin = pp_theta_mass(phi0, w[3], w[4], nu);
            else
                fin = pp_clamp(fin, half_rd(w[3]), hc);
        } else {
            fin = pp_clamp(fin, half_rd(w[3]), hc);
        }
    }
    if (FULL || mp) {
        dc = curv(w[3], w[4], w[5]);
        m4m = m4p;
    }

    // one cell with the window rotated by K (u_k at w[(K + 4 + k) & 7]): the
    // constrained flux, the outgoing mass, then f' = (u - M_out) + M_in; the
    // next value enters from *src, which then moves by inc
    auto step = [&](const T &um3, const T &um2, const T &um1, const T &u0_, const T &u1_, const T &u2, const T &u3,
                    bool flat, T &slot) {
        T phi;
        if (FULL || mp) {
            const T dp = curv(u0_, u1_, u2);
            if (flat) {
                phi = u0_;
                m4m = T(0);
            } else {
                m4p = dm4(dc, dp);
                phi = flux_walk<T, ORDER, FULL>(sh, um3, um2, um1, u0_, u1_, u2, u3, alpha, mp, m4m, m4p);
                m4m = m4p;
            }
            dc = dp;
        } else {
            phi = flux_walk<T, ORDER, FULL>(sh, um3, um2, um1, u0_, u1_, u2, u3, alpha, mp, T(0), T(0));
        }
        T fout = mul_rn(nu, phi);
        if (FULL || pp) {
            const T hn = half_rd(u1_);
            if constexpr (NEG) {
                if (u0_ < T(0) || u1_ < T(0))
                    fout = pp_theta_mass(phi, u0_, u1_, nu);
                else
                    fout = pp_clamp(fout, hc, hn);
            } else {
                fout = pp_clamp(fout, hc, hn);
            }
            hc = hn;
        }
        store(i, (u0_ - fout) + fin);
        fin = fout;
        i += sg;
        slot = *src;
        note(slot);
        src += inc;
    };
#define VP_WALK_STEP(K, FLAT_)                                                                             \
    step(w[(K + 1) & 7], w[(K + 2) & 7], w[(K + 3) & 7], w[(K + 4) & 7], w[(K + 5) & 7], w[(K + 6) & 7],   \
         w[(K + 7) & 7], FLAT_, w[K & 7])
    // One vote decides several steps (the vote, its mask and the branch cost as
    // much as ten instructions, and end the overlap of one step's chain with the
    // next): two for a pair of lines (u_{-1} = u_0 = u_1 = u_2), four for one line
    // (.. = u_4, the next value read ahead), of which the first equality is the
    // last of the block before.  Against a vote per step, Plummer 16^3 x 64^3 in
    // an evolved state: pair drifts 1.88 -> 1.86 ms and kicks 1.70 -> 1.62 ms, the
    // contiguous kick (one line) 2.23 -> 2.13 ms; four steps for a pair skip less
    // there (2.00 ms).
    constexpr bool VOTE = FLAT && FlatSkip<T>::on;
    constexpr int NB = std::is_same<T, P2>::value ? 2 : 4;
    const bool vote = VOTE && (FULL || mp);
    bool eqp = w[3] == w[4];
    auto block_flat = [&](const T &a, const T &b, const T &c, const T &d) -> bool {  // u_0 .. u_3
        if constexpr (!VOTE) return false;
        if (!vote) return false;
        bool all = eqp && a == b;
        if constexpr (NB == 2) {
            eqp = b == c;
        } else {
            all = all && b == c && c == d;
            eqp = d == *src;
        }
        return __all_sync(__activemask(), all && eqp);
    };
#define VP_WALK_STEPS(K, FLAT_)                     \
    VP_WALK_STEP(K, FLAT_);                         \
    VP_WALK_STEP(K + 1, FLAT_);                     \
    if constexpr (NB == 4) {                        \
        VP_WALK_STEP(K + 2, FLAT_);                 \
        VP_WALK_STEP(K + 3, FLAT_);                 \
    }
#define VP_WALK_BLOCK(K)                                                                                  \
    if (block_flat(w[(K + 4) & 7], w[(K + 5) & 7], w[(K + 6) & 7], w[(K + 7) & 7])) {                     \
        VP_WALK_STEPS(K, true)                                                                            \
    } else {                                                                                              \
        VP_WALK_STEPS(K, false)                                                                           \
    }

    // The walk runs in chunks over which the load pointer moves uniformly:
    // inside the staged extent it steps one row per cell; beyond it, it stays
    // on the edge row (zero).  A zero-inflow line whose shift keeps every load
    // inside the extent (|n| <= GP - 4) is a single chunk.
    int t = 0;
    while (t < cnt) {
        const int q = p0 + (t + 8) * sg;  // row of the next load
        int end;
        if (PERIODIC) {
            const int qq = wrap(q);
            src = sm0 + qq * ss;
            inc = sg * ss;
            end = t + (sg > 0 ? L - qq : qq + 1);  // loads before the wrap
        } else if (q < -GP || q > L + GP - 1) {
            src = row(q);
            inc = 0;
            const int back = sg > 0 ? -GP - q : q - (L + GP - 1);  // loads until the extent
            end = back > 0 ? t + back : cnt;
        } else {
            src = sm0 + q * ss;
            inc = sg * ss;
            end = t + (sg > 0 ? L + GP - q : q + GP + 1);  // loads through the far edge
        }
        if (end > cnt) end = cnt;
#pragma unroll 1
        for (; t + 8 <= end; t += 8) {
            VP_WALK_BLOCK(0)
            if constexpr (NB == 2) {
                VP_WALK_BLOCK(2)
            }
            VP_WALK_BLOCK(4)
            if constexpr (NB == 2) {
                VP_WALK_BLOCK(6)
            }
        }
#pragma unroll 1
        for (; t < end; ++t) {
            const bool eq = w[4] == w[5];
            if (vote && __all_sync(__activemask(), eqp && eq))
                VP_WALK_STEP(0, true);
            else
                VP_WALK_STEP(0, false);
            eqp = eq;
            // restore the canonical order (u_-4 in w[0])
            const T w0 = w[0];
#pragma unroll
            for (int kk = 0; kk < 7; ++kk) w[kk] = w[kk + 1];
            w[7] = w0;
        }
    }
#undef VP_WALK_STEP
#undef VP_WALK_STEPS
#undef VP_WALK_BLOCK
    return big >= FD::kBig;
}

template <typename T, int ORDER, bool PERIODIC, bool FULL, int GP, bool NEG = false, bool FLAT = true,
          typename Store, typename SH>
__device__ __forceinline__ bool walk(const T *__restrict__ sm0, int ss, int L, const SH &sh, int r0, int r1, T alpha,
                                     int mp, int pp, Store store) {
    return walk_in_place<T, ORDER, PERIODIC, FULL, GP, NEG, FLAT>(sm0, ss, L, sh, r0, r1, alpha, mp, pp, store);
}

// The walk of one line in the arithmetic of its type: FP64 lines with integer
// comparisons, repeated in plain double where the data ask for it (the store
// writes the same cells again).
template <typename T, int ORDER, bool PERIODIC, bool FULL, int GP, bool FLAT, typename MakeStore>
__device__ __forceinline__ void walk_line(const T *sm0, int ss, int L, const LineShift<T> &sh, int r0, int r1,
                                          T alpha, int mp, int pp, MakeStore store) {
    if constexpr (sizeof(T) == 8) {
        if (!walk<FD, ORDER, PERIODIC, FULL, GP, false, FLAT>(reinterpret_cast<const FD *>(sm0), ss, L,
                                                 reinterpret_cast<const LineShift<FD> &>(sh), r0, r1, FD(alpha), mp,
                                                 pp, store(FD())))
            return;
    }
    walk<T, ORDER, PERIODIC, FULL, GP, false, FLAT>(sm0, ss, L, sh, r0, r1, alpha, mp, pp, store(T()));
}

// Shift decomposition of one line, in double precision so that the integer
// part is exact (reading R2): s = c dt / h, n = nearest integer (halves away
// from zero), zeta = s - n, nu = |zeta|, sigma = sign(zeta); the CSL weights
// are the weight polynomials evaluated at nu.
template <typename T>
__device__ __forceinline__ double split_shift(double speed, double dt, double h, LineShift<T> &sh) {
    const double s = __ddiv_rn(__dmul_rn(speed, dt), h);
    double n = round(s);
    const double z = __dadd_rn(s, -n);
    const double nu = fabs(z);
    // shifts beyond a billion cells only happen with absurd inputs; clamp so
    // the integer conversion stays defined (a zero-inflow line is empty anyway)
    n = fmin(fmax(n, -1.0e9), 1.0e9);
    sh.nu = (T)nu;
    sh.n = (int)n;
    sh.sigma = z < 0.0 ? -1 : 1;
    return nu;
}
__device__ __forceinline__ double csl_weight(const WPoly &wp, int k, double nu) {
    double acc = 0.0;
    for (int j = wp.nterm - 1; j >= 0; --j) acc = fma(acc, nu, wp.c[j][k]);
    return acc;
}
// velocity of cell j of an axis: lo + (j + 1/2) dv, rounded step by step
__device__ __forceinline__ double cell_centre(double lo, double dvel, int j) {
    return __dadd_rn(lo, __dmul_rn((double)j + 0.5, dvel));
}

__device__ __forceinline__ unsigned line_class(const SweepGeo &g, unsigned o, unsigned c) {
    return g.cls_from_inner ? fmod_u(fdiv(c, g.fd_cdiv), g.fd_cmod) : fdiv(o, g.fd_cdiv);
}

// Where a sweep's lines get their shifts: a table with one entry per class,
// or (tab == NULL) from the speeds themselves, decomposed by every CTA for the
// `ncl` consecutive classes (at most) that its tile meets.  The same numbers
// either way.
template <typename T>
struct ShiftSrc {
    const LineShift<T> *tab;
    const double *accel;  // kick: speed of class c is accel[c]; NULL: drift, cell c of the velocity axis
    double lo, dvel, dt, h;
    int ncl;
    WPoly wp;
};

// bytes of shared memory behind a tile of `tile` bytes for ncl shifts
template <typename T>
__host__ __device__ inline size_t shift_smem(size_t tile, int ncl) {
    return ncl ? ((tile + 15) & ~size_t(15)) - tile + (size_t)ncl * (sizeof(LineShift<T>) + sizeof(double)) : 0;
}

// The tile's shifts s[0..ncl), class (q0 + i) mod cmod (no mod for kicks).  Up
// to four classes: eight lanes each of the first warp, every lane splitting the
// shift and taking one weight.  More: the split first (tile_shifts, before the
// tile's barrier), the weights spread over the block after it (tile_weights,
// followed by a barrier of its own): 32 classes cost 1200 cycles of the FP64
// pipe, where one thread per class took 1200 by itself and its own launch.
template <typename T>
__device__ __forceinline__ double class_speed(const ShiftSrc<T> &src, const SweepGeo &g, unsigned q) {
    return src.accel ? src.accel[q] : cell_centre(src.lo, src.dvel, (int)fmod_u(q, g.fd_cmod));
}
template <typename T>
__device__ __forceinline__ void tile_shifts(LineShift<T> *s, unsigned q0, int ncl, const ShiftSrc<T> &src,
                                            const SweepGeo &g) {
    double *nus = reinterpret_cast<double *>(s + src.ncl);
    if (src.ncl <= 4) {
        const int i = threadIdx.x >> 3, k = threadIdx.x & 7;
        if (i < ncl) {
            LineShift<T> sh;
            const double nu = split_shift(class_speed(src, g, q0 + i), src.dt, src.h, sh);
            if (k < 7) {
                s[i].w[k] = (T)csl_weight(src.wp, k, nu);
            } else {
                s[i].nu = sh.nu;
                s[i].n = sh.n;
                s[i].sigma = sh.sigma;
            }
        }
    } else {
        for (int i = threadIdx.x; i < ncl; i += blockDim.x) {
            LineShift<T> sh;
            nus[i] = split_shift(class_speed(src, g, q0 + i), src.dt, src.h, sh);
            s[i].nu = sh.nu;
            s[i].n = sh.n;
            s[i].sigma = sh.sigma;
        }
    }
}
template <typename T>
__device__ __forceinline__ void tile_weights(LineShift<T> *s, int ncl, const ShiftSrc<T> &src) {
    if (src.ncl <= 4) return;
    const double *nus = reinterpret_cast<const double *>(s + src.ncl);
    for (int t = threadIdx.x; t < 7 * ncl; t += blockDim.x) {
        const int i = t / 7, k = t - 7 * i;
        s[i].w[k] = (T)csl_weight(src.wp, k, nus[i]);
    }
    __syncthreads();
}

}  // namespace vp_core
