// nci.cu -- batched FP64 root solver of the numerical dispersion relation of
// a relativistically drifting cold plasma on the hybrid solver's grid (the
// Appendix: Eq. 2dmodesres with the coupling term, the hybrid operators
// [k]E1 = [k]B1 = k1 (plus the Sec. 4 bump), [k]E2 = [k]B2 =
// sin(k2 dx2/2)/(dx2/2), and the cubic Eq. asym1 about the beam resonance).
//
// The roots sought for a (sample, alias) are all zeros of
//   G(w) = [w] D(w) (w' - k1' v0)
// (the relation times the factors that remove its poles: G is entire) in the
// disk |w - w_res| < rho about the beam resonance w' = k1' v0, with
// rho = (wp2/gamma)^(1/3), the scale at which the cubic's leading and
// constant terms balance.  The growth rate of the alias is the largest Im w
// over them (0 if none grows); a sample's growth is the largest over its
// aliases.
//
//  1. The number N of zeros in the disk: the winding of G along the circle
//     (phase steps sampled until none exceeds 0.5 rad).
//  2. Newton's method with G' from the product rule, deflated by the zeros
//     already found (step 1 / (G'/G - sum 1/(w - r_j)), so no zero is found
//     twice), from seeds: the cubic's roots, the resonance itself and rings
//     inside the disk; done when N zeros inside the disk are found.
//  3. If the seeds leave zeros unfound, the rectangle around the disk is split
//     into four pieces whose zeros are counted by their boundary's winding,
//     recursively, and Newton's method is run inside each piece that holds
//     one zero (complete by construction).
//
// A warp takes a group of up to 32 (sample, alias) pairs.  The FP64 pipe bounds
// it (a warp-wide FP64 instruction occupies it for the same time with one live
// lane or with 32), so the work is laid out to keep lanes live: the windings
// with the contour's points across the lanes, one pair after the other; the
// cubic's and the resonance's seeds with one pair per lane; the ring seeds and
// the subdivision, which few pairs need but each for a long time, again one pair
// at a time with seeds and contour points across the lanes.  With one thread per
// pair doing all of it (before), the few hard pairs ran alone for tens of
// milliseconds, 3.6 of 32 lanes live: 69 ms for 32256 samples x 3 aliases, 6.1 ms now, of which
// the counts take a third and the cubic's seeds most of the rest.
//
// Readings (the printed forms are garbled here): s_{l,i} = sinc(k'_i dx_i/2)^(l+1)
// with k' aliased; S_B3 = S'_B3 cos(w dt/2), B's time centring, whose
// expansion about the resonance is the cubic's zeta0 + zeta1 dw'; the current
// filter F(k1) and the j1 correction multiply S_j1, F multiplies S_j2;
// momentum-conserving interpolation.
#include <math.h>

#include "hyb_internal.cuh"

namespace hyb {

struct Z { double re, im; };
__device__ __forceinline__ Z zc(double a, double b) { Z z; z.re = a; z.im = b; return z; }
__device__ __forceinline__ Z zadd(Z a, Z b) { return zc(a.re + b.re, a.im + b.im); }
__device__ __forceinline__ Z zsub(Z a, Z b) { return zc(a.re - b.re, a.im - b.im); }
__device__ __forceinline__ Z zmul(Z a, Z b) { return zc(a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re); }
__device__ __forceinline__ Z zsc(Z a, double s) { return zc(a.re * s, a.im * s); }
__device__ __forceinline__ Z zdiv(Z a, Z b) {
    // scaled division (Smith's method)
    if (fabs(b.re) >= fabs(b.im)) {
        const double r = b.im / b.re, d = b.re + b.im * r;
        return zc((a.re + a.im * r) / d, (a.im - a.re * r) / d);
    }
    const double r = b.re / b.im, d = b.re * r + b.im;
    return zc((a.re * r + a.im) / d, (a.im * r - a.re) / d);
}
__device__ __forceinline__ double zabs(Z a) { return hypot(a.re, a.im); }

__device__ __forceinline__ double dsinc(double x) { return x == 0.0 ? 1.0 : sin(x) / x; }

// The symbols of one (sample, alias).
struct NciMode {
    double h, rh, v0, b, muwg, res, kE1, kE2, k2, SE1, SE2, SB3s, Sj1, Sj2;
    double K2, as, sb, sk, c1, c2, c3, c4;      // the products G uses (see nci_G)
    double c, sc, cc;                           // the resonance, sin(c h), cos(c h)
};

// SIGN = -1: sin x and cos x, SIGN = 1: sinh x and cosh x, by Taylor series for |x| <= 1/2
template <int SIGN>
__device__ __forceinline__ void taylor_trig(double x, double* s, double* c) {
    const double z = SIGN * x * x;
    double a = 1.0 / 1307674368000.0, b = 1.0 / 20922789888000.0;      // 1/15!, 1/16!
    a = fma(a, z, 1.0 / 6227020800.0);  b = fma(b, z, 1.0 / 87178291200.0);
    a = fma(a, z, 1.0 / 39916800.0);    b = fma(b, z, 1.0 / 479001600.0);
    a = fma(a, z, 1.0 / 362880.0);      b = fma(b, z, 1.0 / 3628800.0);
    a = fma(a, z, 1.0 / 5040.0);        b = fma(b, z, 1.0 / 40320.0);
    a = fma(a, z, 1.0 / 120.0);         b = fma(b, z, 1.0 / 720.0);
    a = fma(a, z, 1.0 / 6.0);           b = fma(b, z, 1.0 / 24.0);
    b = fma(b, z, 0.5);
    *s = fma(a * z, x, x);
    *c = fma(b, z, 1.0);
}

// G(w) and G'(w).  With u = w h (h = dt/2): [w] = sin(u)/h, c = cos(u) (B's time
// centring), d[w]/dw = c, dc/dw = -h sin(u) = -h^2 [w].
//   A = [w] (Delta^2) - a Sj1 SE1 w'                                 ([w] x first factor)
//   S = ([w]^2 - K2) Delta - b Sj2 (SE2 [w] - SB3 kE1 v0)             (second factor x Delta)
//   C = b (Sj1 SE1 w' kE2^2 (v0^2 - 1) + Sj2 SE2 kE2^2 Delta
//          + Sj1 kE2 k2 (SE2 kE1 v0 - SB3 v0^2 [w]))                  ([w] x coupling term)
//   G = A S + C Delta,  SB3 = SB3s c.
template <bool DERIV>
__device__ __forceinline__ void nci_G(const NciMode& m, Z w, Z* g, Z* dg) {
    // sin and cos of Re w h = c h + d and sinh and cosh of y = Im w h.  Near the resonance (|d|, |y| <=
    // 1/2: the disk, as long as rho h <= 1/2) from their Taylor series (to x^15 and x^16: the first
    // term left out is below 1e-18) and the addition theorem, about a third of the FP64 instructions of
    // the calls elsewhere
    double su, cu, sh, ch;
    const double d = (w.re - m.c) * m.h, y = w.im * m.h;
    if (fabs(d) <= 0.5 && fabs(y) <= 0.5) {
        double sd, cd;
        taylor_trig<-1>(d, &sd, &cd);
        taylor_trig<1>(y, &sh, &ch);
        su = m.sc * cd + m.cc * sd;
        cu = m.cc * cd - m.sc * sd;
    } else {
        sincos(w.re * m.h, &su, &cu);
        sh = sinh(y);
        ch = cosh(y);
    }
    const Z sn = zc(su * ch, cu * sh);                  // sin(w h)
    const Z cs = zc(cu * ch, -su * sh);                 // cos(w h)
    const Z wb = zsc(sn, m.rh);
    const Z wp = zc(w.re + m.muwg, w.im);
    const Z D = zc(wp.re - m.res, wp.im);               // Delta; dDelta/dw = 1, dw'/dw = 1
    const Z D2 = zmul(D, D);
    const Z A = zsub(zmul(wb, D2), zsc(wp, m.as));
    const Z wb2K = zsub(zmul(wb, wb), zc(m.K2, 0.0));
    const Z S = zsub(zmul(wb2K, D), zsc(zsub(zsc(wb, m.SE2), zsc(cs, m.sk)), m.sb));
    const Z C = zsub(zadd(zadd(zsc(wp, m.c1), zsc(D, m.c2)), zc(m.c3, 0.0)), zsc(zmul(cs, wb), m.c4));
    *g = zadd(zmul(A, S), zmul(C, D));
    if (DERIV) {
        const Z dcs = zsc(sn, -m.h);
        const Z dA = zsub(zadd(zmul(cs, D2), zsc(zmul(wb, D), 2.0)), zc(m.as, 0.0));
        const Z dS = zsub(zadd(zsc(zmul(zmul(wb, cs), D), 2.0), wb2K), zsc(zsub(zsc(cs, m.SE2), zsc(dcs, m.sk)), m.sb));
        const Z dC = zsub(zc(m.c1 + m.c2, 0.0), zsc(zadd(zmul(dcs, wb), zmul(cs, cs)), m.c4));
        *dg = zadd(zadd(zadd(zmul(dA, S), zmul(A, dS)), zmul(dC, D)), C);
    }
}

// Winding number of G along a closed polyline given by point(i), i = 0..n (point(n) =
// point(0)), with the number of points raised until no phase step exceeds 0.5 rad.
// Returns -1 if no sampling up to kMaxWind points resolves it (a zero on the path).
// Called by the whole warp with one mode: the lanes take consecutive points, 32 at a time.
// A step from g0 to g1 is below 0.5 rad when Re(g1 conj g0) > 0 and |Im| <= tan(0.5) Re; the
// steps' sum over 2 pi is the signed number of crossings of the negative real axis, which such a
// step makes exactly when Im g changes sign at Re g < 0 (no arc tangent needed).
constexpr int kMaxWind = 1 << 13;
template <typename Path>
__device__ int winding(const NciMode& m, Path path, int n0) {
    constexpr double kTan = 0.54630248984379051326;      // tan(0.5)
    const int lane = threadIdx.x & 31;
    for (int n = n0; n <= kMaxWind; n *= 4) {
        Z first = zc(0.0, 0.0), last = zc(0.0, 0.0);
        int cross = 0;
        bool ok = true, undefined = false;
        for (int i0 = 0; i0 <= n && ok; i0 += 32) {
            const int i = i0 + lane;
            Z g = first;                                  // point n is point 0
            if (i0 < n) nci_G<false>(m, path(i, n), &g, nullptr);
            Z p = zc(__shfl_up_sync(0xffffffffu, g.re, 1), __shfl_up_sync(0xffffffffu, g.im, 1));
            if (lane == 0) p = last;
            bool bad = false, nan = false;
            if (i0 + lane > 0 && i0 + lane <= n) {
                const double re = g.re * p.re + g.im * p.im, im = g.im * p.re - g.re * p.im;
                nan = isnan(re) || isnan(im);
                bad = !nan && !(re > 0.0 && fabs(im) <= kTan * re);
                if (p.re < 0.0) cross += (p.im >= 0.0 && g.im < 0.0) ? 1 : (p.im < 0.0 && g.im >= 0.0) ? -1 : 0;
            }
            ok = !__any_sync(0xffffffffu, bad);
            undefined = undefined || __any_sync(0xffffffffu, nan);
            if (i0 == 0) first = zc(__shfl_sync(0xffffffffu, g.re, 0), __shfl_sync(0xffffffffu, g.im, 0));
            last = zc(__shfl_sync(0xffffffffu, g.re, 31), __shfl_sync(0xffffffffu, g.im, 31));
        }
        if (ok) return undefined ? 0 : __reduce_add_sync(0xffffffffu, cross);
    }
    return -1;
}

// The same along a circle about a point c of the real axis.  G is real there (its coefficients are
// real), so G(conj w) = conj G(w) and only the points i = 0..n/2 of the upper half are evaluated;
// each step counts with its mirror step.  (zx, zy): cos and sin of the lane's point for n = 64;
// end: G(c - r), the point n/2.
__device__ int winding_circle(const NciMode& m, double c, double r, double zx, double zy, Z end) {
    constexpr double kTan = 0.54630248984379051326;
    const int lane = threadIdx.x & 31;
    for (int n = 64; n <= kMaxWind; n *= 4) {
        Z last = zc(0.0, 0.0);
        int cross = 0;
        bool ok = true, undefined = false;
        for (int i0 = 0; i0 < n / 2 && ok; i0 += 32) {
            if (n > 64) sincospi(2.0 * (i0 + lane) / (double)n, &zy, &zx);
            Z g;
            nci_G<false>(m, zc(c + r * zx, r * zy), &g, nullptr);
            bool bad = false, nan = false;
            auto step = [&](Z a, Z b) {                               // from a to b, and from conj b to conj a
                const double re = b.re * a.re + b.im * a.im, im = b.im * a.re - b.re * a.im;
                const bool undef = isnan(re) || isnan(im);
                nan |= undef;
                bad |= !undef && !(re > 0.0 && fabs(im) <= kTan * re);
                if (a.re < 0.0) cross += (a.im >= 0.0 && b.im < 0.0) ? 1 : (a.im < 0.0 && b.im >= 0.0) ? -1 : 0;
                if (b.re < 0.0) cross += (-b.im >= 0.0 && -a.im < 0.0) ? 1 : (-b.im < 0.0 && -a.im >= 0.0) ? -1 : 0;
            };
            Z p = zc(__shfl_up_sync(0xffffffffu, g.re, 1), __shfl_up_sync(0xffffffffu, g.im, 1));
            if (lane == 0) p = last;
            if (i0 + lane > 0) step(p, g);
            if (i0 + 32 == n / 2 && lane == 31) step(g, end);
            ok = !__any_sync(0xffffffffu, bad);
            undefined = undefined || __any_sync(0xffffffffu, nan);
            last = zc(__shfl_sync(0xffffffffu, g.re, 31), __shfl_sync(0xffffffffu, g.im, 31));
        }
        if (ok) return undefined ? 0 : __reduce_add_sync(0xffffffffu, cross);
    }
    return -1;
}
__device__ int winding_rect(const NciMode& m, double x0, double x1, double y0, double y1) {
    return winding(m, [&](int i, int n) {
        // n points, n/4 per edge, counter-clockwise from (x0, y0)
        const int q = n / 4, e = i / q;
        const double t = (double)(i - e * q) / (double)q;
        if (e == 0) return zc(x0 + (x1 - x0) * t, y0);
        if (e == 1) return zc(x1, y0 + (y1 - y0) * t);
        if (e == 2) return zc(x1 - (x1 - x0) * t, y1);
        return zc(x0, y1 - (y1 - y0) * t);
    }, 128);
}

// One attempt of Newton's method on G deflated by the nf zeros in r[], advanced one step per call:
// 0 = go on, 1 = converged to w, -1 = failed.  An attempt has MAX steps.  Each step is a
// function of w alone, so an attempt that meets a w it has seen (kept at steps 1, 2, 4, 8, ...:
// a limit cycle at rounding level) can never converge and fails at once.
constexpr int kNewtonMax = 80, kNewtonFirst = 40;   // the latter for the first seeds (step 2a)
struct Newton { Z w, seen; int it; };
__device__ __forceinline__ Newton newton_start(Z w) { return Newton{w, zc(nan(""), 0.0), 0}; }
template <int MAX>
__device__ __forceinline__ int newton_step(const NciMode& m, Newton& s, const Z* r, int nf) {
    Z g, dg;
    nci_G<true>(m, s.w, &g, &dg);
    if (g.re == 0.0 && g.im == 0.0) return 1;
    // step = 1 / (G'/G - sum 1/(w - r_j)) = G / (G' - G sum)
    Z sum = zc(0.0, 0.0);
    for (int j = 0; j < nf; j++) {
        const Z d = zsub(s.w, r[j]);
        const double q = 1.0 / (d.re * d.re + d.im * d.im);
        sum = zc(sum.re + d.re * q, sum.im - d.im * q);
    }
    const Z den = zsub(dg, zmul(g, sum));
    if (den.re == 0.0 && den.im == 0.0) return -1;
    const Z step = zdiv(g, den);
    s.w = zsub(s.w, step);
    if (!(isfinite(s.w.re) && isfinite(s.w.im))) return -1;
    // |step| <= 1e-14 max(1, |w|)
    if (step.re * step.re + step.im * step.im <= 1e-28 * fmax(1.0, s.w.re * s.w.re + s.w.im * s.w.im)) return 1;
    if (++s.it == MAX || (s.w.re == s.seen.re && s.w.im == s.seen.im)) return -1;
    if ((s.it & (s.it - 1)) == 0) s.seen = s.w;
    return 0;
}
__device__ bool newton_deflated(const NciMode& m, Z w, const Z* r, int nf, Z* out) {
    Newton s = newton_start(w);
    int st;
    while ((st = newton_step<kNewtonMax>(m, s, r, nf)) == 0) {}
    *out = s.w;
    return st > 0;
}

// Plain Newton's method for one zero inside a rectangle.
__device__ bool newton_in(const NciMode& m, Z w, double x0, double x1, double y0, double y1, Z* out) {
    Z r;
    if (!newton_deflated(m, w, nullptr, 0, &r)) return false;
    if (r.re < x0 || r.re > x1 || r.im < y0 || r.im > y1) return false;
    *out = r;
    return true;
}

constexpr int kMaxRoots = 16;   // zeros kept per (sample, alias); more is reported as an error
constexpr int kStack = 96;      // subdivision stack entries

// the cubic a x^3 + b x^2 + c x + d = 0 (a != 0) by the trigonometric / Cardano forms
__device__ void cubic_roots(double a, double b, double c, double d, Z r[3]) {
    const double A = b / a, B = c / a, C = d / a;
    const double Q = (3.0 * B - A * A) / 9.0, R = (9.0 * A * B - 27.0 * C - 2.0 * A * A * A) / 54.0;
    const double D = Q * Q * Q + R * R;
    if (D >= 0.0) {
        const double sD = sqrt(D);
        const double S = cbrt(R + sD), T = cbrt(R - sD);
        r[0] = zc(-A / 3.0 + (S + T), 0.0);
        r[1] = zc(-A / 3.0 - 0.5 * (S + T), 0.5 * sqrt(3.0) * (S - T));
        r[2] = zc(-A / 3.0 - 0.5 * (S + T), -0.5 * sqrt(3.0) * (S - T));
    } else {
        const double th = acos(R / sqrt(-Q * Q * Q));
        const double sq = 2.0 * sqrt(-Q);
        const double pi = 3.14159265358979323846;
        r[0] = zc(sq * cos(th / 3.0) - A / 3.0, 0.0);
        r[1] = zc(sq * cos((th + 2.0 * pi) / 3.0) - A / 3.0, 0.0);
        r[2] = zc(sq * cos((th + 4.0 * pi) / 3.0) - A / 3.0, 0.0);
    }
}

// one row of the samples array
struct NciSample { double dt, dx1, dx2, gamma, wp2, filt_kc, filt_w, k1, k2, kmod_l, kmod_u, kmod_max; };

__device__ double filt_factor(const NciSample& s) {
    if (!(s.filt_kc > 0.0 && s.filt_kc < 1.0)) return 1.0;
    const double pi = 3.14159265358979323846, kn = pi / s.dx1, k = fabs(s.k1);
    const double kc = s.filt_kc * kn, w = s.filt_w * kn;
    if (k <= kc - 0.5 * w) return 1.0;
    if (k >= kc + 0.5 * w) return 0.0;
    const double c = cos(0.5 * pi * (k - kc + 0.5 * w) / w);
    return c * c;
}

// [k]E1 = [k]B1: k1 plus the Sec. 4 raised-cosine bump between kmod_l and kmod_u (fractions of 2 pi/dx1)
__device__ double k_eff(const NciSample& s) {
    double k = s.k1;
    if (s.kmod_max != 0.0) {
        const double pi = 3.14159265358979323846, kg = 2.0 * pi / s.dx1;
        const double kl = s.kmod_l * kg, ku = s.kmod_u * kg, km = 0.5 * (kl + ku), a = fabs(s.k1);
        if (a >= kl && a <= ku) {
            const double c = cos(0.5 * pi * (a - km) / (kl - km));
            k += copysign(s.kmod_max * kg * c * c, s.k1);
        }
    }
    return k;
}

// error bits of k_nci (the kernel's *err)
enum : int { NCI_ETOOMANY = 1, NCI_EUNRESOLVED = 2 };

// the symbols of a pair, its resonance c (real) and the disk's radius
__device__ void nci_symbols(const NciSample& s, int mu, int nu1, int order, int correct_j1, NciMode& m, double* c, double* rho,
                            double* k1a_out) {
    const double pi = 3.14159265358979323846;
    m.h = 0.5 * s.dt;
    m.rh = 1.0 / m.h;
    m.v0 = sqrt(1.0 - 1.0 / (s.gamma * s.gamma));
    const double wg = 2.0 * pi / s.dt;
    m.muwg = mu * wg;
    const double sgnmu = (mu & 1) ? -1.0 : 1.0;
    const double a = s.wp2 / (s.gamma * s.gamma * s.gamma) * sgnmu;
    m.b = s.wp2 / s.gamma * sgnmu;
    m.k2 = s.k2;
    const double k1a = s.k1 + nu1 * 2.0 * pi / s.dx1;
    const double s1 = dsinc(0.5 * k1a * s.dx1), s2 = dsinc(0.5 * s.k2 * s.dx2);
    double sl1 = s1, sl2 = s2, sm1 = 1.0, sm2 = 1.0;                 // orders l + 1 and l
    for (int q = 0; q < order; q++) { sl1 *= s1; sl2 *= s2; sm1 *= s1; sm2 *= s2; }
    const double sgn = (nu1 & 1) ? -1.0 : 1.0;
    m.kE1 = k_eff(s);
    m.kE2 = sin(0.5 * s.k2 * s.dx2) / (0.5 * s.dx2);
    m.SE1 = sl1 * sl2 * sgn;
    m.SE2 = sl1 * sl2;
    m.SB3s = sl1 * sl2 * sgn;
    const double F = filt_factor(s);
    const double corr = (correct_j1 && s.k1 != 0.0) ? dsinc(0.5 * s.k1 * s.dx1) * s.k1 / m.kE1 : 1.0;
    m.Sj1 = sm1 * sl2 * sgn * F * corr;
    m.Sj2 = sl1 * sm2 * F;
    m.res = k1a * m.v0;
    const double kE2s = m.kE2 * m.kE2;
    m.K2 = m.kE1 * m.kE1 + kE2s;
    m.as = a * m.Sj1 * m.SE1;
    m.sb = m.b * m.Sj2;
    m.sk = m.SB3s * m.kE1 * m.v0;
    m.c1 = m.b * m.Sj1 * m.SE1 * kE2s * (m.v0 * m.v0 - 1.0);
    m.c2 = m.b * m.Sj2 * m.SE2 * kE2s;
    m.c3 = m.b * m.Sj1 * m.kE2 * m.k2 * m.SE2 * m.kE1 * m.v0;
    m.c4 = m.b * m.Sj1 * m.kE2 * m.k2 * m.SB3s * m.v0 * m.v0;
    m.c = *c = m.res - m.muwg;
    sincos(m.c * m.h, &m.sc, &m.cc);
    *rho = cbrt(s.wp2 / s.gamma);
    *k1a_out = k1a;
}

// the cubic of Eq. asym1 (v0 -> 1 in k~1) about the resonance; false if it has no leading term
__device__ bool nci_cubic(const NciMode& m, double k1a, Z cub[3]) {
    const double kt = k1a - m.muwg, hh = m.h;
    const double xi0 = sin(kt * hh) / hh, xi1 = cos(kt * hh), ze0 = cos(kt * hh), ze1 = -sin(kt * hh) * hh;
    const double kE1 = m.kE1, kE2 = m.kE2, SB = m.SB3s;
    const double A2 = 2.0 * xi0 * xi0 * xi0 * xi1;
    const double B2 = xi0 * xi0 * (xi0 * xi0 - kE1 * kE1 - kE2 * kE2 - m.b * m.Sj2 * (m.SE2 * xi1 - ze1 * SB * kE1));
    const double C2 = m.b * (xi0 * xi0 * m.Sj2 * (ze0 * SB * kE1 - m.SE2 * xi0) - xi1 * m.Sj1 * kE2 * m.k2 * m.SE2 * kE1
                             + xi0 * kE2 * (m.Sj2 * m.SE2 * kE2 - m.Sj1 * m.k2 * ze1 * SB * xi0));
    const double D2 = m.b * xi0 * kE2 * m.k2 * m.Sj1 * (m.SE2 * kE1 - ze0 * SB * xi0);
    if (A2 == 0.0) return false;
    cubic_roots(A2, B2, C2, D2, cub);
    return true;
}

// a zero this far from the real axis (in units of rho) and its conjugate are two: nearer ones could be
// one real zero's rounding
constexpr double kPairIm = 1e-4;
constexpr int kRing = 8, kRingSeeds = 3 * kRing;      // three rings of seeds inside the disk

// Step 3 for one pair, by the whole warp (every lane with the same values; the windings' points
// across the lanes): the zeros of the disk by subdivision of a rectangle around it.
__device__ int nci_subdivide(const NciMode& m, Z c, double rho, Z* r, int* e) {
    int nf = 0;
    const double fr[4][2] = {{0.4871, 0.5317}, {0.4413, 0.5689}, {0.5593, 0.4231}, {0.3917, 0.6143}};
    const double hmin = fmax(1e-12 * rho, 1e-9 * fmax(1.0, zabs(c)));
    const double x0 = c.re - rho, x1 = c.re + 1.0007 * rho, y0 = c.im - 1.0003 * rho, y1 = c.im + 1.0011 * rho;
    const int Nr = winding_rect(m, x0, x1, y0, y1);
    if (Nr < 0) *e |= NCI_EUNRESOLVED;
    struct Rect { double x0, x1, y0, y1; int N; };
    Rect st[kStack];
    int sp = 0;
    if (Nr > 0) st[sp++] = Rect{x0, x1, y0, y1, Nr};
    auto keep = [&](Z w) {
        if (nf < kMaxRoots) {
            __syncwarp();
            if ((threadIdx.x & 31) == 0) r[nf] = w;
            nf++;
        } else {
            *e |= NCI_ETOOMANY;
        }
    };
    while (sp > 0) {
        const Rect q = st[--sp];
        if (q.N == 1) {
            Z w;
            if (newton_in(m, zc(q.x0 + fr[0][0] * (q.x1 - q.x0), q.y0 + fr[0][1] * (q.y1 - q.y0)), q.x0, q.x1, q.y0, q.y1, &w)) {
                if (zabs(zsub(w, c)) < rho) keep(w);
                continue;
            }
        }
        if (fmax(q.x1 - q.x0, q.y1 - q.y0) < hmin) {          // a cluster below resolution
            const Z w = zc(0.5 * (q.x0 + q.x1), 0.5 * (q.y0 + q.y1));
            if (zabs(zsub(w, c)) < rho)
                for (int k = 0; k < q.N; k++) keep(w);
            continue;
        }
        bool split = false;
        for (int f = 0; f < 4 && !split; f++) {
            const double xm = q.x0 + fr[f][0] * (q.x1 - q.x0), ym = q.y0 + fr[f][1] * (q.y1 - q.y0);
            const Rect kid[4] = {{q.x0, xm, q.y0, ym, 0}, {xm, q.x1, q.y0, ym, 0}, {q.x0, xm, ym, q.y1, 0}, {xm, q.x1, ym, q.y1, 0}};
            int ns[4], tot = 0;
            bool ok = true;
            for (int k = 0; k < 4 && ok; k++) {
                ns[k] = winding_rect(m, kid[k].x0, kid[k].x1, kid[k].y0, kid[k].y1);
                ok = ns[k] >= 0;
                tot += ns[k];
            }
            if (!ok || tot != q.N) continue;
            split = true;
            for (int k = 0; k < 4; k++) {
                if (ns[k] == 0) continue;
                if (sp >= kStack) { *e |= NCI_EUNRESOLVED; break; }
                st[sp] = kid[k];
                st[sp].N = ns[k];
                sp++;
            }
        }
        if (!split) *e |= NCI_EUNRESOLVED;
    }
    __syncwarp();
    return nf;
}

// A warp (block of kNciThreads / 32 of them) per `group` consecutive pairs (group <= 32, a lane each).
constexpr int kNciThreads = 64;
__global__ void __launch_bounds__(kNciThreads) k_nci(const NciSample* __restrict__ smp, int64_t n, int order, int correct_j1,
                                                     const int* __restrict__ alias, int n_alias, int group,
                                                     double* __restrict__ growth, double2* __restrict__ root, int max_out,
                                                     double2* __restrict__ roots_out, int* __restrict__ count_out,
                                                     int* __restrict__ err) {
    __shared__ NciMode modes[kNciThreads / 32][32];
    __shared__ Z roots[kNciThreads / 32][32][kMaxRoots];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t first = ((int64_t)blockIdx.x * (kNciThreads / 32) + warp) * group;
    const int64_t tid = first + lane, total = n * n_alias;
    const bool live = lane < group && tid < total;
    if (first >= total) return;                                     // the whole warp
    NciMode& m = modes[warp][lane];
    Z* const r = roots[warp][lane];
    double c = 0.0, rho = 0.0, k1a = 0.0;
    int nf = 0, N = 0, e = 0;
    if (live) {
        const int ai = (int)(tid % n_alias);
        nci_symbols(smp[tid / n_alias], alias[2 * ai], alias[2 * ai + 1], order, correct_j1, m, &c, &rho, &k1a);
    }
    __syncwarp();
    // ---- 1. the count, one pair after the other
    double zx, zy;
    sincospi(2.0 * lane / 64.0, &zy, &zx);
    Z end = zc(0.0, 0.0);
    if (live && rho > 0.0) nci_G<false>(m, zc(c - rho, 0.0), &end, nullptr);
    for (unsigned todo = __ballot_sync(0xffffffffu, live && rho > 0.0); todo; todo &= todo - 1) {
        const int j = __ffs(todo) - 1;
        const int w = winding_circle(modes[warp][j], __shfl_sync(0xffffffffu, c, j), __shfl_sync(0xffffffffu, rho, j), zx, zy,
                                     zc(__shfl_sync(0xffffffffu, end.re, j), __shfl_sync(0xffffffffu, end.im, j)));
        if (lane == j) N = w;
    }
    if (N < 0 || N > kMaxRoots) { e |= (N < 0) ? NCI_EUNRESOLVED : NCI_ETOOMANY; N = 0; }
    // ---- 2a. the cubic's roots inside the disk and the resonance as seeds, a pair per lane; one
    // Newton step of every lane's current attempt per turn.  An attempt that converges does so in some ten
    // steps; one that has not after kNewtonFirst would keep the other lanes waiting (with 80 a warp took 72 turns at
    // 8.3 live lanes), and the rings find what it would have.
    {
        Z cub[3];
        bool have = false;
        if (N > 0) have = nci_cubic(m, k1a, cub);
        int q = -1;
        bool skip = false;                                          // the next seed is the last one's conjugate, done
        Newton s = newton_start(zc(0.0, 0.0));
        auto next = [&]() {                                         // the next seed, or q = 4 when done
            if (nf >= N) { q = 4; return; }
            for (q += skip ? 2 : 1, skip = false; q < 4; q++) {
                if (q == 3) { s = newton_start(zc(c + 1e-6 * rho, 1e-7 * rho)); return; }
                const Z w0 = q == 0 ? cub[0] : q == 1 ? cub[1] : cub[2];
                if (have && zabs(zsub(zc(c + w0.re, w0.im), zc(c, 0.0))) < rho) { s = newton_start(zc(c + w0.re, w0.im)); return; }
            }
        };
        next();
        while (__any_sync(0xffffffffu, q < 4)) {
            if (q < 4) {
                const int st = newton_step<kNewtonFirst>(m, s, r, nf);
                if (st > 0 && zabs(zsub(s.w, zc(c, 0.0))) < rho) {
                    r[nf++] = s.w;
                    // G's coefficients are real: the conjugate of a zero well off the real axis is another
                    if (nf < N && fabs(s.w.im) > kPairIm * rho) {
                        r[nf++] = zc(s.w.re, -s.w.im);
                        skip = q == 1;
                    }
                }
                if (st != 0) next();
            }
            __syncwarp();
        }
    }
    // ---- 2b. the rings, one pair after the other, a seed per lane.  The first attempt that finds a zero adds it to
    // the deflation, and all start again from their seeds (one that went on from beside that zero could
    // end on it once more)
    for (unsigned todo = __ballot_sync(0xffffffffu, nf < N); todo; todo &= todo - 1) {
        const int j = __ffs(todo) - 1;
        const NciMode& mj = modes[warp][j];
        Z* const rj = roots[warp][j];
        const Z cj = zc(__shfl_sync(0xffffffffu, c, j), 0.0);
        const double rhoj = __shfl_sync(0xffffffffu, rho, j);
        const int Nj = __shfl_sync(0xffffffffu, N, j);
        int nj = __shfl_sync(0xffffffffu, nf, j);
        const int ring = lane / kRing;
        const double rr = rhoj * (0.15 + 0.3 * ring);
        double sn, cs;
        sincospi((2.0 * (lane % kRing) + 0.5 * ring) / kRing, &sn, &cs);
        const Z seed = zc(cj.re + rr * cs, cj.im + rr * sn);
        Newton s = newton_start(seed);
        bool go = lane < kRingSeeds;
        while (true) {
            const int st = go ? newton_step<kNewtonMax>(mj, s, rj, nj) : 0;
            const unsigned hit = __ballot_sync(0xffffffffu, st > 0 && zabs(zsub(s.w, cj)) < rhoj);
            if (st != 0) go = false;
            if (hit) {
                const int win = __ffs(hit) - 1;
                const bool pair = __shfl_sync(0xffffffffu, fabs(s.w.im) > kPairIm * rhoj, win) && nj + 1 < Nj;
                if (lane == win) {
                    rj[nj] = s.w;
                    if (pair) rj[nj + 1] = zc(s.w.re, -s.w.im);
                }
                __syncwarp();
                nj += pair ? 2 : 1;
                if (nj >= Nj) break;
                s = newton_start(seed);
                go = lane < kRingSeeds;
            }
            if (!__any_sync(0xffffffffu, go)) break;
        }
        // ---- 3. what the seeds left
        int ej = 0;
        if (nj < Nj) nj = nci_subdivide(mj, cj, rhoj, rj, &ej);
        if (lane == j) { nf = nj; e |= ej; }
    }
    __syncwarp();
    if (!live) return;
    double best = 0.0;
    Z broot = zc(c, 0.0);
    for (int k = 0; k < nf; k++)
        if (r[k].im > best) { best = r[k].im; broot = r[k]; }
    growth[tid] = best;
    if (root) root[tid] = make_double2(broot.re, broot.im);
    if (count_out) count_out[tid] = nf;
    if (roots_out)
        for (int k = 0; k < max_out; k++) roots_out[tid * max_out + k] = k < nf ? make_double2(r[k].re, r[k].im) : make_double2(0.0, 0.0);
    if (e && err) atomicOr(err, e);
}

static hyb_status nci_launch(const double* samples, int64_t n, int order, int correct_j1, const int* alias, int n_alias,
                             double* growth, double* root, int max_out, double* roots_out, int* count_out, int* err,
                             void* stream) {
    if (!samples || !alias || !growth || n < 0 || n_alias < 1 || order < 1 || order > 3 || max_out < 0) {
        set_error("hyb_nci_growth: bad arguments");
        return HYB_EINVAL;
    }
    if (n == 0) return HYB_OK;
    const int64_t total = n * n_alias;
    // 32 pairs per warp where that still gives every SM eight warps, fewer on small calls
    int dev = 0, sms = 0;
    HYB_CUDA_TRY(cudaGetDevice(&dev));
    HYB_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int64_t spread = total / ((int64_t)sms * 8);
    const int group = spread >= 32 ? 32 : spread < 1 ? 1 : (int)spread;
    const int64_t per_block = (int64_t)group * (kNciThreads / 32);
    k_nci<<<(unsigned)((total + per_block - 1) / per_block), kNciThreads, 0, (cudaStream_t)stream>>>(
        reinterpret_cast<const NciSample*>(samples), n, order, correct_j1, alias, n_alias, group, growth,
        reinterpret_cast<double2*>(root), max_out, reinterpret_cast<double2*>(roots_out), count_out, err);
    HYB_CUDA_TRY(cudaGetLastError());
    return HYB_OK;
}

}  // namespace hyb

using namespace hyb;

extern "C" hyb_status hyb_nci_growth(const double* samples, int64_t n, int order, int correct_j1,
                                     const int* alias, int n_alias, double* growth, double* root, void* stream) {
    return nci_launch(samples, n, order, correct_j1, alias, n_alias, growth, root, 0, nullptr, nullptr, nullptr, stream);
}

extern "C" hyb_status hyb_nci_roots(const double* samples, int64_t n, int order, int correct_j1, const int* alias,
                                    int n_alias, int max_roots, double* roots, int* count, double* growth, int* err,
                                    void* stream) {
    if (!roots || !count || max_roots < 1) {
        set_error("hyb_nci_roots: bad arguments");
        return HYB_EINVAL;
    }
    return nci_launch(samples, n, order, correct_j1, alias, n_alias, growth, nullptr, max_roots, roots, count, err, stream);
}
