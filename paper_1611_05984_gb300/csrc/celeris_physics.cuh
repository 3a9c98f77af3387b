// Device functions of the method shared by the step kernels and the
// adjoint kernels: KP07 reconstruction and central-upwind flux (Sec. 2.2,
// Eq. 14), friction helpers, the sponge factor (Eq. 30).  They are templates
// on the arithmetic type, so the adjoint can evaluate them on dual numbers
// and get their exact derivatives along the same branches.
#pragma once
#include "celeris_internal.cuh"

namespace cel {

__device__ __forceinline__ int mirror_index(int i, int n)
{
    return i < 0 ? -1 - i : (i >= n ? 2 * n - 1 - i : i);
}

// Eq. 14: u = k(h) P with k(h) = sqrt(2) h / sqrt(h^4 + max(h^4, eps)).
template <typename real>
__device__ __forceinline__ real desing(real h, real eps)
{
    real h2 = h * h;
    real h4 = h2 * h2;
    return real(1.4142135623730951) * h * rsqrt(h4 + fmax(h4, eps));
}

// KP07 step 1: generalized minmod of the three one-sided / central slopes.
template <typename real>
__device__ __forceinline__ real minmod3(real th, real qm, real q0, real qp)
{
    // the three slopes share a sign iff the two one-sided ones do (the
    // central one lies between them); then the one of least magnitude
    real a = th * (q0 - qm), b = real(0.5) * (qp - qm), c = th * (qp - q0);
    real lo = fmin(a, fmin(b, c)), hi = fmax(a, fmax(b, c));
    return lo > real(0) ? lo : (hi < real(0) ? hi : real(0));
}

// KP07 steps 1-2 for one cell along one direction: face values of (w, P, Q)
// at the low and high faces, then the positivity fix of w.
template <typename real>
__device__ __forceinline__ void recon(real th, const real wq[3], const real Pq[3],
                                      const real Qq[3], real Blo, real Bhi, real lo[3],
                                      real hi[3])
{
    real sw = minmod3(th, wq[0], wq[1], wq[2]);
    real sP = minmod3(th, Pq[0], Pq[1], Pq[2]);
    real sQ = minmod3(th, Qq[0], Qq[1], Qq[2]);
    lo[0] = wq[1] - real(0.5) * sw;
    hi[0] = wq[1] + real(0.5) * sw;
    lo[1] = Pq[1] - real(0.5) * sP;
    hi[1] = Pq[1] + real(0.5) * sP;
    lo[2] = Qq[1] - real(0.5) * sQ;
    hi[2] = Qq[1] + real(0.5) * sQ;
    if (hi[0] < Bhi) {
        hi[0] = Bhi;
        lo[0] = real(2) * wq[1] - Bhi;
    } else if (lo[0] < Blo) {
        lo[0] = Blo;
        hi[0] = real(2) * wq[1] - Blo;
    }
}

// KP07 step 3: central-upwind flux.  States are (w, normal, tangential
// discharge); H = (mass, normal momentum, tangential momentum).
template <typename real>
__device__ __forceinline__ void cu_flux(real g, real eps, real wL, real nL, real tL, real wR,
                                        real nR, real tR, real Bf, real H[3])
{
    real hL = fmax(wL - Bf, real(0)), hR = fmax(wR - Bf, real(0));
    real kL = desing(hL, eps), kR = desing(hR, eps);
    real uL = kL * nL, vL = kL * tL, uR = kR * nR, vR = kR * tR;
    real qnL = hL * uL, qtL = hL * vL, qnR = hR * uR, qtR = hR * vR;
    real sL = sqrt(g * hL), sR = sqrt(g * hR);
    real ap = fmax(fmax(uL + sL, uR + sR), real(0));
    real am = fmin(fmin(uL - sL, uR - sR), real(0));
    real den = ap - am;
    if (!(den > real(0))) {
        H[0] = H[1] = H[2] = real(0);
        return;
    }
    real inv = real(1) / den, apam = ap * am;
    real FL1 = qnL * uL + real(0.5) * g * hL * hL, FR1 = qnR * uR + real(0.5) * g * hR * hR;
    H[0] = (ap * qnL - am * qnR + apam * (wR - wL)) * inv;
    H[1] = (ap * FL1 - am * FR1 + apam * (qnR - qnL)) * inv;
    H[2] = (ap * (qnL * vL) - am * (qnR * vR) + apam * (qtR - qtL)) * inv;
}

// ------------------------------------------------- the step kernels' arithmetic
//
// The same reconstruction and flux in the forms the FP64 stencil runs, fewer
// operations for the same function of the same inputs:
//   * slopes from one difference per face and variable (the high difference
//     of a cell is the low one of the next), the depths at a cell's faces
//     serving the positivity test and the flux;
//   * where both depths reach eps^(1/4), Eq. 14's factor is 1/h (h^4 is the
//     larger argument of its max) and h u is the discharge itself;
//   * the flux as the left one plus weighted differences, exact where both
//     sides agree.
// In FP64 every add, multiply and comparison runs on a pipe of two lanes per
// SM, which bounds the FP64 stencil, so comparisons, maxima and halvings work
// on the bit patterns with integer instructions, and reciprocals and roots are
// refined from the hardware's approximations (Householder's third-order step;
// Goldschmidt's iteration and a remainder).  2048 x 2048 beach, both stages and the line solves
// of 2 Euler and 2 full steps: 27.4 ms before, 20.0 ms with these forms, 19.4
// now (the predictor's DFMA, DADD and DMUL per cell from 425 to 309).

// Single operations, each rounded: where an expression could be contracted
// into a fused multiply-add in more than one way, the choice is written out
// (these and fma), so that every kernel that holds the expression gives the
// same bits.
__device__ __forceinline__ float add_r(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_r(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float sub_r(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double sub_r(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float mul_r(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_r(double a, double b) { return __dmul_rn(a, b); }

__device__ __forceinline__ float rcp_r(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// 1/x for normal x: y(1 + e + e^2) with e = 1 - x y, relative error e^3 + rounding.
__device__ __forceinline__ double rcp_r(double x)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}
// x / 2 (FP64: on the exponent; infinities and NaN as they are, and values
// below 2^-1021, which changes a sum by less than that).
__device__ __forceinline__ float half_r(float x) { return 0.5f * x; }
__device__ __forceinline__ double half_r(double x)
{
    const int hi = __double2hiint(x);
    const bool scale = (unsigned)(hi & 0x7ff00000) - 0x00200000u < 0x7fd00000u;   // exponent field 2 .. 0x7fe
    return __hiloint2double(scale ? hi - 0x00100000 : hi, __double2loint(x));
}

__device__ __forceinline__ float sqrt_r(float x) { return sqrtf(x); }
// sqrt(x): from y = 1/sqrt(x) (1 + e) one Goldschmidt step on s = x y and h = y/2
// (both 1 + O(e^2) off), then s + h (x - s^2) with the remainder exact to one
// rounding: what is left is s's own rounding (0.5001 units of the last place).
__device__ __forceinline__ double sqrt_r(double x)
{
    // near the ends of the range (subnormals and infinity among them) the plain root
    if ((unsigned)__double2hiint(x) - 0x01700000u < 0x7e800000u) {
        double y;
        asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
        const double s0 = mul_r(x, y), h0 = half_r(y), r = fma(-s0, h0, 0.5);
        const double s = fma(s0, r, s0), h = fma(h0, r, h0);
        return fma(fma(-s, s, x), h, s);
    }
    return __double_as_longlong(x) == 0 ? 0.0 : sqrt(x);
}

// x < 0 (false for NaN and -0)
__device__ __forceinline__ bool below_zero(float x) { return x < 0.f; }
__device__ __forceinline__ bool below_zero(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x);
    return hi - 0x80000000u < 0x7ff00001u && (hi << 1 | (unsigned)__double2loint(x)) != 0u;
}
// x == 0 (false for NaN)
__device__ __forceinline__ bool is_zero(float x) { return x == 0.f; }
__device__ __forceinline__ bool is_zero(double x) { return (__double_as_longlong(x) << 1) == 0; }
// x > 0, and x >= y for y > 0 (FP64: as integers, a NaN by its sign)
__device__ __forceinline__ bool above_zero(float x) { return x > 0.f; }
__device__ __forceinline__ bool above_zero(double x) { return __double_as_longlong(x) > 0; }
__device__ __forceinline__ bool at_least(float x, float y) { return x >= y; }
__device__ __forceinline__ bool at_least(double x, double y) { return __double_as_longlong(x) >= __double_as_longlong(y); }
// max(x, 0)
__device__ __forceinline__ float pos_r(float x) { return fmaxf(x, 0.f); }
__device__ __forceinline__ double pos_r(double x) { return __double2hiint(x) < 0 ? 0.0 : x; }

// a < b of doubles as integers: sign and magnitude to two's complement.
__device__ __forceinline__ long long order_key(double x)
{
    const long long k = __double_as_longlong(x);
    return k ^ ((k >> 63) & 0x7fffffffffffffffll);
}
// max(a, b, 0) and min(a, b, 0) (FP64: a NaN ranks beyond the infinity of its
// sign, so that of two speeds' extremes one is it)
__device__ __forceinline__ float max_zero(float a, float b)
{
    float d;
    asm("max.ftz.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(0.f));
    return d;
}
__device__ __forceinline__ double max_zero(double a, double b)
{
    const double m = order_key(a) > order_key(b) ? a : b;
    return __double2hiint(m) < 0 ? 0.0 : m;
}
__device__ __forceinline__ double min_zero(double a, double b)
{
    const double m = order_key(a) < order_key(b) ? a : b;
    return __double2hiint(m) < 0 ? m : 0.0;
}

// Minmod of a, b, c where a and c are the one-sided slopes and b lies
// between them: 0 unless a and c share a sign, else the least magnitude.
__device__ __forceinline__ float minmod_r(float a, float b, float c)
{
    float lo, hi;
    asm("min.ftz.f32 %0, %1, %2, %3;" : "=f"(lo) : "f"(a), "f"(b), "f"(c));
    asm("max.ftz.f32 %0, %1, %2, %3;" : "=f"(hi) : "f"(a), "f"(b), "f"(c));
    return fmaxf(lo, fminf(hi, 0.f));   // 0 clamped to [lo, hi]
}
__device__ __forceinline__ double minmod_r(double a, double b, double c)
{
    // bit patterns of one sign order as the magnitudes do
    const unsigned long long ka = (unsigned long long)__double_as_longlong(a);
    const unsigned long long kb = (unsigned long long)__double_as_longlong(b);
    const unsigned long long kc = (unsigned long long)__double_as_longlong(c);
    const unsigned long long ac = ka < kc ? ka : kc, m = ac < kb ? ac : kb;
    return (long long)(ka ^ kc) < 0 ? 0.0 : __longlong_as_double((long long)m);
}

// The same with the choice kept: 1, 2 or 3 for a, b or c, 0 for none (ties to
// a, then to b).
__device__ __forceinline__ int minmod_choice(float a, float b, float c, float &m)
{
    const bool b_c = fabsf(b) <= fabsf(c);
    const float mbc = b_c ? b : c;
    const bool first = fabsf(a) <= fabsf(mbc);
    m = first ? a : mbc;
    int s = first ? 1 : (b_c ? 2 : 3);
    if ((__float_as_int(a) ^ __float_as_int(c)) < 0 || m == 0.f) {
        s = 0;
        m = 0.f;
    }
    return s;
}
__device__ __forceinline__ int minmod_choice(double a, double b, double c, double &m)
{
    const unsigned long long ka = (unsigned long long)__double_as_longlong(a);
    const unsigned long long kb = (unsigned long long)__double_as_longlong(b);
    const unsigned long long kc = (unsigned long long)__double_as_longlong(c);
    const bool b_c = kb <= kc;
    const unsigned long long kbc = b_c ? kb : kc, k = ka <= kbc ? ka : kbc;
    int s = ka <= kbc ? 1 : (b_c ? 2 : 3);
    if ((long long)(ka ^ kc) < 0 || (k << 1) == 0ull) s = 0;
    m = s ? __longlong_as_double((long long)k) : 0.0;
    return s;
}

// x >= 0 (false for NaN) and a >= b (FP64: as integers; for finite values)
__device__ __forceinline__ bool not_below(float x) { return x >= 0.f; }
__device__ __forceinline__ bool not_below(double x) { return __double2hiint(x) >= 0 || (__double_as_longlong(x) << 1) == 0; }
__device__ __forceinline__ bool ge_r(float a, float b) { return a >= b; }
__device__ __forceinline__ bool ge_r(double a, double b)
{
    // -0 and 0 are equal
    const long long ka = order_key(a), kb = order_key(b);
    return ka >= kb || ((__double_as_longlong(a) | __double_as_longlong(b)) << 1) == 0;
}

// One cell's reconstruction along a direction, cells fed in order: q the
// cell's (w, normal, tangential discharge), a four times the half slopes'
// low-side candidate (2 theta times the difference to the cell before it).
template <typename real>
struct FaceSweep {
    real q[3], qm[3], a[3];

    // the first two cells of the sweep
    __device__ __forceinline__ void open(real th2, const real c0[3], const real c1[3])
    {
#pragma unroll
        for (int v = 0; v < 3; v++) {
            qm[v] = c0[v];
            q[v] = c1[v];
            a[v] = mul_r(th2, sub_r(c1[v], c0[v]));
        }
    }

    // KP07 steps 1-2 of the present cell, given the next one: values at its
    // low and high faces (beds Blo, Bhi) and the depths there (>= 0), then
    // the next cell becomes the present one.
    __device__ __forceinline__ void next(real th2, const real qp[3], real Blo, real Bhi, real lo[3], real hi[3],
                                         real &dlo, real &dhi)
    {
#pragma unroll
        for (int v = 0; v < 3; v++) {
            const real c = mul_r(th2, sub_r(qp[v], q[v]));
            const real m = minmod_r(a[v], sub_r(qp[v], qm[v]), c);
            lo[v] = fma(real(-0.25), m, q[v]);
            hi[v] = fma(real(0.25), m, q[v]);
            a[v] = c;
        }
        dlo = sub_r(lo[0], Blo);
        dhi = sub_r(hi[0], Bhi);
        if (below_zero(dhi)) {   // Reading A-L2
            hi[0] = Bhi;
            lo[0] = fma(real(2), q[0], -Bhi);
            dhi = real(0);
            dlo = pos_r(sub_r(lo[0], Blo));
        } else if (below_zero(dlo)) {
            lo[0] = Blo;
            hi[0] = fma(real(2), q[0], -Blo);
            dlo = real(0);
            dhi = pos_r(sub_r(hi[0], Bhi));
        }
#pragma unroll
        for (int v = 0; v < 3; v++) {
            qm[v] = q[v];
            q[v] = qp[v];
        }
    }
};

// KP07 step 3: the central-upwind flux H = (mass, normal, tangential
// momentum) from the face values (w, normal, tangential discharge) and depths.
__device__ __forceinline__ void face_flux_step(double g, double eps, double hwet, double wL, double nL, double tL,
                                               double hL, double wR, double nR, double tR, double hR, double H[3])
{
    const double ghL = mul_r(g, hL), ghR = mul_r(g, hR);
    const double sL = sqrt_r(ghL), sR = sqrt_r(ghR);
    const bool wet = at_least(hL, hwet) && at_least(hR, hwet);
    const double kL = wet ? rcp_r(hL) : desing(hL, eps), kR = wet ? rcp_r(hR) : desing(hR, eps);
    const double uL = mul_r(kL, nL), vL = mul_r(kL, tL), uR = mul_r(kR, nR), vR = mul_r(kR, tR);
    if (!wet) {
        nL = mul_r(hL, uL);
        tL = mul_r(hL, vL);
        nR = mul_r(hR, uR);
        tR = mul_r(hR, vR);
    }
    const double ap = max_zero(add_r(uL, sL), add_r(uR, sR));
    const double am = min_zero(sub_r(uL, sL), sub_r(uR, sR));
    const double den = sub_r(ap, am);
    if (is_zero(den)) {   // both sides dry (Reading A-F1); a NaN goes on into the flux
        H[0] = H[1] = H[2] = 0.0;
        return;
    }
    // (a+ F_L - a- F_R + a+ a- (q_R - q_L)) / (a+ - a-) = F_L + beta (F_R - F_L) - a+ beta (q_R - q_L), beta = -a-/(a+ - a-)
    const double beta = mul_r(-am, rcp_r(den)), nab = mul_r(-ap, beta);
    const double FL1 = fma(0.5, mul_r(ghL, hL), mul_r(nL, uL)), FR1 = fma(0.5, mul_r(ghR, hR), mul_r(nR, uR));
    const double FL2 = mul_r(nL, vL);
    const double dn = sub_r(nR, nL);
    H[0] = fma(nab, sub_r(wR, wL), fma(beta, dn, nL));
    H[1] = fma(nab, dn, fma(beta, sub_r(FR1, FL1), FL1));
    H[2] = fma(nab, sub_r(tR, tL), fma(beta, fma(nR, vR, -FL2), FL2));
}

__device__ __forceinline__ float cbrt_r(float x) { return x > 0.f ? exp2f(__log2f(x) * (1.f / 3.f)) : 0.f; }
__device__ __forceinline__ double cbrt_r(double x) { return cbrt(x); }
// 2^-126 <= h < 2^127: normal in single precision, and so is its reciprocal
__device__ __forceinline__ bool in_single_range(double h) { return (unsigned)__double2hiint(h) - 0x38100000u < 0x0fd00000u; }
// h^(-1/3) for h in that range: one third-order step r(1 + e/3 + 2 e^2/9),
// e = 1 - h r^3, from a single-precision value.
__device__ __forceinline__ double rcbrt_r(double h)
{
    const double r = (double)exp2f(__log2f((float)h) * (-1.f / 3.f));
    const double e = fma(mul_r(-h, r), mul_r(r, r), 1.0);
    return fma(mul_r(fma(2.0 / 9.0, e, 1.0 / 3.0), e), r, r);
}
// The friction's factor of (P, Q) (Eq. 31-32) for a depth hb: f k^2 (Manning:
// f k^(7/3)) with Eq. 14's factor k of max(hb, 0).
template <typename real>
__device__ __forceinline__ real friction_depth(int law, real fric, real hb, real eps, real hwet)
{
    if constexpr (sizeof(real) == 8) {
        if (at_least(hb, hwet) && (law != kFricManning || in_single_range(hb))) {   // k = 1/h
            if (law == kFricManning) {
                const real r = rcbrt_r(hb), r3 = r * r * r;
                return fric * (r3 * r3 * r);
            }
            const real k = rcp_r(hb);
            return fric * (k * k);
        }
    }
    const real k = desing(pos_r(hb), eps);
    const real f = law == kFricManning ? fric * cbrt_r(k) : fric;
    return f * (k * k);
}

__device__ __forceinline__ float cospi_r(float x) { return cospif(x); }
__device__ __forceinline__ double cospi_r(double x) { return cospi(x); }

// Eq. 30 with D the distance from the absorbing face to the cell centre and
// L_s = width cells: a cell idx cells from the side (idx = i for the west) is
// inside when idx < width, with (L_s - D)/L_s = (2 (width - idx) - 1)/(2 width).
template <typename real>
__device__ __forceinline__ real sponge_eq30(int w, int idx)
{
    const real r = real(2 * (w - idx) - 1) / real(2 * w);
    return real(0.5) * (real(1) + cospi_r(r));
}

// The factor of side s for a cell idx cells from it: 1 outside its sponge;
// inside, from the solver's table when the arguments carry one (the same
// expression, evaluated once per side and position), else evaluated here.
template <typename real>
__device__ __forceinline__ real sponge_side(const Coef<real> &c, int s, int idx)
{
    const int w = c.spw[s];
    if (idx >= w) return real(1);
    return c.gam ? c.gam[(size_t)s * c.npos + idx] : sponge_eq30<real>(w, idx);
}

// The smallest gamma over the sponge sides.
template <typename real>
__device__ __forceinline__ real sponge_gamma(const Coef<real> &c, const Geo &g, int i, int j)
{
    return fmin(fmin(sponge_side(c, 0, i), sponge_side(c, 1, g.nx - 1 - i)),
                fmin(sponge_side(c, 2, j), sponge_side(c, 3, g.ny - 1 - j)));
}

// Adjacent still-water depth d and ghost coordinates of table position pos
// (Reading A-B4): west / east sides run along rows j = pos - 2, south /
// north sides along columns i = pos - 2 including the corner columns, where
// d is clamped along the side.  Returns false where the position is unused.
template <typename real>
__device__ inline bool ghost_site(const Geo &g, const real *d_r, int side, int layer, int pos, double &x,
                                  double &y, double &dadj)
{
    const int along = pos - 2;
    if (side < 2) {
        if (along < 0 || along >= g.ny) return false;
        const int gi = side == 0 ? -1 - layer : g.nx + layer;
        x = (gi + 0.5) * g.dx;
        y = (along + 0.5) * g.dy;
        dadj = (double)d_r[(size_t)along * g.px + (side == 0 ? 0 : g.nx - 1)];
    } else {
        if (along < -2 || along > g.nx + 1) return false;
        const int gj = side == 2 ? -1 - layer : g.ny + layer;
        const int ia = along < 0 ? 0 : (along > g.nx - 1 ? g.nx - 1 : along);
        x = (along + 0.5) * g.dx;
        y = (gj + 0.5) * g.dy;
        dadj = (double)d_r[(size_t)(side == 2 ? 0 : g.ny - 1) * g.px + ia];
    }
    return true;
}

// The interior cell whose depth ghost_site reads for table position pos.
__device__ __forceinline__ void ghost_adjacent(const Geo &g, int side, int pos, int &i, int &j)
{
    const int along = pos - 2;
    if (side < 2) {
        i = side == 0 ? 0 : g.nx - 1;
        j = along;
    } else {
        i = along < 0 ? 0 : (along > g.nx - 1 ? g.nx - 1 : along);
        j = side == 2 ? 0 : g.ny - 1;
    }
}

}  // namespace cel
