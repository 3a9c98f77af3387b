// The FP32 stencil stage over one tile: 64 columns, a lane owning two
// neighbouring cells of a row, a warp kR consecutive rows.
//
// With a cell per thread the FP32 stencil was bound by instruction issue, so
// the layout is the one with the fewest instructions per cell:
//   * two cells per lane: additions, multiplications and fused
//     multiply-adds on both at once (.f32x2), 64-bit loads and stores of
//     shared and global memory, and one set of addresses, branches and loop
//     counts for two cells;
//   * a warp marches up its rows, so the reconstruction and fluxes along y and
//     the depth of the row below stay in registers; a cell's x-fluxes come
//     from its own reconstruction and its left neighbour's (shuffles), and
//     none goes through shared memory.
// The faces at the tile's west and east edges, which need cells of the
// neighbouring tiles' lanes, are computed first, one (side, row) per lane.
//
// A face's flux does not depend on which warp or variant computes it (the
// row's one branch, on a negative depth, skips a fix that would change
// nothing), so tiles of different heights give the same bits.
//
// Per cell about 560 thread instructions in the predictor and 495 in the
// corrector with 4 rows per warp, 511 and 451 with 8 (865 and 800 with a cell
// per thread and the fluxes in shared memory).  128 registers, no spills, 4
// blocks of 128 threads per SM: at 16 warps per SM it is bound by the latency
// of its own chains (0.64 of the issue slots with 4 rows per warp, 0.57 with
// 8).  Mean of both stages, with events around the launches: 2048 x 2048 cells
// 115 -> 93 us, 8192 x 8192 1664 -> 1299 us.
#pragma once
#include "celeris_internal.cuh"
#include "celeris_physics.cuh"

namespace cel {
namespace {

using pk = unsigned long long;   // two floats: the cells x and x + 1
constexpr float kLeastNormal = 1.17549435e-38f;   // a speed's reciprocal stays finite (smaller ones are flushed to 0)

__device__ __forceinline__ pk mk(float a, float b)
{
    pk r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void un(pk v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ float px_(pk v)
{
    float a, b;
    un(v, a, b);
    return a;
}
__device__ __forceinline__ float py_(pk v)
{
    float a, b;
    un(v, a, b);
    return b;
}
__device__ __forceinline__ pk add2(pk a, pk b)
{
    pk r;
    asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ pk sub2(pk a, pk b)
{
    pk r;
    asm("sub.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ pk mul2(pk a, pk b)
{
    pk r;
    asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ pk fma2(pk a, pk b, pk c)
{
    pk r;
    asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// f of each half
template <typename F>
__device__ __forceinline__ pk each(pk v, const F &f)
{
    float a, b;
    un(v, a, b);
    return mk(f(a), f(b));
}
__device__ __forceinline__ pk max2(pk v, float m) { return each(v, [=](float x) { return fmaxf(x, m); }); }
__device__ __forceinline__ pk max_zero2(pk v, pk w)
{
    float a, b, c, d;
    un(v, a, b);
    un(w, c, d);
    return mk(max_zero(a, c), max_zero(b, d));
}
__device__ __forceinline__ pk sqrt2(pk v) { return each(v, [](float x) { return sqrtf(x); }); }
__device__ __forceinline__ pk rsqrt2(pk v) { return each(v, [](float x) { return rsqrtf(x); }); }
__device__ __forceinline__ pk rcp2(pk v) { return each(v, [](float x) { return rcp_r(x); }); }
__device__ __forceinline__ pk cbrt2(pk v) { return each(v, [](float x) { return cbrt_r(x); }); }

// The same operations on one cell, so that the arithmetic below is stated once
// for pairs and for single cells and gives both the same bits.
__device__ __forceinline__ float add2(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub2(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float mul2(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fma2(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float max2(float v, float m) { return fmaxf(v, m); }
__device__ __forceinline__ float max_zero2(float v, float w) { return max_zero(v, w); }
__device__ __forceinline__ float sqrt2(float v) { return sqrtf(v); }
__device__ __forceinline__ float rsqrt2(float v) { return rsqrtf(v); }
__device__ __forceinline__ float rcp2(float v) { return rcp_r(v); }
__device__ __forceinline__ float cbrt2(float v) { return cbrt_r(v); }

// Constant k of the arguments
template <typename V>
__device__ __forceinline__ V kc(const StencilArgs<float> &A, int k)
{
    if constexpr (sizeof(V) == 8) return *reinterpret_cast<const pk *>(&A.kk.v[k]);
    else return A.kk.v[k].x;
}
__device__ __forceinline__ pk kc(const StencilArgs<float> &A, int k) { return kc<pk>(A, k); }

__device__ __forceinline__ pk ldp(const float *p) { return *reinterpret_cast<const pk *>(p); }
// The same, read again even where the value was read before.
__device__ __forceinline__ pk ldv(const float *p)
{
    pk r;
    asm volatile("ld.volatile.shared.b64 %0, [%1];" : "=l"(r) : "r"((unsigned)__cvta_generic_to_shared(p)));
    return r;
}
// pair or value k of a global array
template <typename V>
__device__ __forceinline__ V ldo(const float *p, unsigned k) { return reinterpret_cast<const V *>(p)[k]; }
template <typename V>
__device__ __forceinline__ void sto(float *p, unsigned k, V v) { reinterpret_cast<V *>(p)[k] = v; }

constexpr int kPW = kPairCols, kPWarps = kPairWarps;
constexpr int kPThreads = 32 * kPWarps;
constexpr int kPS = kPW + 8;     // row of the w and P tiles: columns x0 - 4 .. x0 + 67
constexpr int kPQ = kPW + 10;    // row of the Q tile (the transposing stores then hit 32 banks)
constexpr int kPB = kPW + 6;     // row of the corners: corner ci at ci - x0 + 2

// Shared memory of a tile of kR rows per warp.
template <int kR>
struct PairSmem {
    static constexpr int TH = kR * kPWarps;
    float w[(TH + 4) * kPS];
    float P[(TH + 4) * kPS];
    float Q[(TH + 4) * kPQ];
    float V[TH * kPW];           // the V* increment, for the transposed store
    float Bc[(TH + 3) * kPB];
    float4 edge[2][TH];          // west and east edge: flux through the face, depth d of the cell beyond
    uint32_t col[kPW];           // dry bits per column
};

// The history a stage reads (Carry), of two cells or one.
template <typename V>
struct CarryV {
    V a, b, r1, r2, p1, p2, Y;
};

template <typename V, int kSpec>
__device__ __forceinline__ CarryV<V> load_carry_v(const StencilArgs<float> &A, int v, unsigned k)
{
    const int kind = kSpec == 1 ? kAB3 : (kSpec == 2 ? kAM4 : A.kind);
    const bool ring = kSpec != 0 ? true : A.ring != 0;
    CarryV<V> c;
    c.a = c.b = c.r1 = c.r2 = c.p1 = c.p2 = c.Y = 0;
    if (kind == kAM4) {
        c.Y = ldo<V>(A.Y[v], k);
    } else if (ring) {
        if (kind == kAB3) {
            c.r1 = ldo<V>(A.R1[v], k);
            c.r2 = ldo<V>(A.R2[v], k);
        }
        if (v > 0 && kind != kEuler0) {
            c.p1 = ldo<V>(A.F1[v], k);
            if (kind == kAB3) c.p2 = ldo<V>(A.F2[v], k);
        }
    } else if (kind == kEuler1) {
        c.a = ldo<V>(A.a[v], k);
    } else if (kind == kAB3) {
        c.a = ldo<V>(A.a[v], k);
        c.b = ldo<V>(A.b[v], k);
    }
    return c;
}

// The single-precision arithmetic, on two cells or one (V).
//
// The order of every operation is part of the result, and a product that is
// rounded on its own before a sum is the addend of a fused multiply-add (the
// compiler may contract a plain sum of two cells with it).  Where a discharge is a small difference of
// large terms (the cross-tank one around an island, of the pressure 1/2 g h^2,
// the bed slope and the third differences of eta) its digits are this order's
// rounding errors over dx: on a 1178 x 1178 island another order, as close to
// 64 bits, parted from this one by 3.7e-5 of the discharge's norm and 2.4e-3
// of its root mean square.  tests/test_gpu_step_kernels.py pins the bits.

// advance(): the increment of U* or V*; of w the increment in the Euler stages
// and w itself in the others (kSpec 1 and 2).  The history is written where ok.
template <typename V, int kSpec>
__device__ __forceinline__ V advance_v(const StencilArgs<float> &A, int v, V X0, V R, V Phi, unsigned k,
                                       const CarryV<V> &c, bool ok)
{
    const int kind = kSpec == 1 ? kAB3 : (kSpec == 2 ? kAM4 : A.kind);
    const bool ring = kSpec != 0 ? true : A.ring != 0;
    if (kind == kAM4) {
        const V s = fma2(kc<V>(A, kc9C24), R, c.Y);
        return v > 0 ? add2(s, Phi) : s;
    }
    V D;
    if (ring) {
        if (ok) {
            sto(A.R0[v], k, R);
            if (v > 0) sto(A.F0[v], k, Phi);
        }
        if (kind != kAB3) {
            if (kind == kEuler1 && v > 0) D = fma2(kc<V>(A, kcDt), R, sub2(Phi, c.p1));
            else D = mul2(kc<V>(A, kcDt), R);
        } else {
            const V s = fma2(kc<V>(A, kc5), c.r2, fma2(kc<V>(A, kc23), R, mul2(kc<V>(A, kcM16), c.r1)));
            const V t = add2(fma2(kc<V>(A, kc19), R, mul2(kc<V>(A, kcM5), c.r1)), c.r2);
            V y;
            if (v > 0) {
                D = add2(fma2(kc<V>(A, kcMThree), c.p1, fma2(kc<V>(A, kcTwo), Phi, mul2(kc<V>(A, kcC12), s))), c.p2);
                y = fma2(kc<V>(A, kcMOne), Phi, mul2(kc<V>(A, kcC24), t));
            } else {
                D = fma2(kc<V>(A, kcOne), X0, mul2(kc<V>(A, kcC12), s));   // w itself
                y = fma2(kc<V>(A, kcC24), t, X0);
            }
            if (ok) sto(A.Y[v], k, y);
        }
        return D;
    }
    V na;
    if (kind == kEuler0) {
        D = mul2(kc<V>(A, kcDt), R);
        na = Phi;
    } else {
        if (kind == kEuler1) D = fma2(kc<V>(A, kcDt), R, sub2(Phi, c.a));
        else D = add2(fma2(kc<V>(A, kcTwo), Phi, mul2(kc<V>(A, kc23C12), R)), add2(c.a, c.b));
        na = fma2(kc<V>(A, kcM16C12), R, mul2(kc<V>(A, kcMThree), Phi));
    }
    if (ok) {
        sto(A.a[v], k, na);
        sto(A.b[v], k, fma2(kc<V>(A, kc5C12), R, Phi));
    }
    return D;
}

// KP07 steps 1-2 for two cells, without the positivity fix: q their (w,
// normal, tangential discharge), qm and qp the cells before and after each;
// values at the low and high faces and the depths there over the beds.
__device__ __forceinline__ void recon_pair(const StencilArgs<float> &A, const pk qm[3], const pk q[3], const pk qp[3],
                                           pk Blo, pk Bhi, pk lo[3], pk hi[3], pk &dlo, pk &dhi)
{
#pragma unroll
    for (int v = 0; v < 3; v++) {
        const pk a = mul2(kc(A, kcTh2), sub2(q[v], qm[v])), b = sub2(qp[v], qm[v]);
        const pk c = mul2(kc(A, kcTh2), sub2(qp[v], q[v]));
        float a0, a1, b0, b1, c0, c1;
        un(a, a0, a1);
        un(b, b0, b1);
        un(c, c0, c1);
        const pk m = mk(minmod_r(a0, b0, c0), minmod_r(a1, b1, c1));
        lo[v] = fma2(kc(A, kcMQ), m, q[v]);
        hi[v] = fma2(kc(A, kcQ), m, q[v]);
    }
    dlo = sub2(lo[0], Blo);
    dhi = sub2(hi[0], Bhi);
}

// The positivity fix (Reading A-L2) where a face depth is negative.
__device__ __forceinline__ void fix_pair(pk w, pk Blo, pk Bhi, pk &lo, pk &hi, pk &dlo, pk &dhi)
{
    float l0, l1, h0, h1, w0, w1, bl0, bl1, bh0, bh1, wl0, wl1, wh0, wh1;
    un(dlo, l0, l1);
    un(dhi, h0, h1);
    un(w, w0, w1);
    un(Blo, bl0, bl1);
    un(Bhi, bh0, bh1);
    un(lo, wl0, wl1);
    un(hi, wh0, wh1);
    auto fix = [](float w, float bl, float bh, float &wl, float &wh, float &l, float &h) {
        if (h < 0.f) {
            wh = bh;
            wl = fma(2.f, w, -bh);
            h = 0.f;
            l = fmaxf(wl - bl, 0.f);
        } else if (l < 0.f) {
            wl = bl;
            wh = fma(2.f, w, -bl);
            l = 0.f;
            h = fmaxf(wh - bh, 0.f);
        }
    };
    fix(w0, bl0, bh0, wl0, wh0, l0, h0);
    fix(w1, bl1, bh1, wl1, wh1, l1, h1);
    lo = mk(wl0, wl1);
    hi = mk(wh0, wh1);
    dlo = mk(l0, l1);
    dhi = mk(h0, h1);
}

// Eq. 14's factor of a depth >= 0 (desing).
template <typename V>
__device__ __forceinline__ V desing_v(const StencilArgs<float> &A, V h)
{
    const V h2 = mul2(h, h), h4 = mul2(h2, h2);
    return mul2(mul2(kc<V>(A, kcRoot2), h), rsqrt2(fma2(kc<V>(A, kcOne), h4, max2(h4, A.c.eps))));
}

// KP07 step 3: left states L = (w, normal, tangential discharge) and depths
// hL >= 0, right states R, depths hR; H = (mass, normal, tangential momentum).
template <typename V>
__device__ __forceinline__ void flux_v(const StencilArgs<float> &A, const V L[3], V hL, const V R[3], V hR, V H[3])
{
    const V kL = desing_v(A, hL), kR = desing_v(A, hR);
    const V uL = mul2(kL, L[1]), vL = mul2(kL, L[2]), uR = mul2(kR, R[1]), vR = mul2(kR, R[2]);
    const V nL = mul2(hL, uL), nR = mul2(hR, uR);
    const V gL = mul2(kc<V>(A, kcHalfG), hL), gR = mul2(kc<V>(A, kcHalfG), hR);
    const V sL = sqrt2(add2(gL, gL)), sR = sqrt2(add2(gR, gR));
    const V ap = max_zero2(add2(uL, sL), add2(uR, sR)), nam = max_zero2(sub2(sL, uL), sub2(sR, uR));   // a+, -a-
    // where both sides are dry (Reading A-F1) every term is 0 and so is the flux
    const V inv = rcp2(max2(add2(ap, nam), kLeastNormal)), nab = mul2(ap, nam);
    const V FL1 = fma2(gL, hL, mul2(nL, uL)), FR1 = fma2(gR, hR, mul2(nR, uR));
    H[0] = mul2(inv, fma2(nab, sub2(L[0], R[0]), fma2(ap, nL, mul2(nam, nR))));
    H[1] = mul2(inv, fma2(nab, sub2(nL, nR), fma2(ap, FL1, mul2(nam, FR1))));
    H[2] = mul2(inv, fma2(nab, fma2(mul2(kc<V>(A, kcMOne), hR), vR, mul2(hL, vL)),
                          fma2(ap, mul2(nL, vL), mul2(nam, mul2(nR, vR)))));
}

// Friction (Eq. 31-32) subtracted from F and G of a cell of depth hb.
template <typename V>
__device__ __forceinline__ void friction_v(const StencilArgs<float> &A, int law, V hb, V P, V Q, V &F, V &G)
{
    const V k = desing_v(A, max2(hb, 0.f)), nk = mul2(kc<V>(A, kcMOne), k);
    V fc = kc<V>(A, kcFric);
    if (law == kFricManning) fc = mul2(fc, cbrt2(k));
    const V mag = sqrt2(fma2(P, P, mul2(Q, Q)));
    F = fma2(mul2(mul2(mul2(fc, P), mag), k), nk, F);
    G = fma2(mul2(mul2(mul2(fc, Q), mag), k), nk, G);
}

// A cell's value c with its neighbours' (for eta two cells out along the axes).
template <typename V>
struct Around {
    V c, e, w, n, s, ne, nw, se, sw, ee, ww, nn, ss;
};

// Eq. 10-11's dispersive terms added to F and G: w around the cell, its depth
// d and the depth's gradient.
template <typename V>
__device__ __forceinline__ void eta_terms_v(const StencilArgs<float> &A, const Around<V> &q, V d, V ddx, V ddy, V &F, V &G)
{
    const V two = kc<V>(A, kcTwo), mtwo = kc<V>(A, kcMTwo);
    const V K2 = mul2(mul2(kc<V>(A, kcBg), d), d), K3 = mul2(K2, d);
    const V exx = mul2(add2(fma2(mtwo, q.c, q.e), q.w), kc<V>(A, kcRdx2));
    const V eyy = mul2(add2(fma2(mtwo, q.c, q.n), q.s), kc<V>(A, kcRdy2));
    const V exy = mul2(add2(sub2(sub2(q.ne, q.se), q.nw), q.sw), kc<V>(A, kcRdxdy4));
    const V exxx = sub2(fma2(two, q.w, fma2(mtwo, q.e, q.ee)), q.ww);   // the third differences undivided
    const V eyyy = sub2(fma2(two, q.s, fma2(mtwo, q.n, q.nn)), q.ss);
    const V exyy = sub2(add2(fma2(mtwo, q.e, q.ne), q.se), add2(fma2(mtwo, q.w, q.nw), q.sw));
    const V exxy = sub2(add2(fma2(mtwo, q.n, q.ne), q.nw), add2(fma2(mtwo, q.s, q.se), q.sw));
    const V x3 = fma2(exxx, kc<V>(A, kcRdx3h), mul2(exyy, kc<V>(A, kcRdxdy2h)));
    const V y3 = fma2(eyyy, kc<V>(A, kcRdy3h), mul2(exxy, kc<V>(A, kcRdx2dyh)));
    const V x2 = fma2(ddx, fma2(two, exx, eyy), mul2(ddy, exy)), y2 = fma2(ddy, fma2(two, eyy, exx), mul2(ddx, exy));
    F = add2(F, fma2(K3, x3, mul2(K2, x2)));
    G = add2(G, fma2(K3, y3, mul2(K2, y2)));
}

// Eq. 12-13's mixed terms: F* from Q, G* from P around the cell (no second
// neighbours).
template <typename V>
__device__ __forceinline__ V mixed_term_v(const StencilArgs<float> &A, const Around<V> &q, V d, V ddx, V ddy)
{
    const V qx = mul2(sub2(q.e, q.w), kc<V>(A, kcHrdx)), qy = mul2(sub2(q.n, q.s), kc<V>(A, kcHrdy));
    const V qxy = mul2(add2(sub2(sub2(q.ne, q.se), q.nw), q.sw), kc<V>(A, kcRdxdy4)), sixth = kc<V>(A, kcSixth);
    return fma2(mul2(mul2(kc<V>(A, kcB3), d), d), qxy,
                fma2(mul2(mul2(d, ddy), qx), sixth, mul2(mul2(mul2(d, ddx), qy), sixth)));
}

// A lane's pair of values at its cells' west faces, from its left neighbour's
// second cell and its own first.
__device__ __forceinline__ pk from_left(pk v)
{
    float a, b;
    un(v, a, b);
    return mk(__shfl_up_sync(0xffffffffu, b, 1), a);
}

// A warp's row of corners: c[ci] for its cells' columns x, x + 1 and x + 2,
// and the sums of neighbours.
struct CornerRow {
    pk c;        // ci = x, x + 1
    float z;     // ci = x + 2
    pk h;        // c[x] + c[x+1], c[x+1] + c[x+2]
};

// Read again (ldv).
__device__ __forceinline__ CornerRow corner_rowv(const float *p)
{
    CornerRow r;
    r.c = ldv(p);
    float a, b, d;
    un(ldv(p + 2), r.z, d);
    un(r.c, a, b);
    r.h = mk(a + b, b + r.z);
    return r;
}

__device__ __forceinline__ CornerRow corner_row(const float *p)
{
    CornerRow r;
    r.c = ldp(p);
    r.z = p[2];
    float a, b;
    un(r.c, a, b);
    r.h = mk(a + b, b + r.z);
    return r;
}

// Cell beds of the row between corner rows lo and hi, as cell_bbar gives them.
__device__ __forceinline__ pk bbar_pair(const StencilArgs<float> &A, const CornerRow &lo, const CornerRow &hi)
{
    float a, b;
    un(hi.c, a, b);
    return mul2(kc(A, kcQ), add2(add2(lo.h, hi.c), mk(b, hi.z)));
}

__device__ __forceinline__ pk depth_pair(const StencilArgs<float> &A, pk Bb)
{
    float a, b;
    un(sub2(kc(A, kcWs), Bb), a, b);
    return mk(fmaxf(a, 0.f), fmaxf(b, 0.f));
}

// The x-neighbours of a row's two cells: w at x - 2, x - 1, x + 2, x + 3, the
// discharges at x - 1 and x + 2.
struct SideRow {
    float wll, wl, wr, wrr, pl, pr, ql, qr;
};

__device__ __forceinline__ SideRow side_row(const float *w, const float *P, const float *Q)
{
    SideRow s;
    un(ldp(w - 2), s.wll, s.wl);
    un(ldp(w + 2), s.wr, s.wrr);
    s.pl = P[-1];
    s.pr = P[2];
    s.ql = Q[-1];
    s.qr = Q[2];
    return s;
}

// The pairs around the pair v at p in shared memory (rows kStrideOf apart, n
// and s those above and below), read again (ldv).
template <int kStrideOf>
__device__ __forceinline__ Around<pk> aroundv(const float *p, pk v, pk n, pk s)
{
    Around<pk> q;
    auto sides = [](const float *r, pk c, pk &e, pk &w, pk &ee, pk &ww) {
        ww = ldv(r - 2);
        ee = ldv(r + 2);
        e = mk(py_(c), px_(ee));
        w = mk(py_(ww), px_(c));
    };
    pk beyond[2];
    q.c = v;
    q.n = n;
    q.s = s;
    sides(p, v, q.e, q.w, q.ee, q.ww);
    sides(p + kStrideOf, n, q.ne, q.nw, beyond[0], beyond[1]);
    sides(p - kStrideOf, s, q.se, q.sw, beyond[0], beyond[1]);
    return q;
}

__device__ __forceinline__ uint32_t spread_bits(uint32_t x)   // bit k of the low half to bit 2k
{
    x &= 0xffffu;
    x = (x | (x << 8)) & 0x00ff00ffu;
    x = (x | (x << 4)) & 0x0f0f0f0fu;
    x = (x | (x << 2)) & 0x33333333u;
    return (x | (x << 1)) & 0x55555555u;
}

// Asynchronous copy of one element from global to shared memory (zero-filled
// when !valid, reading nothing); all of a thread's copies are in flight at
// once and cost no registers.  cp_async_wait_all waits for this thread's.
template <typename real>
__device__ __forceinline__ void cp_async_elem(real *smem, const real *gmem, bool valid)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    if (sizeof(real) == 4)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(s), "l"(gmem), "r"(valid ? 4 : 0)
                     : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(s), "l"(gmem), "r"(valid ? 8 : 0)
                     : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(gmem)
                 : "memory");
}

// The tile's rows of the history arrays this stage reads, asked into L2 (256
// bytes a row), so that the loads in the row loop can come late and hold few
// registers.
template <int kSpec, int TH>
__device__ __forceinline__ void prefetch_history(const StencilArgs<float> &A, int x0, int y0, int tid)
{
    const int j = y0 + (tid & (TH - 1));
    const size_t o = (size_t)j * A.geo.px + x0;
    const bool in = j < A.geo.ny, two = x0 + 32 < A.geo.px;
    auto rows = [&](const float *p) {
        if (in) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + o));
        if (in && two) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + o + 32));
    };
    // groups of TH threads, an array each at a time
    const int grp = tid / TH;
    if constexpr (kSpec == 2) {
        for (int v = grp; v < 3; v += kPThreads / TH) rows(A.Y[v]);
    } else if constexpr (kSpec == 1) {
        for (int k = grp; k < 10; k += kPThreads / TH) {
            const int v = k % 3;
            rows(k < 3 ? A.R1[v] : k < 6 ? A.R2[v] : k < 8 ? A.F1[k - 5] : A.F2[k - 7]);
        }
    }
}

// One tile, by a block of kPThreads threads.
template <int kSpec, int kR>
__device__ __forceinline__ void stencil_tile_pair(const StencilArgs<float> &A, const int x0, const int y0,
                                                  unsigned char *smem_raw)
{
    const int tid = threadIdx.x;
    const StencilArgs<float> &A0 = A;
    using S = PairSmem<kR>;
    constexpr int TH = S::TH;
    S &sm = *reinterpret_cast<S *>(smem_raw);
    const Geo &G = A.geo;
    const Coef<float> &C = A.c;
    const int nx = G.nx, ny = G.ny;
    const int lane = tid & 31, warp = tid >> 5;

    // ---- 1. the state (+ 2 cells) and the corners.  Parts beyond the field
    //         are left as they are: the ghosts below are filled in, and
    //         nothing else outside the grid reaches a cell of it.
    {
        // Q, column-major: four rows per load, a warp's lanes over 8 columns
        // and 4 such groups of rows, transposed into the tile below (every
        // load of a thread is in flight before the first is stored)
        constexpr int nrg = (TH + 8) / 4, ngg = (nrg + 3) / 4, ncg = (kPW + 8) / 8;
        constexpr int nq = (ngg * ncg + kPWarps - 1) / kPWarps;
        float4 q[nq];
        auto q_at = [&](int u, int &r, int &c) -> bool {   // load u's first tile row and column
            const int k = warp + u * kPWarps, rg = (k % ngg) * 4 + (lane & 3);
            c = (k / ngg) * 8 + (lane >> 2);
            r = 4 * rg - 2;
            const int gy = y0 - 4 + 4 * rg, gx = x0 - 4 + c;
            return k < ngg * ncg && rg < nrg && gy >= 0 && gy < G.py && gx >= 0 && gx < nx && c >= 2 && c < kPW + 6;
        };
#pragma unroll
        for (int u = 0; u < nq; u++) {
            int r, c;
            if (q_at(u, r, c))
                q[u] = *reinterpret_cast<const float4 *>(A.Qc_in + (ptrdiff_t)(x0 - 4 + c) * G.py + (y0 - 2 + r));
        }
        // a warp per row: w and P in 16-byte pieces (lanes 0 .. 17), the
        // corners one by one
        const int gx = x0 - 4 + 4 * lane;
        const bool piece = lane < kPS / 4 && gx >= 0 && gx < G.px;
        const float *gw = A.w_in + (ptrdiff_t)(y0 - kHalo + warp) * G.px + gx;
        const ptrdiff_t dP = A.P_in - A.w_in;
        float *sw = sm.w + warp * kPS + 4 * lane;
#pragma unroll
        for (int r = 0; r < TH + 4; r += kPWarps) {
            const int gy = y0 - kHalo + warp + r;
            if (piece && gy >= 0 && gy < ny) {
                cp_async16(sw + r * kPS, gw);
                cp_async16(sw + r * kPS + (TH + 4) * kPS, gw + dP);
            }
            gw += kPWarps * G.px;
        }
        // corners ci = x0 - 1 .. x0 + 65, array index ci + 1
        const float *gb = A.Bc + (size_t)(y0 + warp) * G.pc + x0 + lane;
        float *sb = sm.Bc + warp * kPB + lane + 1;
        const int left = nx + 3 - x0 - lane;
#pragma unroll
        for (int r = 0; r < TH + 3; r += kPWarps) {
            if (warp + r < TH + 3 && y0 + warp + r < ny + 3) {
                if (left > 0) cp_async_elem(sb + r * kPB, gb, true);
                if (left > 32) cp_async_elem(sb + r * kPB + 32, gb + 32, true);
                if (lane < 3 && left > 64) cp_async_elem(sb + r * kPB + 64, gb + 64, true);
            }
            gb += kPWarps * G.pc;
        }
        if (tid < kPW) sm.col[tid] = 0u;
        prefetch_history<kSpec, TH>(A, x0, y0, tid);
#pragma unroll
        for (int u = 0; u < nq; u++) {
            int r, c;
            if (!q_at(u, r, c)) continue;
            float *d = sm.Q + r * kPQ + c;
            if (r >= 0) {
                d[0] = q[u].x;
                d[kPQ] = q[u].y;
            }
            if (r + 2 < TH + 4) {
                d[2 * kPQ] = q[u].z;
                d[3 * kPQ] = q[u].w;
            }
        }
        cp_async_wait_all();
    }
    __syncthreads();

    // ---- 2. ghost layers (Sec. 2.4): x-sides over interior rows, then
    //         y-sides over every column, so corners come by composition.
    const bool westT = x0 == 0, eastT = x0 + kPW + kHalo > nx;
    const bool southT = y0 == 0, northT = y0 + TH + kHalo > ny;
    if (westT || eastT) {
        for (int k = tid; k < 4 * (TH + 2); k += kPThreads) {
            const int r = 1 + k % (TH + 2), which = k / (TH + 2);
            const int gy = y0 - kHalo + r, side = which < 2 ? 0 : 1, kk = which & 1;
            if (gy < 0 || gy >= ny || (side == 0 ? !westT : !eastT)) continue;
            const int gx = side == 0 ? -1 - kk : nx + kk, c = gx - x0 + 4;
            if (c < 2 || c >= kPW + 6) continue;
            const int src = (side == 0 ? kk : nx - 1 - kk) - x0 + 4;
            if ((C.sine >> side) & 1) {
                const float *tb = A.ghost + ghost_index(A.tsel, side, kk, 0, gy + 2, C.npos);
                sm.w[r * kPS + c] = tb[0];
                sm.P[r * kPS + c] = tb[C.npos];
                sm.Q[r * kPQ + c] = tb[2 * C.npos];
            } else {
                sm.w[r * kPS + c] = sm.w[r * kPS + src];
                sm.P[r * kPS + c] = -sm.P[r * kPS + src];
                sm.Q[r * kPQ + c] = sm.Q[r * kPQ + src];
            }
        }
    }
    if (southT || northT) {
        __syncthreads();   // the corner columns' x-ghosts
        for (int k = tid; k < 4 * (kPW + 2); k += kPThreads) {
            const int c = 3 + k % (kPW + 2), which = k / (kPW + 2);
            const int gx = x0 - 4 + c, side = which < 2 ? 2 : 3, kk = which & 1;
            if (side == 2 ? !southT : !northT) continue;
            if (gx > nx + 1) continue;
            const int gy = side == 2 ? -1 - kk : ny + kk, r = gy - y0 + kHalo;
            if (r < 0 || r >= TH + 4) continue;
            const int src = (side == 2 ? kk : ny - 1 - kk) - y0 + kHalo;
            if ((C.sine >> side) & 1) {
                const float *tb = A.ghost + ghost_index(A.tsel, side, kk, 0, gx + 2, C.npos);
                sm.w[r * kPS + c] = tb[0];
                sm.P[r * kPS + c] = tb[C.npos];
                sm.Q[r * kPQ + c] = tb[2 * C.npos];
            } else {
                sm.w[r * kPS + c] = sm.w[src * kPS + c];
                sm.P[r * kPS + c] = sm.P[src * kPS + c];
                sm.Q[r * kPQ + c] = -sm.Q[src * kPQ + c];
            }
        }
    }
    if (westT || eastT || southT || northT) __syncthreads();

    // ---- 3. the faces at the tile's west and east edges and the depths of
    //         the cells beyond them, for this warp's rows
    const int r0 = warp * kR;   // first tile row of the warp
    if (lane < 2 * kR) {
        const int side = lane >= kR ? 1 : 0, r = r0 + (side ? lane - kR : lane);
        const int f = side ? kPW : 0;
        const float *w = sm.w + (r + 2) * kPS + f + 2, *P = sm.P + (r + 2) * kPS + f + 2;   // cell f - 2
        const float *Q = sm.Q + (r + 2) * kPQ + f + 2;
        const float *b = sm.Bc + (r + 1) * kPB + f + 1;                                    // corner f - 1, rows r and r + 1
        const float c0 = b[0], c1 = b[1], c2 = b[2], e0 = b[kPB], e1 = b[kPB + 1], e2 = b[kPB + 2];
        const float Bf = 0.5f * (c1 + e1);
        FaceSweep<float> fs;
        const float q0[3] = {w[0], P[0], Q[0]}, q1[3] = {w[1], P[1], Q[1]};
        const float q2[3] = {w[2], P[2], Q[2]}, q3[3] = {w[3], P[3], Q[3]};
        float lo[3], hi[3], lo2[3], hi2[3], dl, dh, dl2, dh2, H[3];
        fs.open(C.th2, q0, q1);
        fs.next(C.th2, q2, 0.5f * (c0 + e0), Bf, lo, hi, dl, dh);
        fs.next(C.th2, q3, Bf, 0.5f * (c2 + e2), lo2, hi2, dl2, dh2);
        flux_v<float>(A, hi, dh, lo2, dl2, H);
        // the cell beyond: f - 1 on the west, f on the east
        const float Bb = side ? cell_bbar(c1, c2, e1, e2) : cell_bbar(c0, c1, e0, e1);
        sm.edge[side][r] = make_float4(H[0], H[1], H[2], fmaxf(C.ws - Bb, 0.f));
    }
    __syncwarp();

    // ---- 4. the rows.  What a row shares with the next and is dearer to
    //         read again than to keep: the next row's cells, the fluxes and
    //         high sides along y, the depth of the row below.
    const float ws = C.ws;
    const bool bsnq = A.phy.model == kBsnq;
    const int friction = A.phy.friction;
    const int i = x0 + 2 * lane;
    const bool ok0 = i < nx, ok1 = i + 1 < nx, atW = lane == 0, atE = lane == 31;
    const bool sponge_tile = A.final_stage && (x0 < C.spw[0] || x0 + kPW > nx - C.spw[1] || y0 < C.spw[2] ||
                                               y0 + TH > ny - C.spw[3]);
    const float *pw = sm.w + (r0 + 2) * kPS + 2 * lane + 4;
    constexpr int oP = (TH + 4) * kPS;          // from the w tile to the P tile
    const float *pQ = sm.Q + (r0 + 2) * kPQ + 2 * lane + 4;
    const float *pb = sm.Bc + (r0 + 1) * kPB + 2 * lane + 2;   // corner row r0
    float *pv = sm.V + r0 * kPW + 2 * lane;
    const float4 *pe = atE ? &sm.edge[1][r0] : &sm.edge[0][r0];
    unsigned kr = (unsigned)(((size_t)(y0 + r0) * G.px + i) >> 1);   // the lane's pair in a row-major array
    const int rows = ny - (y0 + r0) < kR ? ny - (y0 + r0) : kR;   // rows of this warp inside the grid

    if (rows > 0) {
    pk qn[3], hi[3], Hs[3], dhi;   // row r + 1; cell r's values at its north face; flux through its south face
    pk dS;                         // depth d of row r - 1
    {
        const pk q2[3] = {ldp(pw - 2 * kPS), ldp(pQ - 2 * kPQ), ldp(pw + oP - 2 * kPS)};
        const pk q1[3] = {ldp(pw - kPS), ldp(pQ - kPQ), ldp(pw + oP - kPS)};
        const pk q[3] = {ldp(pw), ldp(pQ), ldp(pw + oP)};
        qn[0] = ldp(pw + kPS);
        qn[1] = ldp(pQ + kPQ);
        qn[2] = ldp(pw + oP + kPS);
        const CornerRow cm = corner_row(pb - kPB), c0 = corner_row(pb), c1 = corner_row(pb + kPB);
        const pk hlf = kc(A, kcHalf);
        pk lo[3], hm[3], dl, dm;
        recon_pair(A, q2, q1, q, mul2(hlf, cm.h), mul2(hlf, c0.h), lo, hm, dl, dm);
        fix_pair(q1[0], mul2(hlf, cm.h), mul2(hlf, c0.h), lo[0], hm[0], dl, dm);
        recon_pair(A, q1, q, qn, mul2(hlf, c0.h), mul2(hlf, c1.h), lo, hi, dl, dhi);
        fix_pair(q[0], mul2(hlf, c0.h), mul2(hlf, c1.h), lo[0], hi[0], dl, dhi);
        flux_v<pk>(A, hm, dm, lo, dl, Hs);
        if (bsnq) dS = depth_pair(A, bbar_pair(A, cm, c0));
    }
#pragma unroll 1
    for (int r = 0; r < rows; r++) {
        // the arguments through an offset the compiler takes for unknown, new
        // in every row: else it keeps every constant and pointer in registers
        // across the loop (some 50 of them) and spills the cells
        unsigned zero;
        asm volatile("mov.b32 %0, 0;" : "=r"(zero));
        const StencilArgs<float> &A = *reinterpret_cast<const StencilArgs<float> *>(reinterpret_cast<const char *>(&A0) + zero);
        const Coef<float> &C = A.c;
        // Reconstructions: of row r + 1 along y (its low side is the right
        // state of row r's north face) and of row r along x.
        const CornerRow c0 = corner_row(pb), c1 = corner_row(pb + kPB), c2 = corner_row(pb + 2 * kPB);
        const pk hlf = kc(A, kcHalf);
        pk ly[3], hy[3], dly, dhy;
        pk lx[3], hx[3], dlx, dhx;
        const pk q[3] = {ldp(pw), ldp(pQ), ldp(pw + oP)};
        const pk By0 = mul2(hlf, c1.h), By1 = mul2(hlf, c2.h);
        {
            const pk qq[3] = {ldp(pw + 2 * kPS), ldp(pQ + 2 * kPQ), ldp(pw + oP + 2 * kPS)};
            recon_pair(A, q, qn, qq, By0, By1, ly, hy, dly, dhy);
        }
        pk Bx0, Bx1, sx;                     // face beds; their sums' differences
        {
            const SideRow side = side_row(pw, pw + oP, pQ);
            float a, b, v0, v1;
            un(add2(c0.c, c1.c), v0, v1);
            const float v2 = c0.z + c1.z;
            const float f0 = 0.5f * v0, f1 = 0.5f * v1, f2 = 0.5f * v2;
            Bx0 = mk(f0, f1);
            Bx1 = mk(f1, f2);
            sx = mk(v1 - v0, v2 - v1);
            pk qm[3], q0[3], qp[3];
            un(q[0], a, b);
            qm[0] = mk(side.wl, a);
            q0[0] = q[0];
            qp[0] = mk(b, side.wr);
            un(q[2], a, b);
            qm[1] = mk(side.pl, a);
            q0[1] = q[2];
            qp[1] = mk(b, side.pr);
            un(q[1], a, b);
            qm[2] = mk(side.ql, a);
            q0[2] = q[1];
            qp[2] = mk(b, side.qr);
            recon_pair(A, qm, q0, qp, Bx0, Bx1, lx, hx, dlx, dhx);
        }
        const pk Bb = bbar_pair(A, c0, c1), sy = sub2(c1.h, c0.h), hb = sub2(q[0], Bb);
        // Fluxes through the north faces and the west faces, and friction.
        // One branch for the row: the fix changes nothing where no depth is
        // negative.  Only faces of the grid's cells count (along x also those
        // of cell nx, whose low side the last face takes), not what lies
        // unwritten beyond them.
        pk Hn[3], H[3];
        float y0m, y1m, x0m, x1m;
        {
            float a, b;
            un(dly, y0m, y1m);
            un(dhy, a, b);
            y0m = fminf(y0m, a);
            y1m = fminf(y1m, b);
            un(dlx, x0m, x1m);
            un(dhx, a, b);
            x0m = fminf(x0m, a);
            x1m = fminf(x1m, b);
        }
        if (__any_sync(0xffffffffu, (ok0 && (y0m < 0.f || x1m < 0.f)) || (ok1 && y1m < 0.f) || (i <= nx && x0m < 0.f))) {
            fix_pair(qn[0], By0, By1, ly[0], hy[0], dly, dhy);
            fix_pair(q[0], Bx0, Bx1, lx[0], hx[0], dlx, dhx);
        }
        {
            const pk Lx[3] = {from_left(hx[0]), from_left(hx[1]), from_left(hx[2])};
            flux_v<pk>(A, hi, dhi, ly, dly, Hn);
            flux_v<pk>(A, Lx, from_left(dhx), lx, dlx, H);
        }
        CarryV<pk> cw, cu, cv;
        if (kSpec == 2 && ok0) {
            cw = load_carry_v<pk, kSpec>(A, 0, kr);
            cu = load_carry_v<pk, kSpec>(A, 1, kr);
            cv = load_carry_v<pk, kSpec>(A, 2, kr);
        }
        // flux differences: south less north, west less east (the next lane's
        // west face; the tile's edge faces from the first pass)
        pk dv[3];
        {
            const pk ry = kc(A, kcRdy), rx = kc(A, kcRdx);
            dv[0] = mul2(ry, sub2(Hs[0], Hn[0]));
            dv[1] = mul2(ry, sub2(Hs[2], Hn[2]));   // the normal discharge is Q
            dv[2] = mul2(ry, sub2(Hs[1], Hn[1]));
            float4 edge = make_float4(0.f, 0.f, 0.f, 0.f);
            if (atW || atE) edge = pe[r];
#pragma unroll
            for (int v = 0; v < 3; v++) {
                hi[v] = hy[v];
                Hs[v] = Hn[v];
                float a, b;
                un(H[v], a, b);
                const float ev = v == 0 ? edge.x : (v == 1 ? edge.y : edge.z);
                float e = __shfl_down_sync(0xffffffffu, a, 1);
                if (atW) a = ev;
                if (atE) e = ev;
                dv[v] = fma2(rx, sub2(mk(a, b), mk(b, e)), dv[v]);
            }
            dhi = dhy;
        }
        // rows r .. r + 2 again from shared memory: kept through the fluxes
        // they would not fit the registers
        const CornerRow e1 = corner_rowv(pb + kPB), e2 = corner_rowv(pb + 2 * kPB);
        const pk u[3] = {ldv(pw), ldv(pQ), ldv(pw + oP)}, cn[3] = {ldv(pw + kPS), ldv(pQ + kPQ), ldv(pw + oP + kPS)};
        const pk uu = ldv(pw + 2 * kPS);
        // the history this stage reads (asked into L2 at the tile's start)
        if (kSpec != 2 && ok0) {
            cw = load_carry_v<pk, kSpec>(A, 0, kr);
            cu = load_carry_v<pk, kSpec>(A, 1, kr);
            cv = load_carry_v<pk, kSpec>(A, 2, kr);
        }
        // right sides: bed slope (half the corner sums' differences), friction, dispersion
        const pk dd = depth_pair(A, Bb);
        const pk gh = mul2(kc(A, kcMHalfG), hb);
        pk F = fma2(mul2(gh, sx), kc(A, kcRdx), dv[1]);
        pk Gq = fma2(mul2(gh, sy), kc(A, kcRdy), dv[2]);
        if (friction != kFricNone) friction_v<pk>(A, friction, hb, u[2], u[1], F, Gq);
        pk Fs = 0, Gs = 0;
        if (bsnq) {
            const pk dN = depth_pair(A, bbar_pair(A, e1, e2));
            float a, b;
            un(dd, a, b);
            float dl = __shfl_up_sync(0xffffffffu, b, 1), dr = __shfl_down_sync(0xffffffffu, a, 1);
            if (atW) dl = pe[r].w;
            if (atE) dr = pe[r].w;
            const pk ddx = mul2(mk(b - dl, dr - a), kc(A, kcHrdx)), ddy = mul2(sub2(dN, dS), kc(A, kcHrdy));
            Around<pk> e = aroundv<kPS>(pw, u[0], cn[0], ldv(pw - kPS));
            e.nn = uu;
            e.ss = ldv(pw - 2 * kPS);
            eta_terms_v(A, e, dd, ddx, ddy, F, Gq);
            Fs = mixed_term_v(A, aroundv<kPQ>(pQ, u[1], cn[1], ldv(pQ - kPQ)), dd, ddx, ddy);
            Gs = mixed_term_v(A, aroundv<kPS>(pw + oP, u[2], cn[2], ldv(pw + oP - kPS)), dd, ddx, ddy);
        }
        // update
        const pk dw = advance_v<pk, kSpec>(A, 0, u[0], dv[0], 0, kr, cw, ok0);
        const pk dU = advance_v<pk, kSpec>(A, 1, 0, F, Fs, kr, cu, ok0);
        const pk dV = advance_v<pk, kSpec>(A, 2, 0, Gq, Gs, kr, cv, ok0);
        float a, b, B0, B1;
        un(kSpec != 0 ? dw : add2(u[0], dw), a, b);
        un(Bb, B0, B1);
        if (a < B0) a = B0;                  // Reading A-D1
        if (b < B1) b = B1;
        if (sponge_tile) {
            const int j = y0 + r0 + r;
            float d0, d1;
            un(dd, d0, d1);
            if (ok0) {
                const float gam = sponge_gamma<float>(C, G, i, j);
                if (gam < 1.f && d0 > 0.f) a = fma(gam, sub_r(a, ws), ws);
            }
            if (ok1) {
                const float gam = sponge_gamma<float>(C, G, i + 1, j);
                if (gam < 1.f && d1 > 0.f) b = fma(gam, sub_r(b, ws), ws);
            }
        }
        if (ok0) {
            sto(A.w_out, kr, mk(a, b));
            sto(A.U_out, kr, dU);
        }
        *reinterpret_cast<pk *>(pv) = dV;
        // dry bits: of the row (two words), of the columns where any is set
        const bool dry0 = ok0 && a - B0 <= 0.f, dry1 = ok1 && b - B1 <= 0.f;
        uint32_t bits = 0u;
        if (__any_sync(0xffffffffu, dry0 || dry1)) {
            const uint32_t e = __ballot_sync(0xffffffffu, dry0), o = __ballot_sync(0xffffffffu, dry1);
            const int sh = lane == 1 ? 16 : 0;
            bits = spread_bits(e >> sh) | (spread_bits(o >> sh) << 1);
            if (dry0) atomicOr(&sm.col[2 * lane], 1u << (r0 + r));
            if (dry1) atomicOr(&sm.col[2 * lane + 1], 1u << (r0 + r));
        }
        if (lane < 2 && (x0 >> 5) + lane < G.nwx)
            A.mask_r[(size_t)(y0 + r0 + r) * G.nwx + (x0 >> 5) + lane] = bits;
        // one row up
{
            qn[0] = uu;
            qn[1] = ldv(pQ + 2 * kPQ);
            qn[2] = ldv(pw + oP + 2 * kPS);
        }
        dS = dd;
        pw += kPS;
        pQ += kPQ;
        pb += kPB;
        pv += kPW;
        kr += (unsigned)G.px >> 1;
    }
    }
    // ---- 5. the V* increment along columns: the warp's own rows, four (or
    //         two) at a time; rows beyond the grid fall into the columns' padding
    __syncwarp();
    if (rows > 0) {
        const float *v = sm.V + r0 * kPW + 2 * lane;
        float *o0 = A.Vc_out + (size_t)i * G.py + y0 + r0, *o1 = o0 + G.py;
        if constexpr (kR % 4 == 0) {
#pragma unroll
            for (int r = 0; r < kR; r += 4) {
                float a[4], b[4];
#pragma unroll
                for (int u = 0; u < 4; u++) un(ldp(v + (r + u) * kPW), a[u], b[u]);
                if (ok0) *reinterpret_cast<float4 *>(o0 + r) = make_float4(a[0], a[1], a[2], a[3]);
                if (ok1) *reinterpret_cast<float4 *>(o1 + r) = make_float4(b[0], b[1], b[2], b[3]);
            }
        } else {
#pragma unroll
            for (int r = 0; r < kR; r += 2) {
                float a[2], b[2];
#pragma unroll
                for (int u = 0; u < 2; u++) un(ldp(v + (r + u) * kPW), a[u], b[u]);
                if (ok0) *reinterpret_cast<float2 *>(o0 + r) = make_float2(a[0], a[1]);
                if (ok1) *reinterpret_cast<float2 *>(o1 + r) = make_float2(b[0], b[1]);
            }
        }
    }
    __syncthreads();
    if (tid < kPW && x0 + tid < nx) {
        const size_t word = (size_t)(x0 + tid) * G.nwy + (y0 >> 5);
        if constexpr (TH == 32) A.mask_c[word] = sm.col[tid];
        else if constexpr (TH == 16) reinterpret_cast<uint16_t *>(A.mask_c)[2 * word + ((y0 >> 4) & 1)] = (uint16_t)sm.col[tid];
        else reinterpret_cast<uint8_t *>(A.mask_c)[4 * word + ((y0 >> 3) & 3)] = (uint8_t)sm.col[tid];
    }
}

}  // namespace
}  // namespace cel
