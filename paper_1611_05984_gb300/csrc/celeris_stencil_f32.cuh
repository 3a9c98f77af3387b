// The FP32 stencil stage over one tile: 64 columns, a lane owning two
// neighbouring cells of a row, a warp kR consecutive rows.
//
// The FP32 stencil is bound by instruction issue, so the layout is the one
// with the fewest instructions per cell:
//   * two cells per lane: additions, multiplications and fused
//     multiply-adds on both at once (.f32x2), 64-bit loads and stores of
//     shared and global memory, and one set of addresses, branches and loop
//     counts for two cells;
//   * a warp marches up its rows, so the reconstruction and fluxes along y,
//     the differences of the rows below and the bed's corner sums stay in
//     registers; a cell's x-fluxes come from its own reconstruction and its
//     left neighbour's (shuffles), and none goes through shared memory;
//   * the mixed and third differences of Eq. 10-13 are differences between
//     rows of each row's own x-differences.
// The faces at the tile's west and east edges, which need cells of the
// neighbouring tiles' lanes, are computed first, one (side, row) per lane.
//
// A face's flux does not depend on which warp or variant computes it (the
// row's one branch only skips what it would not do), so tiles of different
// heights give the same bits.
//
// Per cell about 455 thread instructions in the predictor and 410 in the
// corrector (865 and 800 with a cell per thread and the fluxes in shared
// memory).  128 registers, no spills, 4 blocks of 128 threads per SM: at 16
// warps per SM it is bound by the latency of its own chains (0.6 of the issue
// slots; 0.35 of the FMA pipe).  Mean of both stages, with events around the
// launches: 2048 x 2048 cells 115 -> 96 us, 8192 x 8192 1664 -> 1258 us.
#pragma once
#include "celeris_internal.cuh"
#include "celeris_physics.cuh"

namespace cel {
namespace {

using pk = unsigned long long;   // two floats: the cells x and x + 1

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
__device__ __forceinline__ pk kc(const StencilArgs<float> &A, int k) { return *reinterpret_cast<const pk *>(&A.kk.v[k]); }
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
__device__ __forceinline__ float min4(float a, float b, float c, float d)
{
    float r;
    asm("min.ftz.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return fminf(r, d);
}
__device__ __forceinline__ pk ldp(const float *p) { return *reinterpret_cast<const pk *>(p); }
// The same, read again even where the value was read before.
__device__ __forceinline__ pk ldv(const float *p)
{
    pk r;
    asm volatile("ld.volatile.shared.b64 %0, [%1];" : "=l"(r) : "r"((unsigned)__cvta_generic_to_shared(p)));
    return r;
}
// pair k of a global array
__device__ __forceinline__ pk ldo(const float *p, unsigned k) { return reinterpret_cast<const pk *>(p)[k]; }
__device__ __forceinline__ void sto(float *p, unsigned k, pk v) { reinterpret_cast<pk *>(p)[k] = v; }

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

// The history a stage reads for two cells (Carry, twice).
struct CarryPair {
    pk a, b, r1, r2, p1, p2, Y;
};

template <int kSpec>
__device__ __forceinline__ CarryPair load_carry_pair(const StencilArgs<float> &A, int v, unsigned k)
{
    const int kind = kSpec == 1 ? kAB3 : (kSpec == 2 ? kAM4 : A.kind);
    const bool ring = kSpec != 0 ? true : A.ring != 0;
    CarryPair c;
    c.a = c.b = c.r1 = c.r2 = c.p1 = c.p2 = c.Y = 0;
    if (kind == kAM4) {
        c.Y = ldo(A.Y[v], k);
    } else if (ring) {
        if (kind == kAB3) {
            c.r1 = ldo(A.R1[v], k);
            c.r2 = ldo(A.R2[v], k);
        }
        if (v > 0 && kind != kEuler0) {
            c.p1 = ldo(A.F1[v], k);
            if (kind == kAB3) c.p2 = ldo(A.F2[v], k);
        }
    } else if (kind == kEuler1) {
        c.a = ldo(A.a[v], k);
    } else if (kind == kAB3) {
        c.a = ldo(A.a[v], k);
        c.b = ldo(A.b[v], k);
    }
    return c;
}

// advance() for two cells; the history is written where ok.
template <int kSpec>
__device__ __forceinline__ pk advance_pair(const StencilArgs<float> &A, int v, pk X0, pk R, pk Phi, unsigned k,
                                           const CarryPair &c, bool ok)
{
    const int kind = kSpec == 1 ? kAB3 : (kSpec == 2 ? kAM4 : A.kind);
    const bool ring = kSpec != 0 ? true : A.ring != 0;
    if (kind == kAM4) {
        const pk s = fma2(kc(A, kcAm0), R, c.Y);
        return v > 0 ? add2(s, Phi) : s;
    }
    pk D;
    if (ring) {
        if (ok) {
            sto(A.R0[v], k, R);
            if (v > 0) sto(A.F0[v], k, Phi);
        }
        if (kind != kAB3) {
            D = mul2(kc(A, kcDt), R);
            if (kind == kEuler1 && v > 0) D = add2(D, sub2(Phi, c.p1));
        } else {
            D = fma2(kc(A, kcAb2), c.r2, fma2(kc(A, kcAb1), c.r1, mul2(kc(A, kcAb0), R)));
            pk y = fma2(kc(A, kcAm3), c.r2, fma2(kc(A, kcAm2), c.r1, mul2(kc(A, kcAm1), R)));
            if (v > 0) {
                D = add2(D, fma2(kc(A, kcTwo), Phi, fma2(kc(A, kcMThree), c.p1, c.p2)));
                y = sub2(y, Phi);
            } else {
                y = add2(X0, y);
            }
            if (ok) sto(A.Y[v], k, y);
        }
        return D;
    }
    pk na;
    if (kind == kEuler0) {
        D = mul2(kc(A, kcDt), R);
        na = Phi;
    } else {
        if (kind == kEuler1) D = add2(mul2(kc(A, kcDt), R), sub2(Phi, c.a));
        else D = add2(fma2(kc(A, kcTwo), Phi, mul2(kc(A, kcAb0), R)), add2(c.a, c.b));
        na = fma2(kc(A, kcMThree), Phi, mul2(kc(A, kcAb1), R));
    }
    if (ok) {
        sto(A.a[v], k, na);
        sto(A.b[v], k, fma2(kc(A, kcAb2), R, Phi));
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

// KP07 step 3 on two faces (face_flux_step): left states L, depths hL, right
// states R, depths hR; H = (mass, normal, tangential momentum).  kWet: every
// depth reaches eps^(1/4) (no branch); else each face takes its own form.
template <bool kWet>
__device__ __forceinline__ void flux_pair(const StencilArgs<float> &A, const pk L[3], pk hL, const pk R[3], pk hR,
                                          pk H[3])
{
    float l0, l1, r0, r1, gl0, gl1, gr0, gr1;
    un(hL, l0, l1);
    un(hR, r0, r1);
    const pk ghL = mul2(kc(A, kcG), hL), ghR = mul2(kc(A, kcG), hR);
    un(ghL, gl0, gl1);
    un(ghR, gr0, gr1);
    const pk sL = mk(sqrtf(gl0), sqrtf(gl1)), sR = mk(sqrtf(gr0), sqrtf(gr1));
    pk nL = L[1], tL = L[2], nR = R[1], tR = R[2], uL, vL, uR, vR;
    if (kWet) {
        const pk kL = mk(rcp_r(l0), rcp_r(l1)), kR = mk(rcp_r(r0), rcp_r(r1));
        uL = mul2(kL, nL);
        vL = mul2(kL, tL);
        uR = mul2(kR, nR);
        vR = mul2(kR, tR);
    } else {
        // a face with both depths at eps^(1/4) or above as in the other form
        const bool w0 = fminf(l0, r0) >= A.c.hwet, w1 = fminf(l1, r1) >= A.c.hwet;
        const float eps = A.c.eps;
        const pk kL = mk(w0 ? rcp_r(l0) : desing(l0, eps), w1 ? rcp_r(l1) : desing(l1, eps));
        const pk kR = mk(w0 ? rcp_r(r0) : desing(r0, eps), w1 ? rcp_r(r1) : desing(r1, eps));
        uL = mul2(kL, nL);
        vL = mul2(kL, tL);
        uR = mul2(kR, nR);
        vR = mul2(kR, tR);
        auto pick = [&](pk &q, pk k) {
            float a, b, c, d;
            un(q, a, b);
            un(k, c, d);
            q = mk(w0 ? a : c, w1 ? b : d);
        };
        pick(nL, mul2(hL, uL));
        pick(tL, mul2(hL, vL));
        pick(nR, mul2(hR, uR));
        pick(tR, mul2(hR, vR));
    }
    float p0, p1, q0, q1;
    un(add2(uL, sL), p0, p1);
    un(add2(uR, sR), q0, q1);
    const pk ap = mk(max_zero(p0, q0), max_zero(p1, q1));
    un(sub2(uL, sL), p0, p1);
    un(sub2(uR, sR), q0, q1);
    const pk am = mk(min_zero(p0, q0), min_zero(p1, q1));
    float d0, d1;
    un(sub2(am, ap), d0, d1);   // -(a+ - a-)
    // where both sides are dry (Reading A-F1) all terms are 0 and so is the flux
    const pk ninv = kWet ? mk(rcp_r(d0), rcp_r(d1)) : mk(rcp_r(fminf(d0, -1e-30f)), rcp_r(fminf(d1, -1e-30f)));
    const pk beta = mul2(am, ninv), ab = mul2(ap, beta);
    const pk FL1 = fma2(kc(A, kcHalf), mul2(ghL, hL), mul2(nL, uL)), FR1 = fma2(kc(A, kcHalf), mul2(ghR, hR), mul2(nR, uR));
    const pk FL2 = mul2(nL, vL), FR2 = mul2(nR, vR);
    H[0] = fma2(ab, sub2(L[0], R[0]), fma2(beta, sub2(nR, nL), nL));
    H[1] = fma2(ab, sub2(nL, nR), fma2(beta, sub2(FR1, FL1), FL1));
    H[2] = fma2(ab, sub2(tL, tR), fma2(beta, sub2(FR2, FL2), FL2));
}

// Friction's factor of (P, Q), negated: two cells with depths hb.
template <bool kWet>
__device__ __forceinline__ pk friction_pair(const StencilArgs<float> &A, int law, pk hb, pk P, pk Q)
{
    float h0, h1, m0, m1;
    un(hb, h0, h1);
    un(fma2(Q, Q, mul2(P, P)), m0, m1);
    pk k;
    if (kWet) {
        k = mk(rcp_r(h0), rcp_r(h1));
    } else {
        const float eps = A.c.eps, hw = A.c.hwet;
        k = mk(h0 >= hw ? rcp_r(h0) : desing(fmaxf(h0, 0.f), eps), h1 >= hw ? rcp_r(h1) : desing(fmaxf(h1, 0.f), eps));
    }
    pk f = mul2(mul2(k, k), mk(sqrtf(m0), sqrtf(m1)));
    if (law == kFricManning) {
        float k0, k1;
        un(k, k0, k1);
        f = mul2(f, mk(cbrt_r(k0), cbrt_r(k1)));
    }
    return mul2(f, kc(A, kcMFric));
}

__device__ __forceinline__ float least(pk a, pk b)
{
    float a0, a1, b0, b1;
    un(a, a0, a1);
    un(b, b0, b1);
    return min4(a0, a1, b0, b1);
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

// The x-differences of a row that the rows beside it combine (central
// differences of w, P and Q, second difference of w, undivided).
struct DiffRow {
    pk w, ww, P, Q;
};

__device__ __forceinline__ DiffRow diff_row(const SideRow &s, pk w, pk P, pk Q)
{
    DiffRow d;
    float a, b;
    un(w, a, b);
    const pk m = mk(s.wl, a), p = mk(b, s.wr);
    d.w = sub2(p, m);
    d.ww = sub2(sub2(p, w), sub2(w, m));
    un(P, a, b);
    d.P = sub2(mk(b, s.pr), mk(s.pl, a));
    un(Q, a, b);
    d.Q = sub2(mk(b, s.qr), mk(s.ql, a));
    return d;
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

// One tile, kPThreads threads (tid 0 .. kPThreads - 1), bar() the barrier of
// these threads.
template <int kSpec, int kR, typename Bar>
__device__ __forceinline__ void stencil_tile_pair(const StencilArgs<float> &A, const int x0, const int y0,
                                                  unsigned char *smem_raw, const int tid, const Bar &bar)
{
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
    bar();

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
        bar();   // the corner columns' x-ghosts
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
    if (westT || eastT || southT || northT) bar();

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
        face_flux_step(C.g, C.eps, C.hwet, hi[0], hi[1], hi[2], dh, lo2[0], lo2[1], lo2[2], dl2, H);
        // the cell beyond: f - 1 on the west, f on the east
        const float Bb = side ? cell_bbar(c1, c2, e1, e2) : cell_bbar(c0, c1, e0, e1);
        sm.edge[side][r] = make_float4(H[0], H[1], H[2], fmaxf(C.ws - Bb, 0.f));
    }
    __syncwarp();

    // ---- 4. the rows.  What a row shares with the next and is dearer to
    //         read again than to keep: the next row's cells, the fluxes and
    //         high sides along y, the x-differences of the row below.
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
    DiffRow below;                 // x-differences of row r - 1
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
        flux_pair<false>(A, hm, dm, lo, dl, Hs);
        if (bsnq) {
            below = diff_row(side_row(pw - kPS, pw + oP - kPS, pQ - kPQ), q1[0], q1[2], q1[1]);
            dS = depth_pair(A, bbar_pair(A, cm, c0));
        }
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
        DiffRow here;
        pk w3, Bx0, Bx1, sx;                 // w(x + 2) - w(x - 2); face beds; their sums' differences
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
            here.w = sub2(qp[0], qm[0]);
            here.ww = sub2(sub2(qp[0], q[0]), sub2(q[0], qm[0]));
            here.P = sub2(qp[1], qm[1]);
            here.Q = sub2(qp[2], qm[2]);
            w3 = sub2(mk(side.wr, side.wrr), mk(side.wll, side.wl));
            recon_pair(A, qm, q0, qp, Bx0, Bx1, lx, hx, dlx, dhx);
        }
        const pk Bb = bbar_pair(A, c0, c1), sy = sub2(c1.h, c0.h), hb = sub2(q[0], Bb);
        // Fluxes through the north faces and the west faces, and friction:
        // one branch for the row, on whether every depth reaches eps^(1/4)
        // (then no fix is due, and a cell's own depth, the mean of its
        // faces', reaches it too).
        pk Hn[3], H[3], fr = 0;
        const float thin = fminf(fminf(least(dly, dhy), least(dlx, dhx)), fminf(px_(dhi), py_(dhi)));
        if (__all_sync(0xffffffffu, thin >= C.hwet)) {
            const pk Lx[3] = {from_left(hx[0]), from_left(hx[1]), from_left(hx[2])};
            const pk dL = from_left(dhx);
            flux_pair<true>(A, hi, dhi, ly, dly, Hn);
            flux_pair<true>(A, Lx, dL, lx, dlx, H);
            if (friction != kFricNone) fr = friction_pair<true>(A, friction, hb, q[2], q[1]);
        } else {
            fix_pair(qn[0], By0, By1, ly[0], hy[0], dly, dhy);
            fix_pair(q[0], Bx0, Bx1, lx[0], hx[0], dlx, dhx);
            const pk Lx[3] = {from_left(hx[0]), from_left(hx[1]), from_left(hx[2])};
            const pk dL = from_left(dhx);
            flux_pair<false>(A, hi, dhi, ly, dly, Hn);
            flux_pair<false>(A, Lx, dL, lx, dlx, H);
            if (friction != kFricNone) fr = friction_pair<false>(A, friction, hb, q[2], q[1]);
        }
        CarryPair cw, cu, cv;
        if (kSpec == 2 && ok0) {
            cw = load_carry_pair<kSpec>(A, 0, kr);
            cu = load_carry_pair<kSpec>(A, 1, kr);
            cv = load_carry_pair<kSpec>(A, 2, kr);
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
            cw = load_carry_pair<kSpec>(A, 0, kr);
            cu = load_carry_pair<kSpec>(A, 1, kr);
            cv = load_carry_pair<kSpec>(A, 2, kr);
        }
        // right sides: bed slope (half the corner sums' differences), friction, dispersion
        const pk dd = depth_pair(A, Bb);
        pk F = fma2(fr, u[2], fma2(mul2(hb, kc(A, kcMHgx)), sx, dv[1]));
        pk Gq = fma2(fr, u[1], fma2(mul2(hb, kc(A, kcMHgy)), sy, dv[2]));
        pk Fs = 0, Gs = 0;
        if (bsnq) {
            const pk dN = depth_pair(A, bbar_pair(A, e1, e2));
            const DiffRow above = diff_row(side_row(pw + kPS, pw + oP + kPS, pQ + kPQ), cn[0], cn[2], cn[1]);
            const pk wS = ldp(pw - kPS), wSS = ldp(pw - 2 * kPS), PS = ldp(pw + oP - kPS), QS = ldp(pQ - kPQ);
            float a, b;
            un(dd, a, b);
            float dl = __shfl_up_sync(0xffffffffu, b, 1), dr = __shfl_down_sync(0xffffffffu, a, 1);
            if (atW) dl = pe[r].w;
            if (atE) dr = pe[r].w;
            const pk dDx = mk(b - dl, dr - a), dDy = sub2(dN, dS);
            const pk two = kc(A, kcTwo), mtwo = kc(A, kcMTwo);
            const pk gy = sub2(cn[0], wS);
            const pk eyy = sub2(sub2(cn[0], u[0]), sub2(u[0], wS));
            const pk eyyy = fma2(mtwo, gy, sub2(uu, wSS));
            const pk exxx = fma2(mtwo, here.w, w3);
            const pk exy = mul2(kc(A, kcQ), sub2(above.w, below.w));
            const pk exyy = fma2(mtwo, here.w, add2(above.w, below.w));
            const pk exxy = sub2(above.ww, below.ww);
            // K d^2 / (2 dx) [A (d exxx + 2 d_x exx) + B (d exyy + d_x eyy + d_y exy / 4)], A = 1/dx^2, B = 1/dy^2
            const pk d2 = mul2(dd, dd), Ax = kc(A, kcRdx2), By = kc(A, kcRdy2);
            const pk x1 = fma2(mul2(two, dDx), here.ww, mul2(dd, exxx));
            const pk x2 = fma2(dDy, exy, fma2(dDx, eyy, mul2(dd, exyy)));
            const pk y1 = fma2(mul2(two, dDy), eyy, mul2(dd, eyyy));
            const pk y2 = fma2(dDx, exy, fma2(dDy, here.ww, mul2(dd, exxy)));
            F = fma2(mul2(d2, kc(A, kcKx)), fma2(By, x2, mul2(Ax, x1)), F);
            Gq = fma2(mul2(d2, kc(A, kcKy)), fma2(Ax, y2, mul2(By, y1)), Gq);
            const pk dc = mul2(dd, kc(A, kcC6)), m1 = mul2(dc, dDx), m2 = mul2(dc, dDy), m3 = mul2(d2, kc(A, kcB3xy));
            Fs = fma2(m3, sub2(above.Q, below.Q), fma2(m2, here.Q, mul2(m1, sub2(cn[1], QS))));
            Gs = fma2(m3, sub2(above.P, below.P), fma2(m1, sub2(cn[2], PS), mul2(m2, here.P)));
        }
        // update
        const pk dw = advance_pair<kSpec>(A, 0, u[0], dv[0], 0, kr, cw, ok0);
        const pk dU = advance_pair<kSpec>(A, 1, 0, F, Fs, kr, cu, ok0);
        const pk dV = advance_pair<kSpec>(A, 2, 0, Gq, Gs, kr, cv, ok0);
        float a, b, B0, B1;
        un(kSpec == 2 ? dw : add2(u[0], dw), a, b);   // the AM4 base of w holds w^n
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
        below = here;
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
    bar();
    if (tid < kPW && x0 + tid < nx) {
        const size_t word = (size_t)(x0 + tid) * G.nwy + (y0 >> 5);
        if constexpr (TH == 32) A.mask_c[word] = sm.col[tid];
        else if constexpr (TH == 16) reinterpret_cast<uint16_t *>(A.mask_c)[2 * word + ((y0 >> 4) & 1)] = (uint16_t)sm.col[tid];
        else reinterpret_cast<uint8_t *>(A.mask_c)[4 * word + ((y0 >> 3) & 3)] = (uint8_t)sm.col[tid];
    }
}

}  // namespace
}  // namespace cel
