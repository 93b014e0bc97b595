// Per-row arithmetic of the reverse stencil, shared by the direct-load
// (adjoint_kernel.cu) and TMA-staged (adjoint_tma.cu) adjoint kernels so the
// two give bit-identical gradients.  The caller supplies the values of a
// lane's four cells from wherever it staged them.
//
// Straight-line code: every link's partials are computed in full and the
// branch the forward step took (dry link, limiter, outflow clip) is applied
// by selection, so rows that mix wet and dry links cost the warp no
// divergent paths.  The roughness enters Eq. 2 only through n_link^2, so
// n_link dq'/dn_link = -2 q' fric / D needs no division by n_link, and
// dq'/dq is formed from b h^(-7/3) rather than by dividing by q.
//
// The stencil is bound by issue slots (968 warp instructions a row of 128
// cells), so links go in pairs through the two-wide FP32 instructions, the
// link west of the span is computed by every lane in line with the others,
// and rows without a row below and spans with the grid's last column are
// compiled apart.  Every rounding is spelled out (which products are fused
// into which sums), so the instruction chosen cannot move a gradient.
#pragma once

#include "flood_internal.cuh"
#include "quad.cuh"
#include "sum2.cuh"

namespace flood {

// Partials of one new link flux q' (Eq. 2-3 and the limiter): with respect
// to the depths of its two cells and its old flux, and g2 = n_link dq'/dn_link.
struct LinkD {
    float dh1, dh2, dq, g2;
};

// Two interior links at once (the forward arithmetic and branch decisions of
// link2_q).  ns: the sum of the two cells' roughness; up, dn: their depths
// times dx / (4 dt).
struct Link2D {
    float2 dh1, dh2, dq, g2;
};

template <int LIM>
__device__ __forceinline__ Link2D link2_d(float2 h1, float2 z1, float2 h2, float2 z2, float2 q, float2 ns,
                                          float2 up, float2 dn, const Link2K& k, float dx_4dt)
{
    // the forward quantities, rounded exactly as link2_q rounds them
    const float2 dz = sub2(z2, z1, k.m1);
    const float2 a1 = sub2(h1, make_float2(fmaxf(dz.x, 0.0f), fmaxf(dz.y, 0.0f)), k.m1);
    const float2 a2 = __fadd2_rn(h2, make_float2(fminf(dz.x, 0.0f), fminf(dz.y, 0.0f)));
    const float2 hf = make_float2(fmaxf(a1.x, a2.x), fmaxf(a1.y, a2.y));
    const float2 dS = __fadd2_rn(dz, sub2(h2, h1, k.m1));
    const float2 nt = __fmul2_rn(k.ngdt_dx, hf);
    const float2 num = __ffma2_rn(nt, dS, q);
    const float2 nl = __fmul2_rn(k.sh, ns);
    const float2 b = __fmul2_rn(k.gdt, __fmul2_rn(nl, nl));
    const float2 e = __fmul2_rn(k.p73, make_float2(lg2_approx(hf.x), lg2_approx(hf.y)));
    const float2 ih = make_float2(fminf(ex2_approx(e.x), 1.0e30f), fminf(ex2_approx(e.y), 1.0e30f));
    const float2 fr = __fmul2_rn(__fmul2_rn(b, q), ih);  // the friction, with q's sign
    const float2 invD =
        make_float2(rcp_approx(__fadd_rn(1.0f, fabsf(fr.x))), rcp_approx(__fadd_rn(1.0f, fabsf(fr.y))));
    const float2 qs = __fmul2_rn(num, invD);
    // dq'/dhf = -G dS / D + (7/3) q' fric / (D hf);  dq'/d(dx S) = -G hf / D
    // dq'/dq = (1 - q' b h^(-7/3) sgn q) / D;        n dq'/dn = -2 q' fric / D
    const float2 u = __fmul2_rn(qs, invD);
    const float2 qt = make_float2(__fmul_rn(u.x, fabsf(fr.x)), __fmul_rn(u.y, fabsf(fr.y)));
    const float2 w = __fmul2_rn(__fmul2_rn(dup2(2.33333333f), qt), make_float2(rcp_approx(hf.x), rcp_approx(hf.y)));
    const float2 dd = __ffma2_rn(__fmul2_rn(k.ngdt_dx, dS), invD, w);
    // Eq. 3's tie goes to the first argument
    const bool fx = a1.x >= a2.x, fy = a1.y >= a2.y;
    const float dh1x = __fmaf_rn(-nt.x, invD.x, fx ? dd.x : 0.0f), dh1y = __fmaf_rn(-nt.y, invD.y, fy ? dd.y : 0.0f);
    const float2 dh2 = __ffma2_rn(nt, invD, make_float2(fx ? 0.0f : dd.x, fy ? 0.0f : dd.y));
    const float2 ub = __fmul2_rn(u, __fmul2_rn(b, ih));
    auto signed_as = [](float v, float s) {
        return s != 0.0f ? __uint_as_float(__float_as_uint(v) ^ (__float_as_uint(s) & 0x80000000u)) : 0.0f;
    };
    const float2 dq = sub2(invD, make_float2(signed_as(ub.x, q.x), signed_as(ub.y, q.y)), k.m1);
    const float2 g2 = __fmul2_rn(dup2(-2.0f), qt);
    bool hix = false, hiy = false, lox = false, loy = false;
    if (LIM) {
        hix = qs.x > up.x;
        hiy = qs.y > up.y;
        lox = qs.x < -dn.x;
        loy = qs.y < -dn.y;
    }
    const bool wx = hf.x > k.h_eps, wy = hf.y > k.h_eps;
    const bool frx = wx && !(hix || lox), fry = wy && !(hiy || loy);
    Link2D r;
    r.dh1 = make_float2(frx ? dh1x : ((wx && hix) ? dx_4dt : 0.0f), fry ? dh1y : ((wy && hiy) ? dx_4dt : 0.0f));
    r.dh2 = make_float2(frx ? dh2.x : ((wx && lox) ? -dx_4dt : 0.0f), fry ? dh2.y : ((wy && loy) ? -dx_4dt : 0.0f));
    r.dq = make_float2(frx ? dq.x : 0.0f, fry ? dq.y : 0.0f);
    r.g2 = make_float2(frx ? g2.x : 0.0f, fry ? g2.y : 0.0f);
    return r;
}

// One interior link, the same partials (for the link west of a span).
template <int LIM>
__device__ __forceinline__ LinkD link_d(float h1, float z1, float h2, float z2, float q, float nl,
                                        const FaceK& k)
{
    // the forward quantities, rounded exactly as link_q rounds them
    const float dz = __fsub_rn(z2, z1);
    const float a1 = __fsub_rn(h1, fmaxf(dz, 0.0f));
    const float a2 = __fadd_rn(h2, fminf(dz, 0.0f));
    const float hf = fmaxf(a1, a2);
    const float dS = __fadd_rn(dz, __fsub_rn(h2, h1));
    const float num = __fmaf_rn(-__fmul_rn(k.gdt_dx, hf), dS, q);
    const float b = __fmul_rn(k.gdt, __fmul_rn(nl, nl));
    const float ih = inv_h73(hf);
    const float fric = __fmul_rn(__fmul_rn(b, fabsf(q)), ih);
    const float invD = rcp_approx(__fadd_rn(1.0f, fric));
    const float qs = __fmul_rn(num, invD);
    const float u = __fmul_rn(qs, invD);
    const float qt = __fmul_rn(u, fric);
    const float t = __fmul_rn(k.gdt_dx, hf);
    const float dq_dhf = __fmaf_rn(-__fmul_rn(k.gdt_dx, dS), invD,
                                   __fmul_rn(__fmul_rn(2.33333333f, qt), rcp_approx(hf)));
    const bool first = a1 >= a2;  // Eq. 3's tie goes to the first argument
    const float dh1 = __fmaf_rn(t, invD, first ? dq_dhf : 0.0f);
    const float dh2 = __fmaf_rn(-t, invD, first ? 0.0f : dq_dhf);
    const float ub = __fmul_rn(u, __fmul_rn(b, ih));
    const float dq = __fsub_rn(invD, q > 0.0f ? ub : (q < 0.0f ? -ub : 0.0f));
    bool hi = false, lo = false;
    if (LIM) {
        hi = qs > __fmul_rn(h1, k.dx_4dt);
        lo = qs < -__fmul_rn(h2, k.dx_4dt);
    }
    const bool wet = hf > k.h_eps;
    const bool fr = wet && !(hi || lo);
    LinkD r;
    r.dh1 = fr ? dh1 : ((wet && hi) ? k.dx_4dt : 0.0f);
    r.dh2 = fr ? dh2 : ((wet && lo) ? -k.dx_4dt : 0.0f);
    r.dq = fr ? dq : 0.0f;
    r.g2 = fr ? -2.0f * qt : 0.0f;
    return r;
}

// Free-outflow link (ghost with the edge depth, as outflow_q): dh1 is the
// total derivative with respect to the edge cell's depth.
template <int LIM>
__device__ __forceinline__ LinkD outflow_d(float h, float q, float nl, const FaceK& k)
{
    const float num = __fmaf_rn(-__fmul_rn(k.gdt_dx, h), -k.edge_drop, q);
    const float b = __fmul_rn(k.gdt, __fmul_rn(nl, nl));
    const float ih = inv_h73(h);
    const float fric = __fmul_rn(__fmul_rn(b, fabsf(q)), ih);
    const float invD = rcp_approx(__fadd_rn(1.0f, fric));
    const float qs = __fmul_rn(num, invD);
    const float u = qs * invD;
    const float qt = u * fric;
    const float dh = __fmaf_rn(k.gdt_dx * k.edge_drop, invD, 2.33333333f * qt * rcp_approx(h));
    const float ub = u * (b * ih);
    const float dq = invD - (q > 0.0f ? ub : (q < 0.0f ? -ub : 0.0f));
    const bool hi = LIM && qs > __fmul_rn(h, k.dx_4dt);
    const bool wet = h > k.h_eps;
    const bool fr = wet && !hi && qs > 0.0f;  // only outward flow passes
    LinkD r;
    r.dh1 = fr ? dh : ((wet && hi) ? k.dx_4dt : 0.0f);
    r.dh2 = 0.0f;
    r.dq = fr ? dq : 0.0f;
    r.g2 = fr ? -2.0f * qt : 0.0f;
    return r;
}

// 1 / (sum of the roughness values a link's n_link is made of); a zero sum
// (no friction, so g2 = 0) gives a finite factor and a zero weight.
__device__ __forceinline__ float inv_nsum(float ns) { return rcp_approx(fmaxf(ns, 1.0e-30f)); }

__device__ __forceinline__ float masked(float h_after, float lam)
{
    return signbit(h_after) ? 0.0f : lam;  // clamped cells pass no sensitivity
}

// A row's values of a lane's four cells: depth, bed, roughness, and lambda~
// (the sensitivity to the depth after the step, zero where it was clamped).
struct AdjRow {
    Quad h, z, n, l;
};

// mu = lambda_q' + T (lambda~_2 - lambda~_1) of two links
__device__ __forceinline__ float2 mu2(float2 lq, float2 l1, float2 l2, float2 T, float2 m1)
{
    return __ffma2_rn(T, sub2(l2, l1, m1), lq);
}
__device__ __forceinline__ float2 inv_nsum2(float2 ns) { return make_float2(inv_nsum(ns.x), inv_nsum(ns.y)); }
__device__ __forceinline__ Quad scaled(const Quad& h, float s)
{
    return Quad{__fmul2_rn(h.a, dup2(s)), __fmul2_rn(h.b, dup2(s))};
}

// The strip's north links (the row U above the strip's first row C),
// recomputed: their contributions to the first row's depth and Manning
// sensitivities.
template <int LIM>
__device__ __forceinline__ void north_carry(const AdjRow& U, const Quad& qU, const Quad& lqU, const AdjRow& C, int c,
                                            int nx, const Link2K& k2, float T, const FaceK& k, Quad& carH,
                                            Quad& carN)
{
    const Quad uU = scaled(U.h, k.dx_4dt), uC = scaled(C.h, k.dx_4dt);
    auto pair = [&](float2 h1, float2 z1, float2 n1, float2 l1, float2 u1, float2 h2, float2 z2, float2 n2, float2 l2,
                    float2 u2, float2 q, float2 lq, float2& ch, float2& cn) {
        const float2 ns = __fadd2_rn(n1, n2);
        const Link2D d = link2_d<LIM>(h1, z1, h2, z2, q, ns, u1, u2, k2, k.dx_4dt);
        const float2 mu = mu2(lq, l1, l2, dup2(T), k2.m1);
        ch = __fmul2_rn(mu, d.dh2);
        cn = __fmul2_rn(__fmul2_rn(mu, d.g2), inv_nsum2(ns));
    };
    pair(U.h.a, U.z.a, U.n.a, U.l.a, uU.a, C.h.a, C.z.a, C.n.a, C.l.a, uC.a, qU.a, lqU.a, carH.a, carN.a);
    pair(U.h.b, U.z.b, U.n.b, U.l.b, uU.b, C.h.b, C.z.b, C.n.b, C.l.b, uC.b, qU.b, lqU.b, carH.b, carN.b);
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (c + j >= nx) quad_at(carH, j) = quad_at(carN, j) = 0.0f;
}

// Neighbours of a lane's four cells (E) or of the span's first cell (W, the
// same values in every lane): depth, bed, roughness, lambda~; W also the
// link's old flux and lambda.
struct AdjSide {
    float h, z, n, l, qx, lqx;
};

// One row of the reverse stencil for a lane's four cells.  C: this row, S:
// the row below (HAS_S: there is one), E: the cell east of the lane's last, W:
// the cell west of the span's first (west_halo: there is one).  Writes the
// sensitivities to the step's inputs (lh, lx, ly) and the Manning contribution
// (gnr), updates the north-link carries, and sets this row's rain partial (sum
// of lambda~) and scale partial (sum of mu n dq'/dn over the lane's links, to
// be divided by the scale).  FULL: the span lies wholly inside the grid with
// an interior link east of its last cell (c0 + 128 < nx).  RW: the rain
// partial weighs each cell by rw, the fraction of the rain that stays on it
// (land cover, Section 4.1).
template <bool HAS_S, bool FULL, int LIM, bool RW = false>
__device__ __forceinline__ void adjoint_row(const AdjRow& C, const AdjRow& S, const Quad& qx, const Quad& qy,
                                            const Quad& lqx, const Quad& lqy, const AdjSide& E, bool west_halo,
                                            const AdjSide& W, int c, int nx, int lane, float s, float s_half, float T,
                                            const FaceK& k, const Link2K& k2, int east_out, int south_out, Quad& carH,
                                            Quad& carN, float& gr_row, float& gs_row, Quad& lh, Quad& lx, Quad& ly,
                                            Quad& gnr, const Quad* rw = nullptr)
{
    const float2 T2 = dup2(T);
    const Quad uC = scaled(C.h, k.dx_4dt);
    // east links: mu = lambda_q' + T (lambda~_east - lambda~_here); per link
    // mu dq'/dh1 (this cell), mu dq'/dh2 (the east cell), mu dq'/dq, and the
    // Manning weight mu n dq'/dn / (sum of the n it is made of)
    Quad p1, p2, xE, wE, G;
    {
        const Quad h2{make_float2(C.h.a.y, C.h.b.x), make_float2(C.h.b.y, E.h)};
        const Quad z2{make_float2(C.z.a.y, C.z.b.x), make_float2(C.z.b.y, E.z)};
        const Quad l2{make_float2(C.l.a.y, C.l.b.x), make_float2(C.l.b.y, E.l)};
        const Quad u2{make_float2(uC.a.y, uC.b.x), make_float2(uC.b.y, __fmul_rn(E.h, k.dx_4dt))};
        const Quad ns{make_float2(__fadd_rn(C.n.a.x, C.n.a.y), __fadd_rn(C.n.a.y, C.n.b.x)),
                      make_float2(__fadd_rn(C.n.b.x, C.n.b.y), __fadd_rn(C.n.b.y, E.n))};
        auto pair = [&](float2 h, float2 z, float2 l, float2 u, float2 hh, float2 zz, float2 ll, float2 uu, float2 q,
                        float2 nn, float2 lq, float2& o1, float2& o2, float2& ox, float2& ow, float2& og) {
            const Link2D d = link2_d<LIM>(h, z, hh, zz, q, nn, u, uu, k2, k.dx_4dt);
            const float2 mu = mu2(lq, l, ll, T2, k2.m1);
            og = __fmul2_rn(mu, d.g2);
            o1 = __fmul2_rn(mu, d.dh1);
            o2 = __fmul2_rn(mu, d.dh2);
            ox = __fmul2_rn(mu, d.dq);
            ow = __fmul2_rn(og, inv_nsum2(nn));
        };
        pair(C.h.a, C.z.a, C.l.a, uC.a, h2.a, z2.a, l2.a, u2.a, qx.a, ns.a, lqx.a, p1.a, p2.a, xE.a, wE.a, G.a);
        pair(C.h.b, C.z.b, C.l.b, uC.b, h2.b, z2.b, l2.b, u2.b, qx.b, ns.b, lqx.b, p1.b, p2.b, xE.b, wE.b, G.b);
    }
    if (!FULL) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (c + j >= nx - 1) {  // the grid's last column: its outflow, and nothing past it
                LinkD d{0.0f, 0.0f, 0.0f, 0.0f};
                float mu = 0.0f, w = 0.0f;
                if (c + j == nx - 1) {
                    if (east_out)
                        d = outflow_d<LIM>(quad_at(C.h, j), quad_at(qx, j), __fmul_rn(s, quad_at(C.n, j)), k);
                    mu = __fmaf_rn(-T, quad_at(C.l, j), quad_at(lqx, j));
                    w = inv_nsum(quad_at(C.n, j));
                }
                quad_at(G, j) = __fmul_rn(mu, d.g2);
                quad_at(p1, j) = __fmul_rn(mu, d.dh1);
                quad_at(p2, j) = __fmul_rn(mu, d.dh2);
                quad_at(xE, j) = __fmul_rn(mu, d.dq);
                quad_at(wE, j) = __fmul_rn(quad_at(G, j), w);
            }
    }
    gs_row = __fadd_rn(__fadd_rn(__fadd_rn(G.a.x, G.a.y), G.b.x), G.b.y);
    // west link of the lane's first cell: the lane before's last east link; of
    // the span's first cell: the link across its west side, computed by all
    float pW, wW;
    {
        const float ns = __fadd_rn(W.n, C.n.a.x);
        const LinkD d = link_d<LIM>(W.h, W.z, C.h.a.x, C.z.a.x, W.qx, __fmul_rn(s_half, ns), k);
        const float mu = __fmaf_rn(T, __fsub_rn(C.l.a.x, W.l), W.lqx);
        const float pH = west_halo ? __fmul_rn(mu, d.dh2) : 0.0f;
        const float wH = west_halo ? __fmul_rn(__fmul_rn(mu, d.g2), inv_nsum(ns)) : 0.0f;
        pW = __shfl_up_sync(0xffffffffu, p2.b.y, 1);
        wW = __shfl_up_sync(0xffffffffu, wE.b.y, 1);
        if (lane == 0) {
            pW = pH;
            wW = wH;
        }
    }
    // south links: mu dq'/dh1 enters this row's sum fused, mu dq'/dh2 goes on
    // to the row below
    Quad muS, dS1, cH, wS;
    if (HAS_S) {
        const Quad uS = scaled(S.h, k.dx_4dt);
        auto pair = [&](float2 h, float2 z, float2 n, float2 l, float2 u, float2 hh, float2 zz, float2 nn, float2 ll,
                        float2 uu, float2 q, float2 lq, float2& om, float2& o1, float2& o2, float2& oy, float2& ow,
                        float2& og) {
            const float2 ns = __fadd2_rn(n, nn);
            const Link2D d = link2_d<LIM>(h, z, hh, zz, q, ns, u, uu, k2, k.dx_4dt);
            om = mu2(lq, l, ll, T2, k2.m1);
            o1 = d.dh1;
            o2 = __fmul2_rn(om, d.dh2);
            oy = __fmul2_rn(om, d.dq);
            og = __fmul2_rn(om, d.g2);
            ow = __fmul2_rn(og, inv_nsum2(ns));
        };
        pair(C.h.a, C.z.a, C.n.a, C.l.a, uC.a, S.h.a, S.z.a, S.n.a, S.l.a, uS.a, qy.a, lqy.a, muS.a, dS1.a, cH.a,
             ly.a, wS.a, G.a);
        pair(C.h.b, C.z.b, C.n.b, C.l.b, uC.b, S.h.b, S.z.b, S.n.b, S.l.b, uS.b, qy.b, lqy.b, muS.b, dS1.b, cH.b,
             ly.b, wS.b, G.b);
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            LinkD d{0.0f, 0.0f, 0.0f, 0.0f};
            if (south_out) d = outflow_d<LIM>(quad_at(C.h, j), quad_at(qy, j), __fmul_rn(s, quad_at(C.n, j)), k);
            const float mu = __fmaf_rn(-T, quad_at(C.l, j), quad_at(lqy, j));
            quad_at(muS, j) = mu;
            quad_at(dS1, j) = d.dh1;
            quad_at(cH, j) = __fmul_rn(mu, d.dh2);
            quad_at(ly, j) = __fmul_rn(mu, d.dq);
            quad_at(G, j) = __fmul_rn(mu, d.g2);
            quad_at(wS, j) = __fmul_rn(quad_at(G, j), inv_nsum(quad_at(C.n, j)));
        }
    }
    lh.a = __fadd2_rn(__ffma2_rn(muS.a, dS1.a,
                                 __fadd2_rn(__fadd2_rn(C.l.a, p1.a), make_float2(pW, p2.a.x))), carH.a);
    lh.b = __fadd2_rn(__ffma2_rn(muS.b, dS1.b,
                                 __fadd2_rn(__fadd2_rn(C.l.b, p1.b), make_float2(p2.a.y, p2.b.x))), carH.b);
    lx = xE;
    gnr.a = __fadd2_rn(__fadd2_rn(__fadd2_rn(wE.a, make_float2(wW, wE.a.x)), wS.a), carN.a);
    gnr.b = __fadd2_rn(__fadd2_rn(__fadd2_rn(wE.b, make_float2(wE.a.y, wE.b.x)), wS.b), carN.b);
    carH = cH;
    carN = wS;
    if (!FULL) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (c + j >= nx) {
                quad_at(lh, j) = quad_at(lx, j) = quad_at(ly, j) = quad_at(gnr, j) = 0.0f;
                quad_at(carH, j) = quad_at(carN, j) = quad_at(G, j) = 0.0f;
            }
    }
    gs_row = __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(gs_row, G.a.x), G.a.y), G.b.x), G.b.y);
    gr_row = 0.0f;
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (FULL || c + j < nx)
            gr_row = RW ? __fmaf_rn(quad_at(C.l, j), quad_at(*rw, j), gr_row) : __fadd_rn(gr_row, quad_at(C.l, j));
}

// The drainage partial of a lane's four cells in one row: lambda~ of the
// cells of a draining class (df = 1) that the step left wet.
__device__ __forceinline__ float drain_row(const Quad& lC, const Quad& ha, const float (&df)[4])
{
    float acc = 0.0f;
#pragma unroll
    for (int q = 0; q < 4; ++q) acc += quad_at(ha, q) > 0.0f ? quad_at(lC, q) * df[q] : 0.0f;
    return acc;
}

__device__ __forceinline__ Quad masked(const Quad& ha, const Quad& l)
{
    return Quad{make_float2(masked(ha.a.x, l.a.x), masked(ha.a.y, l.a.y)),
                make_float2(masked(ha.b.x, l.b.x), masked(ha.b.y, l.b.y))};
}

// The lanes' compensated partials of the warp, summed and added in FP64 to the
// warp's slot (one slot per span and strip): rain times rdt (the step's rain
// depth per unit multiplier), scale times rs (1 / scale), with land cover
// (gdpart) drainage times -dt.  In FP64 from the start, and with the division
// by the scale in every warp, this took 40 FP64 instructions of 64 cycles a
// strip: now the lanes sum in two FP32 words, the upper half of the warp the
// scale's, and five FP64 instructions finish all of them, a lane each (1024 x
// 1024, 300 steps and their reverse: 9.03 -> 8.54 ms; the gradients move by
// 5e-14, their error against FP64 not at all).
__device__ __forceinline__ void adjoint_partials(double* gpart, double* gdpart, int nslot, int m, int slot, int lane,
                                                 Sum2 rain, Sum2 scale, Sum2 drain, double rdt, double rs, double dt)
{
    const bool low = lane < 16;
    const Sum2 send = low ? scale : rain;
    Sum2 sum = low ? rain : scale;
    sum.merge(__shfl_xor_sync(0xffffffffu, send.hi, 16), __shfl_xor_sync(0xffffffffu, send.lo, 16));
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) {
        const float h = __shfl_xor_sync(0xffffffffu, sum.hi, off), l = __shfl_xor_sync(0xffffffffu, sum.lo, off);
        sum.merge(h, l);
    }
    if (gdpart) drain.warp_sum();
    if (lane == 1) sum = drain;
    double* const v = lane == 1 ? gdpart + (size_t)m * nslot + slot
                                : gpart + ((size_t)m * nslot + slot) * 2 + (lane >> 4);
    if ((lane & 15) == 0 || (lane == 1 && gdpart)) *v += sum.value() * (lane == 0 ? rdt : lane == 1 ? -dt : rs);
}

}  // namespace flood
