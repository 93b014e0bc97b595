// Reverse mode of the fused local-inertial step (extension beyond the
// paper): given the loss's sensitivities to the state after step j
// (lambda_{j+1} = dL/d(h, qx, qy)), produce those to the state before it
// (lambda_j) and accumulate dL/dn (per cell, per member), dL/d(rain
// multiplier) and dL/d(Manning scale).  The step length is held fixed (the
// recorded schedule); at every kink (Eq. 3's max, the limiter, the wet/dry
// test, the outflow clip, the negative-depth clamp) the derivative of the
// branch taken is used, ties in Eq. 3 going to the first argument.  A cell
// whose depth was clamped carries a negative zero in the recorded state,
// which is how this kernel knows that branch was taken.
//
// Layout and traversal mirror the forward kernel: a warp owns 128 columns
// (float4 per lane) of a strip of rows of one member and marches down; the
// west link comes from the neighbouring lane by shuffle (recomputed by lane 0
// at the span edge), the north link's contribution is carried from the row
// above (recomputed at the strip top).
//
// HBM traffic per member-cell-step: state before the step (12 B), depth after
// it (4 B), lambda in (12 B), lambda out (12 B), per-cell Manning gradient
// read + write (8 B), z and n shared per tile.
#include <type_traits>

#include "adjoint.cuh"
#include "adjoint_row.cuh"
#include "launch.cuh"

namespace flood {

namespace {

constexpr int kSpan = 128;

// RW: land cover (per-member Manning n fields, rain weighed by the runoff
// coefficient, drainage partials), with the registers of three CTAs per SM.
template <int WM, int WC, int LIM, bool RW = false>
__global__ void __launch_bounds__(32 * WM * WC, RW ? 3 : 4) adjoint_kernel(const AdjArgs a)
{
    const int lane = threadIdx.x;
    const int wm = threadIdx.y % WM;
    const int wc = threadIdx.y / WM;
    const int m = blockIdx.x * WM + wm;
    const int span = blockIdx.y * WC + wc;
    const int c0 = span * kSpan;
    pdl_launch();
    pdl_wait();
    if (m >= a.M || c0 >= a.nx) return;

    const int nx = a.nx, ny = a.ny, ld = a.ld;
    const size_t plane = a.plane, mstride = 3 * plane;
    const int c = c0 + 4 * lane;
    const bool act = c < nx;
    const int r0 = blockIdx.z * a.rows_per_strip;
    const int r1 = min(r0 + a.rows_per_strip, ny);
    const float* const lin = a.lam + ((size_t)a.lam_in * a.M + m) * mstride;
    float* __restrict__ lout = a.lam + ((size_t)(1 - a.lam_in) * a.M + m) * mstride;

    const int j = a.seg_end[m] - 1 - a.rev_i;
    if (j < a.seg_first) {  // member idle in this launch: carry lambda over
        if (act)
            for (int r = r0; r < r1; ++r)
                for (int k = 0; k < 3; ++k) {
                    const size_t o = k * plane + (size_t)r * ld + c;
                    *reinterpret_cast<float4*>(lout + o) = *reinterpret_cast<const float4*>(lin + o);
                }
        return;
    }
    const MemberPlan pl = a.log[(size_t)m * a.dt_log_cap + j];
    FaceK k;
    k.gdt_dx = pl.gdt_dx;
    k.gdt = pl.gdt;
    k.dx_4dt = pl.dx_4dt;
    k.h_eps = a.h_eps;
    k.edge_drop = a.edge_drop;
    k.limiter = a.limiter;
    k.q_in = 0.0f;  // no inflow boundary here
    k.in_r0 = k.in_r1 = 0;
    const float T = pl.dt_dx;
    const float s = a.scale[m];
    const float s_half = 0.5f * s;
    const bool interior = c0 + kSpan < nx;  // no east edge in this span

    // lambda and the states are the kernels' before this one, which may still run
    // when this one takes its places: plain loads.  (The read-only path is for
    // what stays as it is from a kernel's start to its end: bed, roughness.)
    const float* const st = a.seg + ((size_t)(j - a.seg_first) * a.M + m) * mstride;
    const float* const sh = st;
    const float* const sqx = st + plane;
    const float* const sqy = st + 2 * plane;
    const float* const h1p = st + (size_t)a.M * mstride;  // depth after the step
    const float* __restrict__ z = a.z;
    const float* __restrict__ n = a.n + (size_t)m * a.n_mstride;
    float* __restrict__ gn = a.gn ? a.gn + (size_t)m * plane : nullptr;
    const bool east_halo = (lane == 31) && (c + 4 < nx);

    const Link2K k2 = link2_k(k, s_half);
    auto ldg_quad = [](const float* p) -> Quad {
        const float4 v = ldg4(p);
        return Quad{make_float2(v.x, v.y), make_float2(v.z, v.w)};
    };
    // a row's values (lambda~: zero where the step clamped)
    auto load_row = [&](size_t o) -> AdjRow {
        return AdjRow{ld_quad(sh + o), ldg_quad(z + o), ldg_quad(n + o), masked(ld_quad(h1p + o), ld_quad(lin + o))};
    };
    const AdjRow none{quad_of(0.0f), quad_of(0.0f), quad_of(0.0f), quad_of(0.0f)};
    AdjRow C = none;
    Quad carH = quad_of(0.0f), carN = quad_of(0.0f);  // north link: mu*dh2, mu*dnl
    if (act) {
        const size_t o = (size_t)r0 * ld + c;
        C = load_row(o);
        if (r0 > 0) {  // the strip's north links, recomputed
            const size_t u = o - ld;
            north_carry<LIM>(load_row(u), ld_quad(sqy + u), ld_quad(lin + 2 * plane + u), C, c, nx, k2, T, k, carH,
                             carN);
        }
    }

    // FP32 compensated sums of the rows' partials (lambda~ for the rain
    // gradient, mu n dq'/dn for the scale gradient), widened to FP64 once per warp
    float gr_s = 0.0f, gr_c = 0.0f, gs_s = 0.0f, gs_c = 0.0f;
    float gd_s = 0.0f, gd_c = 0.0f;  // land cover: drainage partials
    for (int r = r0; r < r1; ++r) {
        const size_t o = (size_t)r * ld + c;
        const bool has_s = (r + 1 < ny);
        AdjRow S = none;
        Quad qxo = quad_of(0.0f), qyo = qxo, lqx = qxo, lqy = qxo;
        if (act) {
            if (has_s) S = load_row(o + ld);
            qxo = ld_quad(sqx + o);
            qyo = ld_quad(sqy + o);
            lqx = ld_quad(lin + plane + o);
            lqy = ld_quad(lin + 2 * plane + o);
        }
        AdjSide E{__shfl_down_sync(0xffffffffu, C.h.a.x, 1), __shfl_down_sync(0xffffffffu, C.z.a.x, 1),
                  __shfl_down_sync(0xffffffffu, C.n.a.x, 1), __shfl_down_sync(0xffffffffu, C.l.a.x, 1), 0.0f, 0.0f};
        if (east_halo) {
            const size_t e = o + 4;
            E.h = sh[e]; E.z = __ldg(z + e); E.n = __ldg(n + e);
            E.l = masked(h1p[e], lin[e]);
        }
        AdjSide W{0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        if (c0 > 0) {  // one cell for the whole warp
            const size_t w = (size_t)r * ld + c0 - 1;
            W.h = sh[w]; W.z = __ldg(z + w); W.n = __ldg(n + w);
            W.qx = sqx[w]; W.lqx = lin[plane + w];
            W.l = masked(h1p[w], lin[w]);
        }
        Quad lh, lx, ly, gnr;
        float gr_row, gs_row;
        Quad rwv = quad_of(0.0f);
        if (RW) {
            float dfv[4] = {0, 0, 0, 0};
            Quad haC = quad_of(0.0f);
            if (act) {
                rwv = ldg_quad(a.rw + o);
                const float4 d = ldg4(a.dflag + o);
                dfv[0] = d.x; dfv[1] = d.y; dfv[2] = d.z; dfv[3] = d.w;
                haC = ld_quad(h1p + o);
            }
            kahan_add(gd_s, gd_c, drain_row(C.l, haC, dfv));
        }
        auto row = [&](auto has_s_t, auto full_t) {
            adjoint_row<decltype(has_s_t)::value, decltype(full_t)::value, LIM, RW>(
                C, S, qxo, qyo, lqx, lqy, E, c0 > 0, W, c, nx, lane, s, s_half, T, k, k2, a.east_out, a.south_out,
                carH, carN, gr_row, gs_row, lh, lx, ly, gnr, &rwv);
        };
        if (interior && has_s)
            row(std::true_type{}, std::true_type{});
        else if (has_s)
            row(std::true_type{}, std::false_type{});
        else
            row(std::false_type{}, std::false_type{});
        kahan_add(gr_s, gr_c, gr_row);
        kahan_add(gs_s, gs_c, gs_row);
        if (act) {
            st_quad(lout + o, lh);
            st_quad(lout + plane + o, lx);
            st_quad(lout + 2 * plane + o, ly);
            if (gn) {
                const Quad g = ld_quad(gn + o);
                st_quad(gn + o, Quad{__fadd2_rn(g.a, gnr.a), __fadd2_rn(g.b, gnr.b)});
            }
        }
        C = S;
    }
    const int slot = blockIdx.z * ((a.nx + kSpan - 1) / kSpan) + span;
    adjoint_partials(a.gpart, RW ? a.gdpart : nullptr, a.nslot, m, slot, lane, Sum2{gr_s, -gr_c}, Sum2{gs_s, -gs_c},
                     Sum2{gd_s, -gd_c}, pl.rdt, a.rscale[m], pl.dt);
}

__global__ void reciprocals_kernel(const float* __restrict__ x, int n, double* __restrict__ out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = 1.0 / (double)x[i];
}

// Loss sensitivity at observation times: the state after step j is observed
// at sample s when sample_step[s][m] == j + 1; dL/dh += 2 (y - d) at the
// gauge cells.
__global__ void seed_kernel(const AdjArgs a, const int32_t* __restrict__ sample_step,
                            const float* __restrict__ y, const double* __restrict__ d,
                            const int32_t* __restrict__ cells, int ns, int G)
{
    pdl_launch();
    pdl_wait();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= a.M * G) return;
    const int m = t / G, g = t % G;
    const int j = a.seg_end[m] - 1 - a.rev_i;
    if (j < a.seg_first) return;
    float* lh = a.lam + ((size_t)a.lam_in * a.M + m) * 3 * a.plane;
    const int cell = cells[g];
    const size_t o = (size_t)(cell / a.nx) * a.ld + cell % a.nx;
    for (int s = 0; s < ns; ++s)
        if (sample_step[(size_t)s * a.M + m] == j + 1)
            lh[o] += (float)(2.0 * ((double)y[((size_t)s * a.M + m) * G + g] - d[(size_t)s * G + g]));
}

// Sum of the per-member Manning gradients in member order (deterministic).
__global__ void reduce_members_kernel(const float* __restrict__ gm, int M, int ny, int nx, int ld,
                                      size_t plane, float* __restrict__ out)
{
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (size_t)ny * nx) return;
    const size_t r = t / nx, c = t % nx;
    const size_t o = r * ld + c;
    float acc = 0.0f;
    for (int m = 0; m < M; ++m) acc += gm[(size_t)m * plane + o];
    out[t] = acc;
}

template <int LIM, bool RW>
void launch_adjoint_lim(const AdjArgs& a, int members_per_cta, cudaStream_t s)
{
    const int spans = (a.nx + kSpan - 1) / kSpan;
    const int strips = (a.ny + a.rows_per_strip - 1) / a.rows_per_strip;
    if (members_per_cta >= 4) {
        dim3 grid((a.M + 3) / 4, spans, strips), block(32, 4);
        launch_pdl(adjoint_kernel<4, 1, LIM, RW>, grid, block, 0, s, a);
    } else {
        dim3 grid(a.M, (spans + 3) / 4, strips), block(32, 4);
        launch_pdl(adjoint_kernel<1, 4, LIM, RW>, grid, block, 0, s, a);
    }
}

}  // namespace

void launch_adjoint(const AdjArgs& a, int members_per_cta, cudaStream_t s)
{
    if (a.rw)
        a.limiter ? launch_adjoint_lim<1, true>(a, members_per_cta, s)
                  : launch_adjoint_lim<0, true>(a, members_per_cta, s);
    else
        a.limiter ? launch_adjoint_lim<1, false>(a, members_per_cta, s)
                  : launch_adjoint_lim<0, false>(a, members_per_cta, s);
}

void launch_seed(const AdjArgs& a, const int32_t* sample_step, const float* y, const double* d,
                 const int32_t* cells, int ns, int G, cudaStream_t s)
{
    const int n = a.M * G;
    launch_pdl(seed_kernel, (n + 127) / 128, 128, 0, s, a, sample_step, y, d, cells, ns, G);
}

void launch_reciprocals(const float* x, int n, double* out, cudaStream_t s)
{
    reciprocals_kernel<<<(n + 127) / 128, 128, 0, s>>>(x, n, out);
}

void launch_reduce_members(const float* gm, int M, int ny, int nx, int ld, size_t plane, float* out,
                           cudaStream_t s)
{
    const size_t n = (size_t)ny * nx;
    reduce_members_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(gm, M, ny, nx, ld, plane, out);
}

}  // namespace flood
