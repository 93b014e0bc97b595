// TMA-staged reverse stencil (same arithmetic and results, bit for bit, as
// adjoint_kernel.cu, through the shared row code of adjoint_row.cuh).
//
// The direct-load adjoint kernel needs about 128 registers per thread, so
// only four CTAs of four warps fit on an SM and its loads cannot keep enough
// bytes in flight.  Here each warp streams its rows through a ring of
// shared-memory stages filled by the tensor memory accelerator, one row of all
// ten planes it reads per stage: the state before the step (h, qx, qy), the
// depth after it, the sensitivities lambda (h, qx, qy), the bed and roughness
// (with land cover the bed and the class codes), and the member's Manning
// gradient, each 136 columns wide (the warp's 128 plus a 4-column halo on each
// side).  Lane 0 keeps kNS - 1 rows in flight ahead of the row being computed.
// Every mbarrier wait is bounded: on timeout the kernel records
// FLOOD_ERR_TIMEOUT, waits (bounded) for its own copies in flight, and
// returns.  Bound by issue slots at 12 warps per SM (what the stages and 160
// registers leave room for); with the row arithmetic in pairs the reverse and
// replay of a step of 1000 x 1000 x 24 went from 412 to 376 us, and short
// strips run faster than with direct loads at every size measured but one
// 300 x 400 pair (24 against 23 us).
#include <type_traits>

#include "adjoint.cuh"
#include "adjoint_row.cuh"
#include "launch.cuh"
#include "tma.cuh"

namespace flood {

namespace {

constexpr int kSpan = 128;
constexpr int kNS = 3;                          // stages per warp
constexpr int kBox = kSpan + 8;                 // columns per tile row
// float offsets inside a stage (each part starts on a 128-byte boundary)
constexpr int kSt = 0;                          // h, qx, qy before the step: 3 x kBox
constexpr int kHa = 416;                        // depth after the step: kBox
constexpr int kLam = 576;                       // lambda h, qx, qy: 3 x kBox
constexpr int kZ = 992;                         // bed: kBox
constexpr int kN = kZ + kBox;                   // roughness: kBox
constexpr int kGn = 1280;                       // Manning gradient: kBox
constexpr int kStageBytes = 5760;
constexpr uint32_t kRowBytes = kBox * 4;
constexpr long long kWaitBudget = 200000000LL;  // clock cycles (~0.1 s) before giving up

static_assert(kHa * 4 >= 3 * kBox * 4 && kHa % 32 == 0, "stage layout");
static_assert(kLam * 4 >= (kHa + kBox) * 4 && kLam % 32 == 0, "stage layout");
static_assert(kZ * 4 >= (kLam + 3 * kBox) * 4 && kZ % 32 == 0, "stage layout");
static_assert(kGn * 4 >= (kN + kBox) * 4 && kGn % 32 == 0, "stage layout");
static_assert(kStageBytes >= (kGn + kBox) * 4 && kStageBytes % 128 == 0, "stage layout");
// Land cover: the roughness plane's place holds each cell's class code (a
// uint32), staged with the bed as in the forward step.

// Shared memory ahead of the stages: barriers, then the class tables of land
// cover (64 bytes a warp).
__host__ __device__ constexpr int head_bytes(int warps)
{
    return 128 * ((8 * kNS * warps + 127) / 128) + 128 * ((64 * warps + 127) / 128);
}

// LC: land cover: the roughness, runoff share and drainage flag of every cell
// from its class (the codes come with the staged rows, the member's class
// table lies in shared memory).
template <int WM, int LIM, bool LC = false>
__global__ void __launch_bounds__(32 * WM, WM == 4 ? 3 : 12) adjoint_tma_kernel(
    const __grid_constant__ AdjTmaArgs t)
{

    extern __shared__ unsigned char smem_raw[];
    const AdjArgs& a = t.a;
    const int lane = threadIdx.x;
    const int w = threadIdx.y;
    const int m = blockIdx.x * WM + w;
    const int span = blockIdx.y;
    const int c0 = span * kSpan;
    pdl_launch();
    pdl_wait();
    if (m >= a.M || c0 >= a.nx) return;  // whole warps; no block-wide barriers below

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
                for (int q = 0; q < 3; ++q) {
                    const size_t o = q * plane + (size_t)r * ld + c;
                    *reinterpret_cast<float4*>(lout + o) = *reinterpret_cast<const float4*>(lin + o);
                }
        return;
    }
    if (*reinterpret_cast<volatile const int*>(a.err) & 2) return;  // an earlier wait gave up

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
    float* __restrict__ gn = a.gn ? a.gn + (size_t)m * plane : nullptr;

    unsigned char* base = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~static_cast<uintptr_t>(127));
    const uint32_t bar0 = smem_u32(base) + 8u * kNS * w;
    float4* const tab = reinterpret_cast<float4*>(base + 128 * ((8 * kNS * WM + 127) / 128)) + 4 * w;
    unsigned char* my_stages = base + head_bytes(WM) + kNS * kStageBytes * w;
    const uint32_t stage0 = smem_u32(my_stages);

    const int slot = j - a.seg_first;                 // seg slot of the state before the step
    const int p_before = (slot * a.M + m) * 3;        // plane index in the seg map
    const int p_after = ((slot + 1) * a.M + m) * 3;   // depth plane after the step
    const int p_lam = (a.lam_in * a.M + m) * 3;
    const uint32_t tx = kRowBytes * (gn ? 10u : 9u);
    const int ra = r0 > 0 ? r0 - 1 : r0;   // first row loaded (north halo)
    const int rb = min(r1 + 1, ny);        // one past the last row loaded

    if (LC && lane < 4)
        tab[lane] = make_float4(a.lc_n[(size_t)m * 4 + lane], a.lc_runoff[lane], a.lc_drains[lane], 0.0f);
    if (lane == 0) {
        for (int i = 0; i < kNS; ++i) mbar_init(bar0 + 8u * i, 1);
        fence_mbar_init();
    }
    __syncwarp();
    auto issue = [&](int row, int slot) {
        const uint32_t bar = bar0 + 8u * slot;
        const uint32_t dsts = stage0 + kStageBytes * slot;
        mbar_arrive_expect_tx(bar, tx);
        tma_load_3d(dsts + 4 * kSt, &t.seg_map, c0 - 4, row, p_before, bar);
        tma_load_3d(dsts + 4 * kHa, &t.seg1_map, c0 - 4, row, p_after, bar);
        tma_load_3d(dsts + 4 * kLam, &t.lam_map, c0 - 4, row, p_lam, bar);
        tma_load_3d(dsts + 4 * kZ, &t.static_map, c0 - 4, row, 0, bar);
        if (gn) tma_load_3d(dsts + 4 * kGn, &t.gn_map, c0 - 4, row, m, bar);
    };
    if (lane == 0)
        for (int i = 0; i < kNS && ra + i < rb; ++i) issue(ra + i, i);
    auto wait_slot = [&](int slot, uint32_t parity) -> bool {
        return mbar_wait_bounded(bar0 + 8u * slot, parity, kWaitBudget);
    };
    auto row_ptr = [&](int slot) -> const float* {
        return reinterpret_cast<const float*>(my_stages + kStageBytes * slot);
    };
    // a row's stage takes the row kNS further on, once the whole warp has read it
    auto release = [&](int row, int slot) {
        __syncwarp();
        if (row + kNS < rb && lane == 0) {
            fence_proxy_async_smem();
            issue(row + kNS, slot);
        }
    };
    // rows [from, to) are still in flight: every copy lands before the warp
    // leaves (bounded each)
    auto drain_and_fail = [&](int from, int to) {
        if (lane == 0) atomicOr(a.err, 2);
        for (int row = from; row < to; ++row) wait_slot((row - ra) % kNS, ((row - ra) / kNS) & 1);
    };

    const int x0 = 4 + 4 * lane;  // this lane's first cell in a tile row
    // roughness of four staged cells, and of one (land cover: of their classes)
    auto n_quad = [&](const float* R) -> Quad {
        if (!LC) return ld_quad(R + kN);
        const uint4 q = *reinterpret_cast<const uint4*>(R + kN);
        return Quad{make_float2(tab[q.x].x, tab[q.y].x), make_float2(tab[q.z].x, tab[q.w].x)};
    };
    auto n_one = [&](const float* R) -> float { return LC ? tab[__float_as_uint(R[kN])].x : R[kN]; };
    // a staged row's values (R: at this lane's first cell)
    auto load_row = [&](const float* R) -> AdjRow {
        return AdjRow{ld_quad(R + kSt), ld_quad(R + kZ), n_quad(R), masked(ld_quad(R + kHa), ld_quad(R + kLam))};
    };
    const Link2K k2 = link2_k(k, s_half);
    int sC = 0;  // slot of row r, of row r + 1 and that row's phase
    if (r0 > 0) {
        if (!wait_slot(0, 0)) {
            drain_and_fail(ra, min(rb, ra + kNS));
            return;
        }
        sC = 1;
    }
    if (!wait_slot(sC, 0)) {
        drain_and_fail(r0, min(rb, ra + kNS));
        return;
    }
    AdjRow C = load_row(row_ptr(sC) + x0);
    Quad carH = quad_of(0.0f), carN = quad_of(0.0f);  // north link: mu*dh2, mu*dnl
    if (r0 > 0) {  // the strip's north links, recomputed
        const float* U = row_ptr(0) + x0;
        north_carry<LIM>(load_row(U), ld_quad(U + kSt + 2 * kBox), ld_quad(U + kLam + 2 * kBox), C, c, nx, k2, T, k,
                         carH, carN);
        release(ra, 0);
    }

    // FP32 compensated sums of the rows' partials (lambda~ for the rain
    // gradient, mu n dq'/dn for the scale gradient), widened to FP64 once per warp
    float gr_s = 0.0f, gr_c = 0.0f, gs_s = 0.0f, gs_c = 0.0f;
    float gd_s = 0.0f, gd_c = 0.0f;  // land cover: drainage partials
    int sN = sC + 1;                 // at most kNS - 1 here
    uint32_t phN = 0;
    size_t o = (size_t)r0 * ld + c;
    auto row = [&](int r, auto has_s_t, auto full_t) -> bool {
        constexpr bool has_s = decltype(has_s_t)::value, full = decltype(full_t)::value;
        if (has_s && !wait_slot(sN, phN)) {
            drain_and_fail(r + 1, min(rb, r + kNS));
            return false;
        }
        const float* R = row_ptr(sC);
        const float* P = R + x0;
        AdjRow S;
        if (has_s) S = load_row(row_ptr(sN) + x0);
        const Quad qxo = ld_quad(P + kSt + kBox), qyo = ld_quad(P + kSt + 2 * kBox);
        const Quad lqx = ld_quad(P + kLam + kBox), lqy = ld_quad(P + kLam + 2 * kBox);
        // east neighbour of the lane's last cell and the span's west
        // neighbour, straight from the tile's halo
        const AdjSide E{P[kSt + 4], P[kZ + 4], n_one(P + 4), masked(P[kHa + 4], P[kLam + 4]), 0.0f, 0.0f};
        const AdjSide W{R[kSt + 3], R[kZ + 3], n_one(R + 3), masked(R[kHa + 3], R[kLam + 3]), R[kSt + kBox + 3],
                        R[kLam + kBox + 3]};
        Quad lh, lx, ly, gnr, rwv;
        float gr_row, gs_row;
        if (LC) {
            float dfv[4];
            const uint4 q = *reinterpret_cast<const uint4*>(P + kN);
            const uint32_t code[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {  // the cells' runoff shares and drainage flags
                const float4 v = tab[code[j]];
                quad_at(rwv, j) = act ? v.y : 0.0f;
                dfv[j] = act ? v.z : 0.0f;
            }
            kahan_add(gd_s, gd_c, drain_row(C.l, ld_quad(P + kHa), dfv));
        }
        adjoint_row<has_s, full, LIM, LC>(C, S, qxo, qyo, lqx, lqy, E, c0 > 0, W, c, nx, lane, s, s_half, T, k, k2,
                                          a.east_out, a.south_out, carH, carN, gr_row, gs_row, lh, lx, ly, gnr, &rwv);
        kahan_add(gr_s, gr_c, gr_row);
        kahan_add(gs_s, gs_c, gs_row);
        if (full || act) {
            st_quad(lout + o, lh);
            st_quad(lout + plane + o, lx);
            st_quad(lout + 2 * plane + o, ly);
            if (gn) {
                const Quad g = ld_quad(P + kGn);
                st_quad(gn + o, Quad{__fadd2_rn(g.a, gnr.a), __fadd2_rn(g.b, gnr.b)});
            }
        }
        o += ld;
        if (has_s) C = S;
        release(r, sC);
        sC = sN;
        if (++sN == kNS) {
            sN = 0;
            phN ^= 1u;
        }
        return true;
    };
    const int rS = min(r1, ny - 1);  // rows with a row below them
    int r = r0;
    if (interior) {
#pragma unroll 1
        for (; r < rS; ++r)
            if (!row(r, std::true_type{}, std::true_type{})) return;
    } else {
#pragma unroll 1
        for (; r < rS; ++r)
            if (!row(r, std::true_type{}, std::false_type{})) return;
    }
    if (r < r1) row(r, std::false_type{}, std::false_type{});
    const int vslot = blockIdx.z * ((a.nx + kSpan - 1) / kSpan) + span;
    adjoint_partials(a.gpart, LC ? a.gdpart : nullptr, a.nslot, m, vslot, lane, Sum2{gr_s, -gr_c}, Sum2{gs_s, -gs_c},
                     Sum2{gd_s, -gd_c}, pl.rdt, a.rscale[m], pl.dt);
}

template <int WM>
size_t adj_smem_bytes()
{
    return 128 + head_bytes(WM) + (size_t)kNS * kStageBytes * WM;
}

template <int LIM, bool LC>
void launch_adjoint_tma_lim(const AdjTmaArgs& t, int members_per_cta, cudaStream_t s)
{
    const AdjArgs& a = t.a;
    const int spans = (a.nx + kSpan - 1) / kSpan;
    const int strips = (a.ny + a.rows_per_strip - 1) / a.rows_per_strip;
    if (members_per_cta >= 4 && a.M >= 4) {
        static bool attr = false;
        const size_t shm = adj_smem_bytes<4>();
        if (!attr) {
            cudaFuncSetAttribute(adjoint_tma_kernel<4, LIM, LC>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm);
            attr = true;
        }
        dim3 grid((a.M + 3) / 4, spans, strips), block(32, 4);
        launch_pdl(adjoint_tma_kernel<4, LIM, LC>, grid, block, shm, s, t);
    } else {
        const size_t shm = adj_smem_bytes<1>();
        dim3 grid(a.M, spans, strips), block(32, 1);
        launch_pdl(adjoint_tma_kernel<1, LIM, LC>, grid, block, shm, s, t);
    }
}

}  // namespace

void launch_adjoint_tma(const AdjTmaArgs& t, int members_per_cta, cudaStream_t s)
{
    if (t.a.lc_n)
        t.a.limiter ? launch_adjoint_tma_lim<1, true>(t, members_per_cta, s)
                    : launch_adjoint_tma_lim<0, true>(t, members_per_cta, s);
    else
        t.a.limiter ? launch_adjoint_tma_lim<1, false>(t, members_per_cta, s)
                    : launch_adjoint_tma_lim<0, false>(t, members_per_cta, s);
}

int adjoint_tma_box_cols() { return kBox; }

}  // namespace flood
