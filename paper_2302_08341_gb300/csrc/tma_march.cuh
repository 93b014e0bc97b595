// The TMA-staged march of one warp over a 128-column span of rows
// [r0, r1) of one grid (an ensemble member or a batched scenario), shared by
// the ensemble (step_tma.cu) and batched (batch_kernel.cu) step kernels.
//
// The warp's rows arrive through a ring of kTmaNS shared-memory stages filled
// by the tensor memory accelerator: one 3-D tiled copy brings a row of h, qx
// and qy (136 columns: the span plus 4 halo columns each side, zero-filled
// past the grid's edges), another the same row of z and n.  Lane 0 keeps the
// ring's rows in flight ahead of the row being computed, so the memory
// latency is covered by the warp's own pipeline; the halo comes with the
// tile, so no scalar edge loads remain.  Every mbarrier wait is bounded: on
// timeout the march records FLOOD_ERR_TIMEOUT in the error word, waits
// (bounded) for its own copies in flight, and returns false.
//
// What bounds it: the issue slots, before memory.  A row of 128 cells took 545
// warp instructions, of which the arithmetic of its 256 links and 128 depths
// is about 290; the rest was bookkeeping, edge tests and the link west of the
// span, which lane 0 computed in a branch of its own.  So links are computed
// in pairs with the two-wide FP32 instructions (link2_q); the link west of
// the span is computed by every lane from one broadcast address, in line with
// the others; cells past the grid's edge are masked in a branch that only the
// spans holding the edge take (the edge spans ran both forms of every link);
// the row's four depths share one test for negative values; a row's depth,
// bed and roughness are read again from its stage rather than carried over,
// so the row loop needs no unrolling to stay free of moves; the row is
// compiled apart for spans without the grid's last column and for its last
// row: 350 instructions a row.  2000 x 2000 cells x 96 members: 1.63 -> 1.39 ms
// per step, where memory binds (7.2 TB/s at 26 bytes a cell, of which some 23
// reach DRAM); 1000 x 1000 x 16: 105 -> 79 us.
// Two spans a warp (one wait and one link west for 256 cells, 12 warps per SM
// instead of 20) measured the same or slower at every size but one.
#pragma once

#include <type_traits>

#include "march.cuh"
#include "quad.cuh"
#include "tma.cuh"

namespace flood {

constexpr int kTmaSpan = 128;
constexpr int kTmaNS = 4;                          // stages per warp
constexpr int kTmaBox = kTmaSpan + 8;              // columns per tile row
constexpr int kTmaStaticOff = 1664;                // bytes: z, n after h, qx, qy (128-aligned)
constexpr int kTmaStageBytes = 2816;               // 128-aligned stage size
constexpr uint32_t kTmaTx = kTmaBox * 3 * 4 + kTmaBox * 2 * 4;  // bytes landing per stage
constexpr long long kTmaWaitBudget = kTmaWaitBudgetDefault;  // clock cycles before giving up
constexpr int kTmaHmOff = kTmaStageBytes;          // running maxima: 128 floats after z, n
static_assert((kTmaNS & (kTmaNS - 1)) == 0, "ring index arithmetic needs a power of two");

// With land cover the static planes are the bed and each cell's class code (a
// uint32 where the roughness would be): the stage keeps its size.
__host__ __device__ constexpr int tma_stage_bytes(bool track) { return kTmaStageBytes + (track ? 512 : 0); }

// Dynamic shared memory of a CTA of `warps` warps: barriers and the land-cover
// class tables (64 bytes a warp), then each warp's stages.
__host__ __device__ constexpr int tma_head_bytes(int warps)
{
    return 128 * ((8 * kTmaNS * warps + 127) / 128) + 128 * ((64 * warps + 127) / 128);
}
__host__ __device__ constexpr size_t tma_march_smem_bytes(int warps, bool track = false)
{
    return 128 + tma_head_bytes(warps) + (size_t)kTmaNS * tma_stage_bytes(track) * warps;
}

// This warp's share of the CTA's dynamic shared memory.
struct TmaSmem {
    uint32_t bar0;            // barriers, 8 bytes each
    float4* tab;              // [4] class table: rain depth, drainage depth, Manning n
    unsigned char* stages;
};

__device__ __forceinline__ TmaSmem tma_march_smem(unsigned char* smem_raw, int warps, int w,
                                                  bool track = false)
{
    unsigned char* base = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~static_cast<uintptr_t>(127));
    TmaSmem m;
    m.bar0 = smem_u32(base) + 8u * kTmaNS * w;
    m.tab = reinterpret_cast<float4*>(base + 128 * ((8 * kTmaNS * warps + 127) / 128)) + 4 * w;
    m.stages = base + tma_head_bytes(warps) + kTmaNS * tma_stage_bytes(track) * w;
    return m;
}

// state_map: (ld, ny, planes) with the source h, qx, qy at planes
// [plane0, plane0 + 3); static_map: (ld, ny, 2) with z then n.  Writes the
// new state to dst (and ck when non-null); TRACK_MAX: also raises the
// running maximum depth at hm, whose old values arrive with each row through
// hm_map (member plane hm_plane, 128 columns from c0); LC: land cover
// (roughness by class from lk, the class's share of the rain and its
// drainage; static_map then holds the bed and each cell's class code, so the
// codes arrive with the row where the roughness would, halo included; the
// class table sits in shared memory, one word of it per lookup).  Each is a
// separate instantiation, so the plain step carries no trace of them.
// Returns false if a wait gave up.  WAIT_HOOK: each row wait may take
// wait_budget clock cycles instead of kTmaWaitBudget (a failure-detection
// hook; the copies still in flight are always drained with the full
// kTmaWaitBudget).
template <bool TRACK_MAX, bool LC, int LIM, bool WAIT_HOOK = false>
__device__ __forceinline__ bool tma_march(const CUtensorMap* state_map, const CUtensorMap* static_map,
                                          int plane0, const TmaSmem& sm,
                                          float* __restrict__ dst, float* ck, float* hm, int* err,
                                          size_t plane,
                                          int ny, int nx, int ld, int c0, int r0, int r1, int lane,
                                          const FaceK& k, float dt_dx, float s, float dr,
                                          int east_out, int south_out, MarchOut& out,
                                          const LandK* lk = nullptr,
                                          long long wait_budget = kTmaWaitBudget,
                                          const CUtensorMap* hm_map = nullptr, int hm_plane = 0)
{
    constexpr int kNS = kTmaNS;
    constexpr int kStage = tma_stage_bytes(TRACK_MAX);
    constexpr uint32_t kTx = kTmaTx + (TRACK_MAX ? 512u : 0u);
    constexpr int kZ = kTmaStaticOff / 4;
    constexpr int kN = kZ + kTmaBox;
    constexpr int kQx = kTmaBox, kQy = 2 * kTmaBox;
    const uint32_t stage0 = smem_u32(sm.stages);
    const float s_half = 0.5f * s;
    const Link2K lk2 = link2_k(k, s_half);
    const float2 lim2 = dup2(k.dx_4dt), dtdx2 = dup2(dt_dx), dr2 = dup2(dr);

    const int c = c0 + 4 * lane;
    const bool full = c0 + kTmaSpan < nx;  // every cell and its east neighbour inside
    const int ra = r0 > 0 ? r0 - 1 : r0;   // first row loaded
    const int rb = min(r1 + 1, ny);        // one past the last row loaded

    if (LC && lane < 4) sm.tab[lane] = make_float4(lk->dr, lk->dd, lk->n, 0.0f);
    if (lane == 0) {
        for (int i = 0; i < kNS; ++i) mbar_init(sm.bar0 + 8u * i, 1);
        fence_mbar_init();
    }
    __syncwarp();
    auto issue = [&](int row, int slot) {
        const uint32_t bar = sm.bar0 + 8u * slot;
        mbar_arrive_expect_tx(bar, kTx);
        const uint32_t d = stage0 + kStage * slot;
        tma_load_3d(d, state_map, c0 - 4, row, plane0, bar);
        tma_load_3d(d + kTmaStaticOff, static_map, c0 - 4, row, 0, bar);
        if (TRACK_MAX) tma_load_3d(d + kTmaHmOff, hm_map, c0, row, hm_plane, bar);
    };
    if (lane == 0)
        for (int i = 0; i < kNS && ra + i < rb; ++i) issue(ra + i, i);
    auto wait_slot = [&](int slot, uint32_t parity, long long budget) -> bool {
        return mbar_wait_bounded(sm.bar0 + 8u * slot, parity, budget);
    };
    const long long budget = WAIT_HOOK ? wait_budget : kTmaWaitBudget;
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
        if (lane == 0) atomicOr(err, 2);
        for (int row = from; row < to; ++row)
            wait_slot((row - ra) % kNS, ((row - ra) / kNS) & 1, kTmaWaitBudget);
    };
    auto row_ptr = [&](int slot) -> const float* {
        return reinterpret_cast<const float*>(sm.stages + kStage * slot);
    };
    // Manning n of the class of a staged cell (LC)
    auto class_n = [&](const float* code) -> float {
        return reinterpret_cast<const float*>(sm.tab + *reinterpret_cast<const uint32_t*>(code))[2];
    };
    auto quad_n = [&](const float* p) -> Quad {  // roughness of four staged cells
        if (!LC) return ld_quad(p);
        const uint4 q = *reinterpret_cast<const uint4*>(p);
        const float* t = reinterpret_cast<const float*>(sm.tab) + 2;
        return Quad{make_float2(t[4 * q.x], t[4 * q.y]), make_float2(t[4 * q.z], t[4 * q.w])};
    };
    // links of four cells with the four south of them (or the row above with this one)
    auto south_links = [&](const Quad& h1, const Quad& z1, const Quad& n1, const Quad& u1, const Quad& h2,
                           const Quad& z2, const Quad& n2, const Quad& u2, const Quad& q) -> Quad {
        return Quad{link2_q<LIM>(h1.a, z1.a, h2.a, z2.a, q.a, __fadd2_rn(n1.a, n2.a), u1.a, u2.a, lk2),
                    link2_q<LIM>(h1.b, z1.b, h2.b, z2.b, q.b, __fadd2_rn(n1.b, n2.b), u1.b, u2.b, lk2)};
    };
    auto bounds = [&](const Quad& h) -> Quad {  // the limiter's bounds of four cells
        return Quad{__fmul2_rn(h.a, lim2), __fmul2_rn(h.b, lim2)};
    };

    const int x0 = 4 + 4 * lane;  // this lane's first cell in a tile row
    int sC = 0;                   // slot of row r, of row r + 1 and that row's phase
    if (r0 > 0) {
        if (!wait_slot(0, 0, budget)) {
            drain_and_fail(ra, min(rb, ra + kNS));
            return false;
        }
        sC = 1;
    }
    if (!wait_slot(sC, 0, budget)) {
        drain_and_fail(r0, min(rb, ra + kNS));
        return false;
    }
    const float* F = row_ptr(sC) + x0;
    Quad nC = quad_n(F + kN);
    Quad qN = quad_of(0.0f);
    if (r0 > 0) {
        const float* U = row_ptr(0) + x0;
        const Quad hU = ld_quad(U), hF = ld_quad(F);
        qN = south_links(hU, ld_quad(U + kZ), quad_n(U + kN), bounds(hU), hF, ld_quad(F + kZ), nC,
                         bounds(hF), ld_quad(U + kQy));
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (!full && c + j >= nx) quad_at(qN, j) = 0.0f;
        release(ra, 0);
    }

    float hmax = 0.0f;
    float out_s = 0.0f, out_c = 0.0f, clamp = 0.0f, drn_s = 0.0f, drn_c = 0.0f;
    int sN = sC + 1;
    uint32_t phN = 0;
    float* pd = dst + (size_t)r0 * ld + c;
    float* pc = ck ? ck + (size_t)r0 * ld + c : nullptr;
    float* ph = TRACK_MAX ? hm + (size_t)r0 * ld + c : nullptr;

    // One row.  HAS_S: not the grid's last row; FULL: a span without the grid's
    // last column.  False if the wait for the row below gave up.
    auto row = [&](int r, auto has_s_t, auto full_t) -> bool {
        constexpr bool has_s = decltype(has_s_t)::value, full = decltype(full_t)::value;
        if (has_s && !wait_slot(sN, phN, budget)) {
            drain_and_fail(r + 1, min(rb, r + kNS));
            return false;
        }
        const float* R = row_ptr(sC);
        const float* P = R + x0;
        const Quad hC = ld_quad(P), zC = ld_quad(P + kZ);
        if (!LC) nC = ld_quad(P + kN);
        // east links: cells 0 1 2 3 with 1 2 3 and the next lane's first,
        // straight from the tile
        const Quad qx = ld_quad(P + kQx), qy = ld_quad(P + kQy);
        const float hE = P[4], zE = P[kZ + 4], nE = LC ? class_n(P + kN + 4) : P[kN + 4];
        // the link west of the span, from the tile's halo: every lane computes
        // it from lane 0's addresses, lane 0 keeps it
        float hW = 0.0f, zW = 0.0f, nW = 0.0f, qWo = 0.0f;
        if (c0 > 0) {
            hW = R[3];
            zW = R[kZ + 3];
            nW = LC ? class_n(R + kN + 3) : R[kN + 3];
            qWo = R[kQx + 3];
        }
        uint4 codes;
        if (LC) codes = *reinterpret_cast<const uint4*>(P + kN);
        Quad hmo;
        if (TRACK_MAX) hmo = ld_quad(R + kTmaHmOff / 4 + 4 * lane);
        // with tracked maxima (16 warps an SM and registers to spare) the row
        // goes into registers whole and its stage takes a later row before the
        // arithmetic: over twenty sizes 0.1 to 2.4 % less a step (us: 777 x 1013 x
        // 12 60.3 -> 59.6, 1200 x 1310 x 32 259.1 -> 253.0, 2000 x 2000 x 24 480.5
        // -> 480.1; with land cover 1000 x 1000 x 24 136.3 -> 133.2, 1500 x 1500 x
        // 40 441.3 -> 432.0); with 20 warps that costs more than it hides (1000 x
        // 1000 x 16, 68 steps: 5.76 -> 6.22 ms)
        if (TRACK_MAX) release(r, sC);
        const Quad uC = bounds(hC);
        Quad qE, qS, nS;
        qE.a = link2_q<LIM>(hC.a, zC.a, make_float2(hC.a.y, hC.b.x), make_float2(zC.a.y, zC.b.x), qx.a,
                            make_float2(__fadd_rn(nC.a.x, nC.a.y), __fadd_rn(nC.a.y, nC.b.x)), uC.a,
                            make_float2(uC.a.y, uC.b.x), lk2);
        qE.b = link2_q<LIM>(hC.b, zC.b, make_float2(hC.b.y, hE), make_float2(zC.b.y, zE), qx.b,
                            make_float2(__fadd_rn(nC.b.x, nC.b.y), __fadd_rn(nC.b.y, nE)), uC.b,
                            make_float2(uC.b.y, __fmul_rn(hE, k.dx_4dt)), lk2);
        float qH = (r >= k.in_r0 && r < k.in_r1) ? k.q_in : 0.0f;  // west edge: wall or inflow
        if (c0 > 0)
            qH = link_q<LIM>(hW, zW, hC.a.x, zC.a.x, qWo, __fmul_rn(s_half, __fadd_rn(nW, nC.a.x)), k);
        if (has_s) {
            const float* Q = row_ptr(sN) + x0;
            const Quad hS = ld_quad(Q);
            nS = quad_n(Q + kN);
            qS = south_links(hC, zC, nC, uC, hS, ld_quad(Q + kZ), nS, bounds(hS), qy);
        } else {
            nS = nC;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                quad_at(qS, j) =
                    south_out ? outflow_q<LIM>(quad_at(hC, j), quad_at(qy, j), __fmul_rn(s, quad_at(nC, j)), k)
                              : 0.0f;
        }
        if (!full) {  // the span holds the grid's last column: its east link, and nothing past it
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int cj = c + j;
                if (cj >= nx - 1) {
                    quad_at(qE, j) =
                        (east_out && cj == nx - 1)
                            ? outflow_q<LIM>(quad_at(hC, j), quad_at(qx, j), __fmul_rn(s, quad_at(nC, j)), k)
                            : 0.0f;
                    if (cj >= nx) quad_at(qS, j) = 0.0f;
                }
            }
        }
        // west links: the east links of the cells before, the first from the lane before
        float qW0 = __shfl_up_sync(0xffffffffu, qE.b.y, 1);
        if (lane == 0) qW0 = qH;
        const float2 wa = make_float2(__fsub_rn(qW0, qE.a.x), __fsub_rn(qE.a.x, qE.a.y));
        const float2 wb = make_float2(__fsub_rn(qE.a.y, qE.b.x), __fsub_rn(qE.b.x, qE.b.y));
        const float2 na = __fadd2_rn(wa, sub2(qN.a, qS.a, lk2.m1));
        const float2 nb = __fadd2_rn(wb, sub2(qN.b, qS.b, lk2.m1));
        // the step's increment (fluxes and rain) is formed first and added
        // to the depth once: adding the same rain depth to every cell on its
        // own rounds every cell of a binade the same way, a bias that builds
        // up in the stored volume
        Quad hN;
        if (!LC) {
            hN.a = __fadd2_rn(hC.a, __ffma2_rn(dtdx2, na, dr2));
            hN.b = __fadd2_rn(hC.b, __ffma2_rn(dtdx2, nb, dr2));
            if (!full) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (c + j >= nx) quad_at(hN, j) = 0.0f;
            }
        } else {
            const uint32_t code[4] = {codes.x, codes.y, codes.z, codes.w};
            const float net[4] = {na.x, na.y, nb.x, nb.y};
            float row_sink = 0.0f;  // the row's drained depth, compensated once per row
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float2 sd = *reinterpret_cast<const float2*>(sm.tab + code[j]);
                const bool in = full || c + j < nx;
                const float hp = in ? __fadd_rn(quad_at(hC, j), __fmaf_rn(dt_dx, net[j], sd.x)) : 0.0f;
                const float sink = fminf(sd.y, fmaxf(hp, 0.0f));
                // drainage that took all the water present leaves a depth
                // that does not depend on the one before: marked like a
                // clamped cell
                quad_at(hN, j) = (hp > 0.0f && sink == hp) ? -0.0f : __fsub_rn(hp, sink);
                row_sink = __fadd_rn(row_sink, sink);
            }
            kahan_add(drn_s, drn_c, row_sink);
        }
        // wet/dry clamp: a negative depth is rare (the limiter leaves only
        // rounding), so the four cells share one test.  Clamped cells keep a
        // negative zero: the adjoint reads the sign bit to know the branch
        if (fminf(fmin3(hN.a.x, hN.a.y, hN.b.x), hN.b.y) < 0.0f) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (quad_at(hN, j) < 0.0f) {
                    clamp = __fsub_rn(clamp, quad_at(hN, j));
                    quad_at(hN, j) = -0.0f;
                }
        }
        // a NaN anywhere stays in the maximum
        hmax = fmax3_nan(fmax3_nan(hmax, hN.a.x, hN.a.y), hN.b.x, hN.b.y);
        if ((!full && east_out) || (!has_s && south_out)) {  // the same for the whole warp
            // links leaving the domain this row: the east edge link (one lane)
            // and, on the last row, the south edge links
            float ev = 0.0f;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (c + j == nx - 1 && east_out) ev = quad_at(qE, j);
            if (!has_s && south_out)
                ev = __fadd_rn(ev, __fadd_rn(__fadd_rn(qS.a.x, qS.a.y), __fadd_rn(qS.b.x, qS.b.y)));
            kahan_add(out_s, out_c, ev);
        }
        if (full || c < nx) {
            st_quad(pd, hN);
            st_quad(pd + plane, qE);
            st_quad(pd + 2 * plane, qS);
            if (ck) {
                st_quad(pc, hN);
                st_quad(pc + plane, qE);
                st_quad(pc + 2 * plane, qS);
            }
            if (TRACK_MAX) {
                *reinterpret_cast<float4*>(ph) = make_float4(fmaxf(hmo.a.x, hN.a.x), fmaxf(hmo.a.y, hN.a.y),
                                                             fmaxf(hmo.b.x, hN.b.x), fmaxf(hmo.b.y, hN.b.y));
            }
        }
        pd += ld;
        if (ck) pc += ld;
        if (TRACK_MAX) ph += ld;
        // march: this row's south links are the next row's north links
        qN = qS;
        if (LC) nC = nS;
        if (!TRACK_MAX) release(r, sC);
        sC = sN;
        sN = (sN + 1) & (kNS - 1);
        if (sN == 0) phN ^= 1u;
        return true;
    };
    const int rS = min(r1, ny - 1);  // rows with a row below them
    int r = r0;
    if (full) {
#pragma unroll 1
        for (; r < rS; ++r)
            if (!row(r, std::true_type{}, std::true_type{})) return false;
    } else {
#pragma unroll 1
        for (; r < rS; ++r)
            if (!row(r, std::true_type{}, std::false_type{})) return false;
    }
    if (r < r1) row(r, std::false_type{}, std::false_type{});

    out.hmax = hmax;
    out.bad = !(hmax <= 3.0e38f);  // a NaN or an overflow anywhere
    out.out = Sum2{out_s, -out_c};
    out.clamp = clamp;
    out.drn = Sum2{drn_s, -drn_c};
    return true;
}

}  // namespace flood
