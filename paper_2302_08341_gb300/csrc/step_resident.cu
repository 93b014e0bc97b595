// Many steps in one launch for ensembles that fit on the chip.
//
// Where a member's state fits in shared memory, reading and writing it through
// L2 every step and launching two kernels per step costs more than the step:
// a 256 x 256 model took 10.6 us per step, of which its arithmetic is well
// under one.  Here one cooperative launch runs up to 240 steps.  Every member
// is cut into bands of whole rows, one CTA each, which keep h, qx, qy, the bed
// and the roughness in shared memory from the first step to the last; a step
// exchanges a row of depths with the bands above and below and the bands'
// maximum depths with all of the member's bands (Eq. 4).  Members never wait
// for one another.
//
// A step of a band:
//   1. links: east links of its rows, south links of its rows and of the row
//      above (which both bands compute, each from its own copy of that row's
//      old flux and with the same rounding, so the copies stay equal);
//   2. depths, and the first and last row's into the exchange rows, every
//      value in a 64-bit word with the step's number;
//   3. the band publishes its maximum, with the step's number in the same
//      word, and waits for the member's other words: the barrier and the
//      reduction in one round trip through L2, without a fence (a release
//      waits for all of an SM's stores; with flags and fences a step took
//      8.5 us whatever its size).  The other warps fetch the neighbours' rows
//      meanwhile, and warp 0 plans the next step.
// Exchange rows and words are kept twice, by the step's parity: a band can
// write step j + 2's only after every band has published step j + 1, hence
// read step j's.  Step numbers go on from launch to launch, so no word has to
// be cleared.  Waits are bounded: one that gives up records FLOOD_ERR_TIMEOUT
// and the band leaves; the others' waits then give up in turn.
//
// The links and depths are those of the march, operation by operation, so
// the results are the same bit for bit.
#include <algorithm>

#include "grid.cuh"
#include "launch.cuh"
#include "march.cuh"
#include "quad.cuh"
#include "resident.cuh"
#include "sum2.cuh"

namespace flood {

namespace {

constexpr int kThreads = 512;
// Clock cycles a band may wait for another (about 2 s; a step takes
// microseconds).  The launch is cooperative, so no band starts before all have
// their places: a kernel of another stream that held an SM's shared memory for
// 3 s held the launch up for as long, and no wait ran out.
constexpr long long kBandWaitBudget = 4000000000LL;
constexpr int kWarps = kThreads / 32;
constexpr int kWords = 5;      // 152 bands: a member's most

__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_relaxed_u64(unsigned long long* p, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
// Quad depths of an exchange row, each in a 64-bit word with the step's number
// above it: a word that carries the number it waits for is the value itself,
// so no fence orders the row before a flag.
__device__ __forceinline__ void st_tagged(unsigned long long* p, float4 v, uint32_t tag)
{
    const unsigned long long t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(t | __float_as_uint(v.x)),
                 "l"(t | __float_as_uint(v.y)) : "memory");
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p + 2), "l"(t | __float_as_uint(v.z)),
                 "l"(t | __float_as_uint(v.w)) : "memory");
}
__device__ __forceinline__ bool ld_tagged(const unsigned long long* p, float4& v, uint32_t tag)
{
    unsigned long long w[4];
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(w[0]), "=l"(w[1]) : "l"(p) : "memory");
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(w[2]), "=l"(w[3]) : "l"(p + 2) : "memory");
    v = make_float4(__uint_as_float((uint32_t)w[0]), __uint_as_float((uint32_t)w[1]),
                    __uint_as_float((uint32_t)w[2]), __uint_as_float((uint32_t)w[3]));
    return (uint32_t)(w[0] >> 32) == tag && (uint32_t)(w[1] >> 32) == tag && (uint32_t)(w[2] >> 32) == tag &&
           (uint32_t)(w[3] >> 32) == tag;
}

// A step's constants, from warp 0 to the band.
struct BandPlan {
    FaceK k;
    float dt_dx, dr;
    float2 dt;                // the step length in two words
    int active, fail, ckpt;
};

// (row, quad) of a thread's items, kThreads apart, without a division each
struct Item {
    int r, q;
    __device__ __forceinline__ Item(int i, int nq) : r(i / nq), q(i % nq) {}
    __device__ __forceinline__ void next(int dr, int dq, int nq)
    {
        r += dr;
        q += dq;
        if (q >= nq) {
            q -= nq;
            ++r;
        }
    }
};

template <bool TRACK, bool LC, int LIM>
__global__ void __launch_bounds__(kThreads, 1) step_resident_kernel(const __grid_constant__ ResidentArgs t)
{
    extern __shared__ __align__(16) float sm[];
    __shared__ BandPlan bp;
    __shared__ unsigned s_max[kWarps];
    __shared__ float2 s_src[4];   // land cover: rain and drainage depth of a class this step
    __shared__ float2 s_red[3][kWarps];
    const StepArgs& a = t.a;
    if (*reinterpret_cast<volatile const int*>(a.err) & 2) return;  // an earlier wait gave up
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m = blockIdx.x / t.bands, band = blockIdx.x % t.bands;
    const int ny = a.ny, nx = a.nx, ld = a.ld;
    const int b0 = band * t.rows, b1 = min(b0 + t.rows, ny), R = b1 - b0;
    const int nq = (nx + 3) / 4, P = 4 * nq + 4;
    const int dr_i = kThreads / nq, dq_i = kThreads % nq;
    // rows -1..R of h, z, n; rows 0..R-1 of qx; rows -1..R-1 of qy
    float* const H = sm + P;
    float* const Z = H + (size_t)P * (R + 2);
    float* const N = Z + (size_t)P * (R + 2);
    float* const QE = N + (size_t)P * (R + 1);
    float* const QS = QE + (size_t)P * (R + 1);
    float* const HM = QS + (size_t)P * R;              // running maxima (TRACK)
    uint32_t* const CL = reinterpret_cast<uint32_t*>(HM + (TRACK ? (size_t)P * R : 0));  // classes, four a word (LC)
    const MemberClock in = a.ms_in[m];
    const size_t mstride = 3 * a.plane;
    float* const st = a.state + (size_t)(in.cur * a.M + m) * mstride;

    for (int i = tid; i < P * (5 * R + 7); i += kThreads) sm[i] = 0.0f;
    __syncthreads();
    for (Item e(tid, nq); e.r < R + 2; e.next(dr_i, dq_i, nq)) {
        const int r = e.r - 1, g = b0 + r, c = 4 * e.q;
        if (g < 0 || g >= ny) continue;
        const size_t o = (size_t)g * ld + c;
        const int s = r * P + c;
        st_quad(H + s, ld_quad(st + o));
        st_quad(Z + s, ld_quad(a.z + o));
        if (LC) {
            const uint32_t w = cls_word(a.cls, o);
            const float* tn = a.lc_n + (size_t)m * 4;
            *reinterpret_cast<float4*>(N + s) = make_float4(tn[w & 3], tn[(w >> 8) & 3], tn[(w >> 16) & 3],
                                                            tn[(w >> 24) & 3]);
            if (r >= 0 && r < R) CL[r * nq + e.q] = w;
        } else {
            st_quad(N + s, ld_quad(a.n + o));
        }
        if (r < R) st_quad(QS + s, ld_quad(st + 2 * a.plane + o));
        if (r >= 0 && r < R) {
            st_quad(QE + s, ld_quad(st + a.plane + o));
            if (TRACK) st_quad(HM + s, ld_quad(a.hmax_field + (size_t)m * a.plane + o));
        }
    }

    // the member's clock and step plan, carried by warp 0 (every lane the same).
    // An FP64 operation takes some 60 cycles, a division about 900, and the plan
    // sits between two steps: what depends on the clock alone (the rain block
    // and its edge) is kept until the clock reaches the edge, the step length's
    // constants until it changes; the capped step is planned while the other
    // bands' maxima are awaited, and Eq. 4's root and division follow only
    // where they do not clearly give more than the cap
    double clk = in.t, rain_acc = 0.0, inflow_acc = 0.0;
    double stop = -1.0, rate = 0.0, rain_area = 0.0, inflow_area = 0.0, dt = 0.0, nxt = 0.0;
    bool lands = false;
    bool on_block = false;       // stop, rate and q_in belong to the clock
    float q_in = 0.0f;
    const float cap_h = a.cap_h;
    const bool floor_capped = a.h_floor < (double)cap_h;
    int64_t steps = in.steps;
    uint32_t hmax = in.hmax_bits;
    const float rain_mult = a.rain_mult[m], scale = a.scale[m], s_half = 0.5f * scale;
    const uint32_t seq0 = t.seq[m];
    if (tid == 0 && band == 0) {
        rain_acc = a.rain_acc[m];
        if (a.inflow) inflow_acc = a.inflow_acc[m];
    }
    MemberPlan mp{};             // the last plan
    mp.dt = -1.0;
    Sum2 vout, vclamp, vdrn;     // over all steps of the launch: two words each
    bool bad = false;
    unsigned long long* const words[2] = {t.words + (size_t)m * t.bands,
                                          t.words + ((size_t)a.M + m) * t.bands};
    // exchange rows: [parity][member][band][first, last][ld]
    auto xrow = [&](int parity, int b, int last) -> unsigned long long* {
        return t.xch + ((((size_t)parity * a.M + m) * t.bands + b) * 2 + last) * ld;
    };
    // warp 0: the plan of the step from clk with step length d (before landing)
    // into bp, as PlanQuad makes it
    auto set_plan = [&](double d) {
        bool fresh = false;  // the step's constants change
        if (!on_block) {
            const double blk = floor(__ddiv_rn(clk, a.rain_block));
            stop = __dmul_rn(blk + 1.0, a.rain_block);
            if (a.t_end >= 0.0 && a.t_end < stop) stop = a.t_end;
            const int b = (int)blk;
            rate = (blk >= 0.0 && b < a.nb) ? (double)a.hyeto[b] : 0.0;
            if (a.inflow) {
                const double Q = (blk >= 0.0 && b < a.inflow_blocks) ? (double)a.inflow[b] : 0.0;
                q_in = (float)(Q / (a.dxd * (double)(a.in_r1 - a.in_r0)));
            }
            fresh = on_block = true;
        }
        const bool active = !(a.t_end >= 0.0 && clk >= a.t_end);
        nxt = __dadd_rn(clk, d);
        lands = nxt >= stop;
        if (lands) {
            d = __dsub_rn(stop, clk);
            nxt = stop;
        }
        dt = d;
        if (fresh || dt != mp.dt) {
            if (dt != mp.dt) {  // three divisions, one a lane
                const double qv = (lane == 0 ? a.g * dt : lane == 1 ? a.dxd : dt) / (lane == 1 ? 4.0 * dt : a.dxd);
                const float qf = (float)qv;
                mp.gdt_dx = __shfl_sync(0xffffffffu, qf, 0);
                mp.dx_4dt = __shfl_sync(0xffffffffu, qf, 1);
                mp.dt_dx = __shfl_sync(0xffffffffu, qf, 2);
                mp.gdt = (float)(a.g * dt);
                mp.dt = dt;
            }
            mp.rdt = __dmul_rn(dt, rate);
            mp.dr = (float)__dmul_rn(mp.rdt, (double)rain_mult);
            rain_area = (double)mp.dr * a.cell_area;
            inflow_area = (double)q_in * a.dxd * (double)(a.in_r1 - a.in_r0);
            if (LC && lane < 4)
                s_src[lane] = make_float2(__fmul_rn(mp.dr, a.lc_runoff[lane]),
                                          __fmul_rn(__fmul_rn(a.lc_drain[m], a.lc_drains[lane]), (float)dt));
            if (lane == 0) {
                bp.k.gdt_dx = mp.gdt_dx;
                bp.k.gdt = mp.gdt;
                bp.k.dx_4dt = mp.dx_4dt;
                bp.k.q_in = q_in;
                bp.dt_dx = mp.dt_dx;
                bp.dr = mp.dr;
                bp.dt = make_float2((float)dt, (float)(dt - (double)(float)dt));
            }
        }
        mp.t_next = nxt;
        mp.active = active ? 1 : 0;
        mp.ckpt = -1;
        if (a.ckpt && active && (steps + 1) % a.ckpt_every == 0 && steps + 1 <= a.dt_log_cap)
            mp.ckpt = (int)((steps + 1) / a.ckpt_every);
        mp.q_in = active ? q_in : 0.0f;
        if (lane == 0) {
            bp.active = mp.active;
            bp.ckpt = mp.ckpt;
        }
    };
    auto capped_plan = [&]() { set_plan(a.dt_fixed > 0.0 ? a.dt_fixed : a.dt_cap); };
    // where the maximum depth does not leave the cap binding: Eq. 4
    auto settle_plan = [&]() {
        if (a.dt_fixed > 0.0 || (__uint_as_float(hmax) < cap_h && floor_capped)) return;
        double hm = (double)__uint_as_float(hmax);
        hm = hm > a.h_floor ? hm : a.h_floor;
        const double d = __ddiv_rn(a.alpha_dx, __dsqrt_rn(__dmul_rn(a.g, hm)));
        if (!(d > a.dt_cap)) set_plan(d);
    };
    // the planned step has been taken: clock, sums, log
    auto commit = [&]() {
        if (band == 0) {
            rain_acc += rain_area * a.ncell;
            if (a.inflow) inflow_acc += inflow_area * dt;
            if (a.log && lane == 0 && steps < a.dt_log_cap) a.log[(size_t)m * a.dt_log_cap + steps] = mp;
        }
        clk = nxt;
        ++steps;
        // half a step short of the edge the clock's quotient by the block is
        // safely below it; closer, the block is looked up anew
        on_block = !lands && __dadd_rn(nxt, 0.5 * dt) < stop;
    };

    if (warp == 0) {
        mp.cur = in.cur;
        if (lane == 0) {
            bp.k.h_eps = a.h_eps;
            bp.k.edge_drop = a.edge_drop;
            bp.k.limiter = a.limiter;
            bp.k.in_r0 = a.in_r0;
            bp.k.in_r1 = a.in_r1;
            bp.fail = 0;
        }
        capped_plan();
        settle_plan();
    }
    int j = 0;
    for (; j < t.n_steps; ++j) {
        const uint32_t want = seq0 + (uint32_t)j + 1u;
        __syncthreads();
        if (bp.fail || !bp.active) break;
        const FaceK k = bp.k;
        const Link2K k2 = link2_k(k, s_half);
        const float2 lim2 = dup2(k.dx_4dt);
        // 1. links: R rows of east links, then R + 1 rows of south links
        for (Item e(tid, nq); e.r < 2 * R + 1; e.next(dr_i, dq_i, nq)) {
            const int c = 4 * e.q;
            if (e.r < R) {
                const int s = e.r * P + c;
                const Quad h = ld_quad(H + s), z = ld_quad(Z + s), n = ld_quad(N + s), q = ld_quad(QE + s);
                const float hE = H[s + 4], zE = Z[s + 4], nE = N[s + 4];
                const float2 ua = __fmul2_rn(h.a, lim2), ub = __fmul2_rn(h.b, lim2);
                Quad v;
                v.a = link2_q<LIM>(h.a, z.a, make_float2(h.a.y, h.b.x), make_float2(z.a.y, z.b.x), q.a,
                                   make_float2(__fadd_rn(n.a.x, n.a.y), __fadd_rn(n.a.y, n.b.x)), ua,
                                   make_float2(ua.y, ub.x), k2);
                v.b = link2_q<LIM>(h.b, z.b, make_float2(h.b.y, hE), make_float2(z.b.y, zE), q.b,
                                   make_float2(__fadd_rn(n.b.x, n.b.y), __fadd_rn(n.b.y, nE)), ub,
                                   make_float2(ub.y, __fmul_rn(hE, k.dx_4dt)), k2);
                if (c + 4 >= nx) {  // the grid's last column: its outflow, and nothing past it
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (c + i >= nx - 1)
                            quad_at(v, i) = (a.east_out && c + i == nx - 1)
                                            ? outflow_q<LIM>(H[s + i], QE[s + i], __fmul_rn(scale, N[s + i]), k)
                                            : 0.0f;
                }
                st_quad(QE + s, v);
            } else {
                const int r = e.r - R - 1, g = b0 + r, s = r * P + c;
                if (g < 0) continue;  // north of the grid: a wall
                Quad v;
                if (g + 1 < ny) {
                    const Quad h = ld_quad(H + s), z = ld_quad(Z + s), n = ld_quad(N + s), q = ld_quad(QS + s);
                    const Quad hS = ld_quad(H + s + P), zS = ld_quad(Z + s + P), nS = ld_quad(N + s + P);
                    v.a = link2_q<LIM>(h.a, z.a, hS.a, zS.a, q.a, __fadd2_rn(n.a, nS.a), __fmul2_rn(h.a, lim2),
                                       __fmul2_rn(hS.a, lim2), k2);
                    v.b = link2_q<LIM>(h.b, z.b, hS.b, zS.b, q.b, __fadd2_rn(n.b, nS.b), __fmul2_rn(h.b, lim2),
                                       __fmul2_rn(hS.b, lim2), k2);
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        quad_at(v, i) = a.south_out
                                        ? outflow_q<LIM>(H[s + i], QS[s + i], __fmul_rn(scale, N[s + i]), k)
                                        : 0.0f;
                }
                if (c + 4 > nx) {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (c + i >= nx) quad_at(v, i) = 0.0f;
                }
                st_quad(QS + s, v);
            }
        }
        __syncthreads();
        // 2. depths
        const float2 dtdx2 = dup2(bp.dt_dx), dr2 = dup2(bp.dr);
        float hm = 0.0f;
        for (Item e(tid, nq); e.r < R; e.next(dr_i, dq_i, nq)) {
            const int r = e.r, g = b0 + r, c = 4 * e.q, s = r * P + c;
            const Quad h = ld_quad(H + s), qE = ld_quad(QE + s), qS = ld_quad(QS + s), qN = ld_quad(QS + s - P);
            const float qW = e.q > 0 ? QE[s - 1] : (g >= k.in_r0 && g < k.in_r1) ? k.q_in : 0.0f;
            const float2 na = __fadd2_rn(make_float2(__fsub_rn(qW, qE.a.x), __fsub_rn(qE.a.x, qE.a.y)),
                                         sub2(qN.a, qS.a, k2.m1));
            const float2 nb = __fadd2_rn(make_float2(__fsub_rn(qE.a.y, qE.b.x), __fsub_rn(qE.b.x, qE.b.y)),
                                         sub2(qN.b, qS.b, k2.m1));
            Quad v;
            if (!LC) {
                v.a = __fadd2_rn(h.a, __ffma2_rn(dtdx2, na, dr2));
                v.b = __fadd2_rn(h.b, __ffma2_rn(dtdx2, nb, dr2));
            } else {
                const uint32_t w = CL[r * nq + e.q];
                const float net[4] = {na.x, na.y, nb.x, nb.y}, hh[4] = {h.a.x, h.a.y, h.b.x, h.b.y};
                float row_sink = 0.0f;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float2 sd = s_src[(w >> (8 * i)) & 3];
                    const float hp = c + i < nx ? __fadd_rn(hh[i], __fmaf_rn(dtdx2.x, net[i], sd.x)) : 0.0f;
                    const float sink = fminf(sd.y, fmaxf(hp, 0.0f));
                    quad_at(v, i) = (hp > 0.0f && sink == hp) ? -0.0f : __fsub_rn(hp, sink);
                    row_sink = __fadd_rn(row_sink, sink);
                }
                vdrn.add(row_sink);
            }
            if (c + 4 > nx) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (c + i >= nx) quad_at(v, i) = 0.0f;
            }
            if (fminf(fmin3(v.a.x, v.a.y, v.b.x), v.b.y) < 0.0f) {  // wet/dry clamp (rare): keeps a negative zero
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (quad_at(v, i) < 0.0f) {
                        vclamp.add(-quad_at(v, i));
                        quad_at(v, i) = -0.0f;
                    }
            }
            hm = fmax3_nan(fmax3_nan(hm, v.a.x, v.a.y), v.b.x, v.b.y);
            if (a.east_out && c + 4 >= nx) {  // the grid's last column
                const float e4[4] = {qE.a.x, qE.a.y, qE.b.x, qE.b.y};
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (c + i == nx - 1) vout.add_product(e4[i], bp.dt);
            }
            if (a.south_out && g == ny - 1) {
                vout.add_product(qS.a.x, bp.dt);
                vout.add_product(qS.a.y, bp.dt);
                vout.add_product(qS.b.x, bp.dt);
                vout.add_product(qS.b.y, bp.dt);
            }
            st_quad(H + s, v);
            if (TRACK) {
                const Quad o = ld_quad(HM + s);
                *reinterpret_cast<float4*>(HM + s) = make_float4(fmaxf(o.a.x, v.a.x), fmaxf(o.a.y, v.a.y),
                                                                 fmaxf(o.b.x, v.b.x), fmaxf(o.b.y, v.b.y));
            }
            const float4 v4 = make_float4(v.a.x, v.a.y, v.b.x, v.b.y);
            if (r == 0 && b0 > 0) st_tagged(xrow(j & 1, band, 0) + c, v4, want);
            if (r == R - 1 && b1 < ny) st_tagged(xrow(j & 1, band, 1) + c, v4, want);
            if (bp.ckpt >= 0) {
                float* ck = a.ckpt + ((size_t)bp.ckpt * a.M + m) * mstride + (size_t)g * ld + c;
                st_quad(ck, v);
                st_quad(ck + a.plane, qE);
                st_quad(ck + 2 * a.plane, qS);
            }
        }
        const bool b_now = !(hm <= 3.0e38f);  // a NaN or an overflow
        bad |= b_now;
        const unsigned wm = __reduce_max_sync(0xffffffffu, b_now ? 0u : __float_as_uint(hm) & 0x7fffffffu);
        if (lane == 0) s_max[warp] = wm;
        __syncthreads();
        // 3. publish, wait for the member's other bands; the neighbours' rows
        bool ok = true;
        if (warp == 0) {
            unsigned hb = __reduce_max_sync(0xffffffffu, lane < kWarps ? s_max[lane] : 0u);
            if (lane == 0 && t.bands > 1)
                st_relaxed_u64(words[j & 1] + band, ((unsigned long long)want << 32) | hb);
            commit();
            if (j + 1 < t.n_steps) capped_plan();
            // a lane looks at up to kWords words at a time, all in flight at once
            for (int i0 = lane; t.bands > 1 && ok && i0 < t.bands; i0 += 32 * kWords) {
                const long long t0 = clock64();
                while (true) {
                    unsigned long long v[kWords];
#pragma unroll
                    for (int i = 0; i < kWords; ++i)
                        v[i] = ld_relaxed_u64(words[j & 1] + min(i0 + 32 * i, t.bands - 1));
                    bool all = true;
#pragma unroll
                    for (int i = 0; i < kWords; ++i) all &= (uint32_t)(v[i] >> 32) == want;
                    if (all) {
#pragma unroll
                        for (int i = 0; i < kWords; ++i) hb = max(hb, (unsigned)v[i]);
                        break;
                    }
                    if (clock64() - t0 > kBandWaitBudget) {
                        ok = false;
                        break;
                    }
                }
            }
            hmax = __reduce_max_sync(0xffffffffu, hb);
            if (j + 1 < t.n_steps) settle_plan();
        } else if (t.bands > 1 && j + 1 < t.n_steps) {
            for (int i = tid - 32; ok && i < 2 * nq; i += kThreads - 32) {
                const bool up = i < nq;
                if (up ? b0 == 0 : b1 == ny) continue;
                const int q = up ? i : i - nq;
                const unsigned long long* x = xrow(j & 1, up ? band - 1 : band + 1, up ? 1 : 0) + 4 * q;
                float4 v;
                const long long t0 = clock64();
                while (!ld_tagged(x, v, want))
                    if (clock64() - t0 > kBandWaitBudget) {
                        ok = false;
                        break;
                    }
                *reinterpret_cast<float4*>((up ? H - P : H + (size_t)R * P) + 4 * q) = v;
            }
        }
        if (!ok) {  // a wait ran out: the band leaves at the next step's start
            atomicOr(a.err, 2);
            bp.fail = 1;
        }
        // (the next step's plan is followed by a block barrier before anything is read)
    }
    __syncthreads();
    if (bad) atomicOr(a.err, 1);
    // the state back in place, the member's clock, the volume sums
    for (Item e(tid, nq); e.r < R; e.next(dr_i, dq_i, nq)) {
        const int s = e.r * P + 4 * e.q;
        const size_t o = (size_t)(b0 + e.r) * ld + 4 * e.q;
        st_quad(st + o, ld_quad(H + s));
        st_quad(st + a.plane + o, ld_quad(QE + s));
        st_quad(st + 2 * a.plane + o, ld_quad(QS + s));
        if (TRACK) st_quad(a.hmax_field + (size_t)m * a.plane + o, ld_quad(HM + s));
    }
    if (band == 0 && tid == 0) {
        MemberClock c;
        c.t = clk;
        c.steps = steps;
        c.hmax_bits = hmax;
        c.cur = in.cur;
        t.ms_end[m] = c;
        t.ms_next[m].hmax_bits = 0u;  // the slot the next step's maximum goes to
        a.rain_acc[m] = rain_acc;
        if (a.inflow) a.inflow_acc[m] = inflow_acc;
        t.seq[m] = seq0 + (uint32_t)t.n_steps + 1u;
    }
    if (LC) vdrn.warp_sum();
    vout.warp_sum();
    vclamp.warp_sum();
    if (lane == 0) {
        s_red[0][warp] = make_float2(vout.hi, vout.lo);
        s_red[1][warp] = make_float2(vclamp.hi, vclamp.lo);
        s_red[2][warp] = make_float2(vdrn.hi, vdrn.lo);
    }
    __syncthreads();
    if (tid < 3) {
        Sum2 sum;
        for (int w = 0; w < kWarps; ++w) sum.merge(s_red[tid][w].x, s_red[tid][w].y);
        const double v = sum.value();
        const size_t slot = (size_t)m * a.nslot + band;
        if (tid == 0 && v != 0.0) a.vacc[slot * 2] += v * a.dxd;
        if (tid == 1 && v != 0.0) a.vacc[slot * 2 + 1] += v * a.cell_area;
        if (tid == 2 && LC && v != 0.0) a.dacc[slot] += v * a.cell_area;
    }
}

template <bool TRACK, bool LC>
const void* kernel_of(bool lim)
{
    return lim ? reinterpret_cast<const void*>(step_resident_kernel<TRACK, LC, 1>)
               : reinterpret_cast<const void*>(step_resident_kernel<TRACK, LC, 0>);
}

const void* kernel_for(bool track, bool lc, bool lim)
{
    return track ? (lc ? kernel_of<true, true>(lim) : kernel_of<true, false>(lim))
                 : (lc ? kernel_of<false, true>(lim) : kernel_of<false, false>(lim));
}

size_t band_bytes(int nx, int rows, bool track, bool lc)
{
    const size_t nq = (nx + 3) / 4, P = 4 * nq + 4;
    return 4 * (P * (5 * (size_t)rows + 7) + (track ? P * rows : 0) + (lc ? nq * rows : 0));
}

}  // namespace

// Bands of a member, and their rows: as many as give every CTA an SM of its
// own, no more than the rows need.  No bands (0) where the state does not fit.
ResidentShape resident_shape(int ny, int nx, int M, int n_sm, size_t smem_max, bool track, bool lc)
{
    ResidentShape sh{0, 0, 0};
    if (M > n_sm) return sh;
    const int most = n_sm / M;
    const int rows = (ny + most - 1) / most;
    const size_t bytes = band_bytes(nx, rows, track, lc);
    if (bytes + 2048 > smem_max) return sh;
    sh.rows = rows;
    sh.bands = (ny + rows - 1) / rows;
    sh.smem = bytes;
    return sh;
}

cudaError_t launch_resident(const ResidentArgs& t, const ResidentShape& sh, cudaStream_t s)
{
    const bool track = t.a.hmax_field != nullptr, lc = t.a.lc_on != 0, lim = t.a.limiter != 0;
    const void* f = kernel_for(track, lc, lim);
    const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh.smem);
    if (e != cudaSuccess) return e;
    void* args[] = {const_cast<ResidentArgs*>(&t)};
    return cudaLaunchCooperativeKernel(f, dim3(t.a.M * sh.bands), dim3(kThreads), args, sh.smem, s);
}

}  // namespace flood
