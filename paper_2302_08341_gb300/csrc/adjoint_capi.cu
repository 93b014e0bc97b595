// flood_adjoint: gradients of a gauge-misfit loss by reverse mode (extension
// beyond the paper).  Forward: the ensemble advances through the observation
// times exactly as flood_step would, logging each member's step lengths and
// keeping every state where memory allows (the steps then go from slot to slot
// of the kept states), else storing its state every ckpt_every steps.  Reverse:
// the adjoint kernel runs backwards through the states, seeded with the loss
// sensitivities at the observation times; from checkpoints segment by segment
// from the last, the segment's states recomputed bit for bit before (replay
// kernel).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

#include "adjoint.cuh"
#include "tma.cuh"
#include "grid.cuh"
#include "pf_kernels.cuh"

using flood::MemberClock;
#define CK FLOOD_CK

namespace {

cudaStream_t S(void* s) { return reinterpret_cast<cudaStream_t>(s); }

// Room for `count` values, kept from one adjoint to the next (its buffers were
// freed and allocated again by every call).
template <class T>
int grow(flood_grid* g, T** p, size_t& have, size_t count)
{
    if (*p && have >= count) return FLOOD_OK;
    have = 0;
    const int rc = flood::dalloc(g, p, count);
    if (!rc) have = count;
    return rc;
}

// The reverse stencil's automatic strip height.  The scalar gradients are FP64
// sums of one compensated FP32 sum per strip and lane, so their last digits
// (1e-7 relative) follow the strips: this rule keeps them where they are.  It
// is within 8 % of the best height at the sizes measured (us per step, replay
// included: 1000 x 1000 x 24 376 at its 32 rows, 364 at 16; 1024 x 1024 x 1 42 at
// 4, 40 at 6; 600 x 707 x 8 98 at 4, 90 at 8).
int reverse_rows(int ny, int nx, int M, int n_sm)
{
    const int spans = (nx + 127) / 128;
    int rh = 64;
    while (rh > 4 && (int64_t)M * spans * ((ny + rh - 1) / rh) < (int64_t)n_sm * 32) rh /= 2;
    return rh;
}

// The memory of kept states comes from a stream-ordered pool, one a device for
// every ensemble of the process, and goes back to it with the call.  What the
// pool holds unused the driver hands to any allocation of the process that
// finds too little memory otherwise (a buffer of the ensemble's own would be
// lost to the rest of the program, tens of GB of it), and the next window
// finds it mapped: 20 GB in 4 us, 18.7 ms the first time.  It holds at most a
// quarter of the device's memory, an eighth once an ensemble is destroyed.
struct StatePool {
    cudaMemPool_t pool = nullptr;  // (null: none can be had)
    size_t total = 0;              // the device's memory
};

StatePool state_pool()
{
    static std::mutex mu;
    static std::map<int, StatePool> pools;
    int dev = 0;
    size_t free_b = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return {};
    std::lock_guard<std::mutex> lock(mu);
    const auto it = pools.find(dev);
    if (it != pools.end()) return it->second;
    StatePool p;
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    uint64_t most = 0;
    if (cudaMemGetInfo(&free_b, &p.total) == cudaSuccess && cudaMemPoolCreate(&p.pool, &props) == cudaSuccess) {
        most = p.total / 4;
        cudaMemPoolSetAttribute(p.pool, cudaMemPoolAttrReleaseThreshold, &most);
    }
    cudaGetLastError();
    return p.pool ? pools[dev] = p : p;  // (a refusal may pass: asked again next time)
}

// The kept states of one call.
struct KeptStates {
    flood_grid* g;
    cudaStream_t s;
    KeptStates(flood_grid* g_, cudaStream_t s_) : g(g_), s(s_) {}
    ~KeptStates()
    {
        if (!g->kept) return;
        release();
        cudaStreamSynchronize(s);  // the memory is the pool's to give away once the free has run
    }
    void release()
    {
        if (g->kept) cudaFreeAsync(g->kept, s);
        g->kept = nullptr;
    }
    // Whether to keep every state of a window (`floats` of them in all) instead
    // of checkpoints to recompute from: the recomputation moves 26 bytes per
    // member-cell-step and takes a quarter of the gradient's time, the slots
    // cost nothing extra to write (24 members of 1000 x 1000, 60 steps, 20 GB:
    // 28.9 ms recomputing, 21.9 ms keeping).  Memory that the pool holds
    // already, or up to a third of what is free, and no more than it holds on to.
    bool keep(size_t floats)
    {
        release();
        const StatePool p = state_pool();
        const size_t bytes = floats * sizeof(float);
        size_t free_b = 0, total_b = 0;
        uint64_t held = 0, used = 0;
        if (p.pool && bytes <= p.total / 4 &&
            cudaMemPoolGetAttribute(p.pool, cudaMemPoolAttrReservedMemCurrent, &held) == cudaSuccess &&
            cudaMemPoolGetAttribute(p.pool, cudaMemPoolAttrUsedMemCurrent, &used) == cudaSuccess &&
            (bytes <= held - used || (cudaMemGetInfo(&free_b, &total_b) == cudaSuccess &&
                                      bytes <= (free_b + (size_t)(held - used)) / 3))) {
            void* mem = nullptr;
            if (cudaMallocFromPoolAsync(&mem, bytes, p.pool, s) == cudaSuccess) g->kept = static_cast<float*>(mem);
        }
        cudaGetLastError();
        g->kept_any |= g->kept != nullptr;
        return g->kept != nullptr;
    }
};

// The checkpoints of the window at hand: every state where they are kept.
float* window_states(const flood_grid* g) { return g->kept ? g->kept : g->ckpt; }

// The ensemble's volume counters (rain and inflow per member, outflow and clamp
// per slot, drained volume per slot with land cover) to or from g->vol0.
int copy_volumes(flood_grid* g, bool restore, cudaStream_t s)
{
    const size_t M = g->M, slots = M * g->nslot;
    double* at = g->vol0;
    const std::pair<double*, size_t> parts[] = {
        {g->rain_acc, M}, {g->vacc, slots * 2}, {g->inflow_acc, M}, {g->dacc, g->dacc ? slots : 0}};
    for (const auto& [p, n] : parts) {
        if (n)
            CK(g, cudaMemcpyAsync(restore ? p : at, restore ? at : p, sizeof(double) * n, cudaMemcpyDeviceToDevice, s));
        at += n;
    }
    return FLOOD_OK;
}

// Put the state saved in ckpt slot 0 back into each member's current buffer
// and restore the saved clocks and volume counters (a forward that overflowed
// the step log is redone).
int restore_start(flood_grid* g, const std::vector<MemberClock>& c0, cudaStream_t s)
{
    const int M = g->M;
    const size_t ms = 3 * g->plane;
    std::vector<MemberClock> now;
    int rc = flood::read_clocks(g, now, s);
    if (rc) return rc;
    std::vector<MemberClock> back = c0;
    for (int m = 0; m < M; ++m) {
        back[m].cur = now[m].cur;
        back[m].steps = 0;
        CK(g, cudaMemcpyAsync(g->state + (size_t)(now[m].cur * M + m) * ms, window_states(g) + (size_t)m * ms,
                              sizeof(float) * ms, cudaMemcpyDeviceToDevice, s));
    }
    CK(g, cudaMemcpyAsync(g->ms + (g->k % 3) * M, back.data(), sizeof(MemberClock) * M,
                          cudaMemcpyHostToDevice, s));
    if ((rc = copy_volumes(g, true, s))) return rc;
    CK(g, cudaStreamSynchronize(s));
    return FLOOD_OK;
}

// Where the steps went from kept slot to slot, each member's last state back
// into the ensemble's current buffer.
int slots_to_state(flood_grid* g, cudaStream_t s)
{
    const int M = g->M;
    const size_t ms = 3 * g->plane;
    std::vector<MemberClock> c(M);
    CK(g, cudaMemcpyAsync(c.data(), g->ms + (g->k % 3) * M, sizeof(MemberClock) * M, cudaMemcpyDeviceToHost, s));
    CK(g, cudaStreamSynchronize(s));
    for (int m = 0; m < M; ++m)
        CK(g, cudaMemcpyAsync(g->state + (size_t)(c[m].cur * M + m) * ms,
                              g->kept + ((size_t)flood::kept_slot(c[m].steps, g->log_cap) * M + m) * ms,
                              sizeof(float) * ms, cudaMemcpyDeviceToDevice, s));
    return FLOOD_OK;
}

// The window's forward: its steps are logged, and go from slot to slot where
// `slots`.  However it ends, later steps do neither, and the ensemble holds
// the state that its clocks stand at.
struct Logging {
    flood_grid* g;
    cudaStream_t s;
    Logging(flood_grid* g_, bool slots, cudaStream_t s_) : g(g_), s(s_)
    {
        g->logging = true;
        g->slots = slots;
    }
    ~Logging()
    {
        if (!g->logging) return;
        const std::string msg = g->msg;  // of the error that ends it
        end();
        g->msg = msg;
    }
    int end()
    {
        const int rc = g->slots ? slots_to_state(g, s) : FLOOD_OK;
        g->logging = g->slots = false;
        return rc;
    }
};

struct Events {
    cudaEvent_t e[3] = {nullptr, nullptr, nullptr};
    ~Events()
    {
        for (cudaEvent_t v : e)
            if (v) cudaEventDestroy(v);
    }
};

}  // namespace

namespace flood {

void trim_state_pool()
{
    const StatePool p = state_pool();
    if (p.pool) cudaMemPoolTrimTo(p.pool, p.total / 8);
}

}  // namespace flood

extern "C" int flood_adjoint(flood_grid* g, const flood_loss_spec* L, int ckpt_every, float* grad_n,
                             double* grad_rain, double* grad_scale, float* grad_h0, double* loss_out,
                             void* stream)
{
    const flood::TraceRange range("flood_adjoint");
    if (!g) return flood::fail(nullptr, FLOOD_ERR_ARG, "grid is NULL");
    if (g->M == 0) return flood::fail(g, FLOOD_ERR_STATE, "flood_ensemble_init has not been called");
    if (!L || L->n_samples < 1 || !(L->sample_dt > 0) || L->n_gauges < 1 || !L->cells || !L->d)
        return flood::fail(g, FLOOD_ERR_ARG, "invalid flood_loss_spec");
    if (ckpt_every < 0) return flood::fail(g, FLOOD_ERR_ARG, "ckpt_every must be >= 0");
    cudaStream_t s = S(stream);
    const int M = g->M, ns = L->n_samples, G = L->n_gauges;
    const size_t ms = 3 * g->plane;

    std::vector<MemberClock> c0;
    int rc = flood::read_clocks(g, c0, s);
    if (rc) return rc;
    const double t0 = c0[0].t;
    for (int m = 1; m < M; ++m)
        if (c0[m].t != t0) return flood::fail(g, FLOOD_ERR_STATE, "members are not at the same time");
    std::vector<int32_t> cells(G);
    std::vector<double> d((size_t)ns * G);
    CK(g, cudaMemcpy(cells.data(), L->cells, sizeof(int32_t) * G, cudaMemcpyDefault));
    CK(g, cudaMemcpy(d.data(), L->d, sizeof(double) * ns * G, cudaMemcpyDefault));
    for (int k = 0; k < G; ++k)
        if (cells[k] < 0 || (int64_t)cells[k] >= (int64_t)g->ny * g->nx)
            return flood::fail(g, FLOOD_ERR_ARG, "gauge cell index out of range");

    // saved start: clocks, volume counters (restored if the forward is redone)
    flood_grid::AdjointRoom& room = g->adj_room;
    if ((rc = grow(g, &g->vol0, room.vol0, (size_t)M * (2 + 3 * g->nslot)))) return rc;
    if ((rc = copy_volumes(g, false, s))) return rc;

    const double T = ns * L->sample_dt;
    const double dt_ref = g->p.dt_fixed > 0 ? g->p.dt_fixed : g->p.dt_cap;
    int cap = (int)std::ceil(T / dt_ref) + 2 * ns + 8;
    std::vector<int64_t> steps0(M);
    for (int m = 0; m < M; ++m) steps0[m] = c0[m].steps;
    std::vector<int> K_m(M);
    std::vector<int32_t> samp_step((size_t)ns * M);
    int K = 0;
    bool keep = false;  // every state of the window is kept: nothing is recomputed
    KeptStates kept(g, s);
    size_t n_ckpt = 0;
    Events ev;
    for (cudaEvent_t& e : ev.e) CK(g, cudaEventCreate(&e));
    // the gauges' cells, for the samples and the seeds
    if ((rc = grow(g, &g->samp_cells, room.samp_cells, G))) return rc;
    CK(g, cudaMemcpyAsync(g->samp_cells, cells.data(), sizeof(int32_t) * G, cudaMemcpyHostToDevice, s));
    for (int attempt = 0;; ++attempt) {
        keep = ckpt_every == 0 && kept.keep((size_t)(cap + 1) * M * ms);
        K = ckpt_every > 0 ? ckpt_every : keep ? 1 : std::max(1, (int)std::lround(std::sqrt((double)cap)));
        n_ckpt = (size_t)cap / K + 1;
        if (!keep && (rc = grow(g, &g->ckpt, g->ckpt_floats, n_ckpt * M * ms))) return rc;
        float* const states = window_states(g);
        // where every state is kept the TMA step goes from slot to slot (the
        // resident steps write each state to its slot as a checkpoint)
        const bool slots = keep && g->engine == 1 && g->maps_ok && g->wait_budget < 0 && !flood::steps_resident(g) &&
                           flood::encode_map_3d(&g->ckpt_map, states, g->ld, g->ny, (uint64_t)n_ckpt * M * 3,
                                                sizeof(float) * g->ld, sizeof(float) * g->plane,
                                                flood::tma_box_cols(), 1, 3) == 0;
        if ((rc = grow(g, &g->log, room.log, (size_t)M * cap))) return rc;
        if ((rc = grow(g, &g->samp_y, room.samp_y, (size_t)ns * M * G))) return rc;
        g->log_cap = cap;
        g->ckpt_every = K;
        // checkpoint 0: the starting state; clocks count steps from 0
        std::vector<MemberClock> cz;
        if ((rc = flood::read_clocks(g, cz, s))) return rc;
        for (int m = 0; m < M; ++m) {
            CK(g, cudaMemcpyAsync(states + (size_t)m * ms, g->state + (size_t)(cz[m].cur * M + m) * ms,
                                  sizeof(float) * ms, cudaMemcpyDeviceToDevice, s));
            cz[m].steps = 0;
        }
        CK(g, cudaMemcpyAsync(g->ms + (g->k % 3) * M, cz.data(), sizeof(MemberClock) * M,
                              cudaMemcpyHostToDevice, s));
        Logging log(g, slots, s);
        CK(g, cudaEventRecord(ev.e[0], s));
        int64_t kmax = 0;
        for (int sidx = 1; sidx <= ns; ++sidx) {
            if ((rc = flood_step(g, 0, t0 + sidx * L->sample_dt, stream))) return rc;
            if (slots)
                flood::launch_gauge_slots(states, g->ms + (g->k % 3) * M, cap, g->samp_cells, G, M, g->ld, g->nx,
                                          g->plane, g->samp_y + (size_t)(sidx - 1) * M * G, s);
            else
                flood::launch_gauge(g->state, g->ms + (g->k % 3) * M, g->samp_cells, G, M, g->ld, g->nx,
                                    g->plane, g->samp_y + (size_t)(sidx - 1) * M * G, s);
            g->launches++;
            std::vector<MemberClock> cc;
            if ((rc = flood::read_clocks(g, cc, s))) return rc;
            for (int m = 0; m < M; ++m) {
                samp_step[(size_t)(sidx - 1) * M + m] = (int32_t)cc[m].steps;
                K_m[m] = (int)std::min<int64_t>(cc[m].steps, INT32_MAX);
                kmax = std::max<int64_t>(kmax, cc[m].steps);
            }
        }
        if ((rc = log.end())) return rc;  // the window's end is the ensemble's state
        CK(g, cudaEventRecord(ev.e[1], s));
        if (kmax <= cap) break;
        if (attempt >= 4) return flood::fail(g, FLOOD_ERR_STATE, "step log could not hold the window");
        if ((rc = restore_start(g, c0, s))) return rc;
        cap = (int)std::min<int64_t>((int64_t)kmax * 2 + 8, INT32_MAX / 2);
    }

    // loss per member from the recorded gauge outputs
    std::vector<float> yh((size_t)ns * M * G);
    CK(g, cudaMemcpy(yh.data(), g->samp_y, sizeof(float) * yh.size(), cudaMemcpyDeviceToHost));
    if (loss_out)
        for (int m = 0; m < M; ++m) {
            double acc = 0.0;
            for (int si = 0; si < ns; ++si)
                for (int k = 0; k < G; ++k) {
                    const double e = (double)yh[((size_t)si * M + m) * G + k] - d[(size_t)si * G + k];
                    acc += e * e;
                }
            loss_out[m] = acc;
        }

    // reverse sweep buffers
    // the states the reverse pass reads: a segment recomputed from its
    // checkpoint, or the whole window's slots
    if (keep) K = cap;
    const size_t n_slots = keep ? n_ckpt : (size_t)K + 1;
    if (!keep && (size_t)(K + 1) * M * ms > g->seg_floats) {
        if ((rc = grow(g, &g->seg, g->seg_floats, (size_t)(K + 1) * M * ms))) return rc;
    }
    float* const seg = keep ? g->kept : g->seg;
    if ((rc = grow(g, &g->lam, room.lam, 2 * (size_t)M * ms))) return rc;
    const int rrows = g->launch_fixed ? g->rows_per_strip : reverse_rows(g->ny, g->nx, M, g->n_sm);
    const int nslot = flood::step_nslot(g->ny, g->nx, rrows);
    if ((rc = grow(g, &g->gpart, room.gpart, (size_t)M * nslot * 2 + M))) return rc;
    if ((rc = grow(g, &g->seg_end, room.seg_end, M))) return rc;
    if ((rc = grow(g, &g->samp_step, room.samp_step, (size_t)ns * M))) return rc;
    if ((rc = grow(g, &g->samp_d, room.samp_d, (size_t)ns * G))) return rc;
    if (grad_n) {
        if ((rc = grow(g, &g->gnm, room.gnm, (size_t)M * g->plane))) return rc;
        if ((rc = grow(g, &g->gn_out, room.gn_out, (size_t)g->ny * g->nx))) return rc;
        CK(g, cudaMemsetAsync(g->gnm, 0, sizeof(float) * M * g->plane, s));
    }
    CK(g, cudaMemsetAsync(g->lam, 0, sizeof(float) * 2 * M * ms, s));
    CK(g, cudaMemsetAsync(g->gpart, 0, sizeof(double) * M * nslot * 2, s));
    double* const rscale = g->gpart + (size_t)M * nslot * 2;  // 1 / scale of every member, behind the partials
    flood::launch_reciprocals(g->scale, M, rscale, s);
    g->launches++;
    if (g->lc_on) {
        if ((rc = grow(g, &g->gdpart, room.gdpart, (size_t)M * nslot))) return rc;
        CK(g, cudaMemsetAsync(g->gdpart, 0, sizeof(double) * M * nslot, s));
    }
    CK(g, cudaMemcpyAsync(g->samp_step, samp_step.data(), sizeof(int32_t) * ns * M,
                          cudaMemcpyHostToDevice, s));
    CK(g, cudaMemcpyAsync(g->samp_d, d.data(), sizeof(double) * ns * G, cudaMemcpyHostToDevice, s));

    const size_t plane = g->plane;
    // tensor maps of the TMA-staged replay and reverse stencil (direct loads
    // otherwise)
    flood::AdjTmaArgs tma{};
    bool use_tma = g->engine == 1 && g->maps_ok;
    if (use_tma) {
        const int bc = flood::adjoint_tma_box_cols();
        const uint64_t s1 = sizeof(float) * g->ld, s2 = sizeof(float) * g->plane;
        use_tma =
            flood::encode_map_3d(&tma.seg_map, seg, g->ld, g->ny, (uint64_t)n_slots * M * 3, s1,
                                 s2, bc, 1, 3) == 0 &&
            flood::encode_map_3d(&tma.seg1_map, seg, g->ld, g->ny, (uint64_t)n_slots * M * 3, s1,
                                 s2, bc, 1, 1) == 0 &&
            flood::encode_map_3d(&tma.lam_map, g->lam, g->ld, g->ny, (uint64_t)2 * M * 3, s1, s2, bc,
                                 1, 3) == 0 &&
            (!grad_n || flood::encode_map_3d(&tma.gn_map, g->gnm, g->ld, g->ny, (uint64_t)M, s1, s2,
                                             bc, 1, 1) == 0);
        // with land cover the bed and the class codes, as the forward stages them
        tma.static_map = g->lc_on ? g->static_map_lc : g->static_map;
    }
    // land cover with direct loads: each member's Manning n field and the share
    // of the rain that stays, from the classes (the TMA form looks them up)
    const bool fields = g->lc_on && !use_tma;
    if (fields && (rc = flood::land_adjoint_fields(g, s))) return rc;

    // the steps whose result some member is observed after
    std::vector<std::vector<int32_t>> seen(M);
    for (int m = 0; m < M; ++m)
        for (int si = 0; si < ns; ++si) seen[m].push_back(samp_step[(size_t)si * M + m]);

    const int kmax = *std::max_element(K_m.begin(), K_m.end());
    const int n_seg = (kmax + K - 1) / K;
    int lam_in = 0;
    std::vector<int> seg_end(M);
    for (int cs = n_seg - 1; cs >= 0; --cs) {
        const int first = cs * K;
        int len = 0;
        for (int m = 0; m < M; ++m) {
            seg_end[m] = std::min(first + K, K_m[m]);
            len = std::max(len, seg_end[m] - first);
        }
        if (len <= 0) continue;
        CK(g, cudaMemcpyAsync(g->seg_end, seg_end.data(), sizeof(int) * M, cudaMemcpyHostToDevice, s));
        if (!keep)
            CK(g, cudaMemcpyAsync(g->seg, g->ckpt + (size_t)cs * M * ms, sizeof(float) * M * ms,
                                  cudaMemcpyDeviceToDevice, s));
        flood::StepArgs a = flood::step_args(g, -1.0);
        a.log = g->log;
        a.dt_log_cap = g->log_cap;
        a.ckpt = nullptr;
        a.seg = seg;
        a.seg_end = g->seg_end;
        a.seg_first = first;
        flood::TmaArgs rt;
        if (use_tma) {
            rt.state_map = tma.seg_map;
            rt.static_map = g->lc_on ? g->static_map_lc : g->static_map;
        }
        for (int i = 0; i < len && !keep; ++i) {
            a.replay_i = i;
            if (use_tma) {
                rt.a = a;
                flood::launch_replay_tma(rt, g->members_per_cta, s);
            } else {
                flood::launch_replay(a, g->members_per_cta, s);
            }
            g->launches++;
        }
        flood::AdjArgs b{};
        b.seg = seg;
        b.lam = g->lam;
        b.gn = grad_n ? g->gnm : nullptr;
        b.gpart = g->gpart;
        b.z = g->z;
        b.n = fields ? g->lc_adj + plane : g->n;
        b.n_mstride = fields ? plane : 0;
        b.rw = fields ? g->lc_adj + (size_t)(M + 1) * plane : nullptr;
        b.dflag = fields ? g->lc_adj + (size_t)(M + 2) * plane : nullptr;
        b.gdpart = g->lc_on ? g->gdpart : nullptr;
        if (g->lc_on) {
            b.lc_n = g->lc_n;
            for (int q = 0; q < 4; ++q) {
                b.lc_runoff[q] = g->lc_runoff[q];
                b.lc_drains[q] = g->lc_drains[q];
            }
        }
        b.scale = g->scale;
        b.rscale = rscale;
        b.log = g->log;
        b.seg_end = g->seg_end;
        b.dt_log_cap = g->log_cap;
        b.seg_first = first;
        b.plane = g->plane;
        b.ny = g->ny; b.nx = g->nx; b.ld = g->ld; b.M = M;
        b.rows_per_strip = rrows;
        b.nslot = nslot;
        b.g = g->p.g;
        b.dxd = g->p.dx;
        b.h_eps = (float)g->p.h_eps;
        b.edge_drop = (float)(g->p.edge_slope * g->p.dx);
        b.limiter = g->p.limiter;
        b.east_out = g->p.east_outflow;
        b.south_out = g->p.south_outflow;
        b.err = g->err;
        for (int i = 0; i < len; ++i) {
            b.rev_i = i;
            b.lam_in = lam_in;
            // sensitivities of the loss enter where a member's step ends at an
            // observation: few steps, the others launch nothing
            bool seed = false;
            for (int m = 0; m < M && !seed; ++m) {
                const int after = seg_end[m] - i;  // the step's result, counted from the start
                seed = after > first && std::binary_search(seen[m].begin(), seen[m].end(), after);
            }
            if (seed) {
                flood::launch_seed(b, g->samp_step, g->samp_y, g->samp_d, g->samp_cells, ns, G, s);
                g->launches++;
            }
            if (use_tma) {
                tma.a = b;
                flood::launch_adjoint_tma(tma, g->members_per_cta, s);
            } else {
                flood::launch_adjoint(b, g->members_per_cta, s);
            }
            g->launches++;
            lam_in = 1 - lam_in;
        }
        CK(g, cudaGetLastError());
    }
    CK(g, cudaEventRecord(ev.e[2], s));
    CK(g, cudaStreamSynchronize(s));
    if ((rc = flood::check_err(g))) return rc;
    float fms = 0.0f, rms = 0.0f;
    cudaEventElapsedTime(&fms, ev.e[0], ev.e[1]);
    cudaEventElapsedTime(&rms, ev.e[1], ev.e[2]);
    g->adj_fwd_ms = fms;
    g->adj_rev_ms = rms;

    if (grad_h0)
        for (int m = 0; m < M; ++m)
            CK(g, cudaMemcpy2DAsync(grad_h0 + (size_t)m * g->ny * g->nx, sizeof(float) * g->nx,
                                    g->lam + ((size_t)lam_in * M + m) * ms, sizeof(float) * g->ld,
                                    sizeof(float) * g->nx, g->ny, cudaMemcpyDefault, s));
    if (grad_n) {
        flood::launch_reduce_members(g->gnm, M, g->ny, g->nx, g->ld, g->plane, g->gn_out, s);
        g->launches++;
        CK(g, cudaMemcpyAsync(grad_n, g->gn_out, sizeof(float) * g->ny * g->nx, cudaMemcpyDefault, s));
    }
    if (grad_rain || grad_scale) {
        std::vector<double> gp((size_t)M * nslot * 2);
        CK(g, cudaMemcpyAsync(gp.data(), g->gpart, sizeof(double) * gp.size(), cudaMemcpyDeviceToHost, s));
        CK(g, cudaStreamSynchronize(s));
        for (int m = 0; m < M; ++m) {
            double gr = 0.0, gs = 0.0;
            for (int k = 0; k < nslot; ++k) {
                gr += gp[((size_t)m * nslot + k) * 2];
                gs += gp[((size_t)m * nslot + k) * 2 + 1];
            }
            if (grad_rain) grad_rain[m] = gr;
            if (grad_scale) grad_scale[m] = gs;
        }
    }
    g->adj_gdrain.assign(M, 0.0);
    if (g->lc_on) {
        std::vector<double> gp((size_t)M * nslot);
        CK(g, cudaMemcpyAsync(gp.data(), g->gdpart, sizeof(double) * gp.size(), cudaMemcpyDeviceToHost, s));
        CK(g, cudaStreamSynchronize(s));
        for (int m = 0; m < M; ++m)
            for (int k = 0; k < nslot; ++k) g->adj_gdrain[m] += gp[(size_t)m * nslot + k];
    }
    // clocks keep counting from where they were
    std::vector<MemberClock> ce;
    if ((rc = flood::read_clocks(g, ce, s))) return rc;
    for (int m = 0; m < M; ++m) ce[m].steps += steps0[m];
    CK(g, cudaMemcpyAsync(g->ms + (g->k % 3) * M, ce.data(), sizeof(MemberClock) * M,
                          cudaMemcpyHostToDevice, s));
    CK(g, cudaStreamSynchronize(s));
    // what a calibration step may use: the gradients of this ensemble as it is now
    g->adj_epoch = g->epoch;
    g->adj_gn = grad_n != nullptr;
    g->adj_ns = ns;
    g->adj_G = G;
    g->adj_nslot = nslot;
    return FLOOD_OK;
}

extern "C" int flood_adjoint_timing(const flood_grid* g, double* forward_ms, double* reverse_ms)
{
    if (!g) return flood::fail(nullptr, FLOOD_ERR_ARG, "grid is NULL");
    if (forward_ms) *forward_ms = g->adj_fwd_ms;
    if (reverse_ms) *reverse_ms = g->adj_rev_ms;
    return FLOOD_OK;
}
