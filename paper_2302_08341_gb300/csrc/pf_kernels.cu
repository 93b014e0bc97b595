// Particle-filter kernels (Section 2.2, Section 3.3 DA steps (I)-(V),
// perturbation of Section 4.4), all on the device so the ensemble never
// leaves HBM: gauge sampling, weights / N_eff / systematic resampling /
// slot assignment in one single-block kernel, and a grid-stride copy of the
// duplicated members' states.  Also the per-member storage and max-depth
// reductions.
#include "flood_internal.cuh"
#include "pf_kernels.cuh"

namespace flood {

namespace {

// DA step (I): y[i][k] = depth of member i at gauge cell k.
__device__ __forceinline__ void gauge_one(const float* state, const MemberClock* ms, const int32_t* cells, int G,
                                          int M, int ld, int nx, size_t plane, float* y)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= M * G) return;
    const int m = t / G, k = t % G;
    const int cell = cells[k];
    const int r = cell / nx, c = cell % nx;
    const float* h = state + (size_t)(ms[m].cur * M + m) * 3 * plane;
    y[t] = h[(size_t)r * ld + c];
}

__global__ void gauge_kernel(const float* __restrict__ state, const MemberClock* __restrict__ ms,
                             const int32_t* __restrict__ cells, int G, int M, int ld, int nx,
                             size_t plane, float* __restrict__ y)
{
    gauge_one(state, ms, cells, G, M, ld, nx, plane, y);
}

__global__ void gauge_args_kernel(const float* __restrict__ state, const MemberClock* __restrict__ ms,
                                  const __grid_constant__ GaugeCells cells, int G, int M, int ld, int nx, size_t plane,
                                  float* __restrict__ y)
{
    gauge_one(state, ms, cells.cell, G, M, ld, nx, plane, y);
}

// The same from checkpoint slots: each member's state after its steps so far.
__global__ void gauge_slots_kernel(const float* __restrict__ slots, const MemberClock* __restrict__ ms, int last,
                                   const int32_t* __restrict__ cells, int G, int M, int ld, int nx, size_t plane,
                                   float* __restrict__ y)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= M * G) return;
    const int m = t / G, k = t % G;
    const int cell = cells[k];
    y[t] = slots[((size_t)kept_slot(ms[m].steps, last) * M + m) * 3 * plane + (size_t)(cell / nx) * ld + cell % nx];
}

// DA steps (II)-(IV) and the bookkeeping of step (V), one block.
//
// Bound by latency: a few hundred FP64 operations per member on a GPU whose
// FP64 pipe is narrow.  Everything that does not depend on an order runs one
// member per thread (log-weights, exponentials, divisions, the search of each
// offset in the cumulative weights, slot map, parameters).  The three sums
// whose order the results depend on (the normaliser, sum w^2 and the
// cumulative weights) stay sequential in index order, a bare chain of FP64
// additions each, the last two side by side in two warps, so every result is
// the one of the sequential definition.  96 members x 6 gauges: 231 us when
// one thread did all of it, 23 us now (launch alone, cold caches).
constexpr int kPfThreads = 256;
constexpr int kPfMaxMembers = 3072;  // the block's shared memory: 32 B per member
__host__ __device__ constexpr size_t pf_smem(int M) { return (size_t)M * 32; }

// Positions (of [0, n)) where keep(i) holds, in order, into out; the warp's
// lanes take 32 at a time.  Returns their number.
template <class Keep, class Put>
__device__ __forceinline__ int warp_compact(int n, Keep keep, Put put)
{
    const int lane = threadIdx.x & 31;
    int at = 0;
    for (int base = 0; base < n; base += 32) {
        const int i = base + lane;
        const bool k = i < n && keep(i);
        const unsigned mask = __ballot_sync(0xffffffffu, k);
        if (k) put(at + __popc(mask & ((1u << lane) - 1u)), i);
        at += __popc(mask);
    }
    return at;
}

__global__ void __launch_bounds__(kPfThreads) pf_kernel(PfArgs a)
{
    extern __shared__ double sm[];
    const int M = a.M, G = a.G, tid = threadIdx.x, nt = blockDim.x;
    double* __restrict__ lw = sm;          // [M] log-weights, exponentials, then weights
    double* __restrict__ cw = sm + M;      // [M] cumulative weights
    float* rm_old = (float*)(sm + 2 * M);  // [M]
    float* sc_old = rm_old + M;            // [M]
    int* idx = (int*)(sc_old + M);         // [M]
    int* cnt = idx + M;                    // [M]
    __shared__ double s_wmax[kPfThreads / 32], s_sum;
    __shared__ int s_resample, s_nc;

    double lmax = -INFINITY;
    for (int i = tid; i < M; i += nt) {
        double chi2 = 0.0;
        for (int k = 0; k < G; ++k) {
            double s = a.sigma_rel > 0.0 ? a.sigma_rel * a.d[k] : a.sigma[k];
            double e = ((double)a.y[(size_t)i * G + k] - a.d[k]) / s;
            chi2 += e * e;
        }
        const double l = log(a.w[i]) - 0.5 * chi2;   // log of Eq. 10
        lw[i] = l;
        lmax = l > lmax ? l : lmax;
        rm_old[i] = a.rain_mult[i];
        sc_old[i] = a.scale[i];
        cnt[i] = 0;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const double o = __shfl_xor_sync(0xffffffffu, lmax, off);
        lmax = o > lmax ? o : lmax;
    }
    if ((tid & 31) == 0) s_wmax[tid >> 5] = lmax;
    __syncthreads();
    lmax = s_wmax[0];
    for (int k = 1; k < nt / 32; ++k) lmax = s_wmax[k] > lmax ? s_wmax[k] : lmax;
    if (!(lmax > -INFINITY)) {  // every weight zero: leave the ensemble untouched
        if (tid == 0) {
            *a.status = 1;
            *a.resampled = 0;
            *a.n_copy = 0;
            *a.neff = 0.0;
        }
        for (int i = tid; i < M; i += nt) a.idx[i] = i;
        return;
    }
    for (int i = tid; i < M; i += nt) lw[i] = exp(lw[i] - lmax);
    __syncthreads();
    if (tid == 0) {
        double sum = 0.0;
        for (int i = 0; i < M; ++i) sum += lw[i];
        s_sum = sum;
    }
    __syncthreads();
    const double sum = s_sum;
    for (int i = tid; i < M; i += nt) {
        const double w = lw[i] / sum;      // Eq. 11
        lw[i] = w;
        a.w_post[i] = w;
    }
    __syncthreads();
    if (tid == 0) {
        double s2 = 0.0;
        for (int i = 0; i < M; ++i) {
            const double w = lw[i];
            s2 += w * w;
        }
        const double neff = 1.0 / s2;      // Eq. 12
        *a.neff = neff;
        *a.status = 0;
        const bool resample = a.force || neff < a.n_thr_frac * (double)M;
        *a.resampled = resample ? 1 : 0;
        s_resample = resample ? 1 : 0;
        if (!resample) *a.n_copy = 0;
    } else if (tid == 32) {
        double acc = 0.0;
        for (int i = 0; i < M; ++i) {
            acc += lw[i];
            cw[i] = acc;
        }
    }
    __syncthreads();
    if (!s_resample) {
        for (int i = tid; i < M; i += nt) {
            a.w[i] = lw[i];
            a.idx[i] = i;
        }
        return;
    }
    // systematic resampling: particle i owns [c_{i-1}, c_i), c_{M-1} set to 1;
    // the offset's particle is the first i with c_i above it, the last one
    // failing that (the weights are non-negative, so c never decreases)
    for (int j = tid; j < M; j += nt) {
        const double uj = (a.u + (double)j) / (double)M;
        int lo = 0, hi = M - 1;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (cw[mid] <= uj) lo = mid + 1; else hi = mid;
        }
        idx[j] = lo;
        a.idx[j] = lo;
        atomicAdd(&cnt[lo], 1);
    }
    __syncthreads();
    // DA step (V): duplicates per particle; survivors keep their slot, extra
    // copies (in particle order) fill dropped slots (in slot order).  idx is
    // sorted, so every entry equal to the one before it is an extra copy
    if (tid < 32) {
        const int nc = warp_compact(M, [&](int s) { return cnt[s] == 0; },
                                    [&](int q, int s) { a.copy_dst[q] = s; });
        if (tid == 0) {
            *a.n_copy = nc;
            s_nc = nc;
        }
    } else if (tid < 64) {
        warp_compact(M, [&](int j) { return j > 0 && idx[j] == idx[j - 1]; },
                     [&](int q, int j) { a.copy_src[q] = idx[j]; });
    }
    for (int s = tid; s < M; s += nt) a.src[s] = s;
    __syncthreads();
    const int nc = s_nc;
    // the copied members inherit their source's maximum depth (same time)
    for (int q = tid; q < nc; q += nt) {
        const int s = a.copy_dst[q], p = a.copy_src[q];
        a.src[s] = p;
        a.ms[s].hmax_bits = a.ms[p].hmax_bits;
    }
    __syncthreads();
    // parameters follow their particle; rain multiplier perturbed by beta
    for (int s = tid; s < M; s += nt) {
        const int p = a.src[s];
        a.rain_mult[s] = rm_old[p] * a.beta[s];
        a.scale[s] = sc_old[p];
        a.w[s] = 1.0 / (double)M;
    }
}

// DA step (V): copy the duplicated particles' h, qx, qy planes into the
// dropped slots.  Grid-stride over (copy, plane, float4); reads the device
// copy count so that the launch needs no host synchronisation.
__global__ void copy_kernel(float* __restrict__ state, const MemberClock* __restrict__ ms,
                            const int32_t* __restrict__ n_copy, const int32_t* __restrict__ dsts,
                            const int32_t* __restrict__ srcs, int M, size_t plane4)
{
    const int nc = *n_copy;
    if (nc == 0) return;
    const size_t per = 3 * plane4;  // float4s per member
    const size_t total = (size_t)nc * per;
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (size_t)gridDim.x * blockDim.x) {
        const int q = (int)(t / per);
        const size_t e = t - (size_t)q * per;
        const int d = dsts[q], s = srcs[q];
        const float4* from = reinterpret_cast<const float4*>(state) + (size_t)(ms[s].cur * M + s) * per;
        float4* to = reinterpret_cast<float4*>(state) + (size_t)(ms[d].cur * M + d) * per;
        to[e] = from[e];
    }
}

// Systematic resampling alone (DA step (IV)), one thread.
__global__ void resample_kernel(int M, const double* __restrict__ w, double u,
                                int32_t* __restrict__ idx)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    double acc = w[0];
    double ci = (M == 1) ? 1.0 : acc;
    int i = 0;
    for (int j = 0; j < M; ++j) {
        const double uj = (u + (double)j) / (double)M;
        while (i < M - 1 && ci <= uj) {
            ++i;
            acc += w[i];
            ci = (i == M - 1) ? 1.0 : acc;
        }
        idx[j] = i;
    }
}

// Per-member FP64 storage partials: block b of member m sums a fixed set of
// rows in a fixed order; the final pass adds the partials in index order.
__global__ void storage_partial_kernel(const float* __restrict__ state,
                                       const MemberClock* __restrict__ ms, int M, int ny, int nx,
                                       int ld, size_t plane, int rows_per_block,
                                       double* __restrict__ part)
{
    const int m = blockIdx.y;
    const float* h = state + (size_t)(ms[m].cur * M + m) * 3 * plane;
    const int r0 = blockIdx.x * rows_per_block, r1 = min(r0 + rows_per_block, ny);
    double acc = 0.0;
    for (int r = r0; r < r1; ++r)
        for (int c = threadIdx.x; c < nx; c += blockDim.x) acc += (double)h[(size_t)r * ld + c];
    __shared__ double red[256];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[(size_t)m * gridDim.x + blockIdx.x] = red[0];
}

__global__ void storage_final_kernel(const double* __restrict__ part, int nb, int M,
                                     double area, double* __restrict__ out)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    double acc = 0.0;
    for (int b = 0; b < nb; ++b) acc += part[(size_t)m * nb + b];
    out[m] = acc * area;
}

// Maximum depth of each member's current state (initialisation of the
// Eq. 4 input); non-negative floats order like their bit patterns.
__global__ void hmax_kernel(const float* __restrict__ state, MemberClock* __restrict__ ms, int M,
                            int ny, int nx, int ld, size_t plane)
{
    const int m = blockIdx.y;
    const float* h = state + (size_t)(ms[m].cur * M + m) * 3 * plane;
    unsigned best = 0u;
    const size_t n = (size_t)ny * nx;
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (size_t)gridDim.x * blockDim.x) {
        const size_t r = t / nx, c = t % nx;
        best = max(best, __float_as_uint(fmaxf(h[r * ld + c], 0.0f)) & 0x7fffffffu);
    }
    best = __reduce_max_sync(0xffffffffu, best);
    if ((threadIdx.x & 31) == 0) atomicMax(&ms[m].hmax_bits, best);
}

}  // namespace

void launch_gauge(const float* state, const MemberClock* ms, const int32_t* cells, int G, int M,
                  int ld, int nx, size_t plane, float* y, cudaStream_t s)
{
    const int n = M * G;
    gauge_kernel<<<(n + 127) / 128, 128, 0, s>>>(state, ms, cells, G, M, ld, nx, plane, y);
}

void launch_gauge_args(const float* state, const MemberClock* ms, const GaugeCells& cells, int G, int M, int ld,
                       int nx, size_t plane, float* y, cudaStream_t s)
{
    gauge_args_kernel<<<(M * G + 127) / 128, 128, 0, s>>>(state, ms, cells, G, M, ld, nx, plane, y);
}

void launch_gauge_slots(const float* slots, const MemberClock* ms, int last, const int32_t* cells, int G, int M,
                        int ld, int nx, size_t plane, float* y, cudaStream_t s)
{
    gauge_slots_kernel<<<(M * G + 127) / 128, 128, 0, s>>>(slots, ms, last, cells, G, M, ld, nx, plane, y);
}

cudaError_t launch_pf(const PfArgs& a, cudaStream_t s)
{
    // the shared memory of more members is refused here, before anything is
    // launched that would read what the filter did not write
    if (a.M > kPfMaxMembers) return cudaErrorInvalidValue;
    if (pf_smem(a.M) > 32 * 1024) {  // each time: the attribute is the current device's
        const cudaError_t e = cudaFuncSetAttribute(pf_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)pf_smem(kPfMaxMembers));
        if (e != cudaSuccess) return e;
    }
    pf_kernel<<<1, kPfThreads, pf_smem(a.M), s>>>(a);
    return cudaGetLastError();
}

void launch_copy(float* state, const MemberClock* ms, const int32_t* n_copy, const int32_t* dsts,
                 const int32_t* srcs, int M, size_t plane, int n_sm, cudaStream_t s)
{
    copy_kernel<<<n_sm * 4, 512, 0, s>>>(state, ms, n_copy, dsts, srcs, M, plane / 4);
}

void launch_resample(int M, const double* w, double u, int32_t* idx, cudaStream_t s)
{
    resample_kernel<<<1, 32, 0, s>>>(M, w, u, idx);
}

int launch_storage(const float* state, const MemberClock* ms, int M, int ny, int nx, int ld,
                   size_t plane, double area, double* part, int part_cap, double* out,
                   cudaStream_t s)
{
    const int rows = 16;
    const int nb = (ny + rows - 1) / rows;
    if (nb > part_cap) return -1;
    storage_partial_kernel<<<dim3(nb, M), 256, 0, s>>>(state, ms, M, ny, nx, ld, plane, rows, part);
    storage_final_kernel<<<(M + 127) / 128, 128, 0, s>>>(part, nb, M, area, out);
    return 0;
}

void launch_hmax(const float* state, MemberClock* ms, int M, int ny, int nx, int ld, size_t plane,
                 int n_sm, cudaStream_t s)
{
    const size_t n = (size_t)ny * nx;
    int bx = (int)((n + 255) / 256);
    if (bx > n_sm * 2) bx = n_sm * 2;
    hmax_kernel<<<dim3(bx, M), 256, 0, s>>>(state, ms, M, ny, nx, ld, plane);
}

}  // namespace flood
