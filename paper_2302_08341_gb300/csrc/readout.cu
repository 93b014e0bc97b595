// Reading results out: a member's state into the caller's device memory, the
// per-member scalars, and the stored volume of every scenario of a batch.
//
// These calls were bound by host round trips: a state cost 39 us, most of it a
// 24-byte copy of the member's clock (which buffer is current) and the wait
// for it, the scalars five copies, and a batch's volumes two launches per
// scenario (419 us for 16).  The kernels read the clock where it is, gather
// the scalars into one block, and take every scenario in one launch: reading
// the 96 states of a 2000 x 2000 ensemble after 30 steps takes 5 ms less of
// 50.7, an assimilation with its scalars and two states 291 us instead of 396,
// the volumes and states of 16 scenarios 0.75 ms less of 4.97.
#include "readout.cuh"

#include <cudaTypedefs.h>

namespace flood {

namespace {

// Rows of the current h, qx, qy planes (blockIdx.y) without their padding.
// VEC: rows of whole float4s in 16-byte aligned arrays; otherwise the rows of
// the output start anywhere, and a thread has eight words in flight instead.
template <bool VEC>
__global__ void read_state_kernel(const float* __restrict__ state, size_t buffer, const MemberClock* clk, int ny,
                                  int nx, int ld, size_t plane, float* h, float* qx, float* qy)
{
    float* const out = blockIdx.y == 0 ? h : blockIdx.y == 1 ? qx : qy;
    if (!out) return;
    const float* const src = state + (size_t)clk->cur * buffer + blockIdx.y * plane;
    for (int r = blockIdx.x * blockDim.y + threadIdx.y; r < ny; r += gridDim.x * blockDim.y) {
        const float* p = src + (size_t)r * ld;
        float* o = out + (size_t)r * nx;
        if (VEC) {
            for (int c = 4 * threadIdx.x; c < nx; c += 4 * blockDim.x)
                *reinterpret_cast<float4*>(o + c) = *reinterpret_cast<const float4*>(p + c);
            continue;
        }
        constexpr int kWords = 8;
        for (int c = threadIdx.x; c < nx; c += kWords * blockDim.x) {
            float v[kWords];
#pragma unroll
            for (int i = 0; i < kWords; ++i)
                if (c + i * (int)blockDim.x < nx) v[i] = __ldg(p + c + i * blockDim.x);
#pragma unroll
            for (int i = 0; i < kWords; ++i)
                if (c + i * (int)blockDim.x < nx) o[c + i * blockDim.x] = v[i];
        }
    }
}

__global__ void pack_members_kernel(const MemberClock* __restrict__ clk, const float* __restrict__ rain,
                                    const float* __restrict__ scale, const double* __restrict__ w, int M,
                                    MemberRow* __restrict__ out)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    MemberRow r;
    r.t = clk[m].t;
    r.steps = clk[m].steps;
    r.w = w[m];
    r.rain = rain[m];
    r.scale = scale[m];
    r.hmax = __uint_as_float(clk[m].hmax_bits);
    r.pad = 0.0f;
    out[m] = r;
}

// As storage_partial_kernel and storage_final_kernel (pf_kernels.cu), for the
// entries [e0, e0 + gridDim.y) of a batch, each with its own grid.
constexpr int kRows = 16;

__global__ void batch_storage_partial_kernel(const ScenDesc* __restrict__ desc, const MemberClock* __restrict__ ms,
                                             int e0, double* __restrict__ part, int nb_max)
{
    const int e = e0 + blockIdx.y;
    const int ny = desc[e].ny, nx = desc[e].nx, ld = desc[e].ld;
    const int r0 = blockIdx.x * kRows, r1 = min(r0 + kRows, ny);
    if (r0 >= ny) return;
    const float* h = desc[e].state + (size_t)ms[e].cur * 3 * desc[e].plane;
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
    if (threadIdx.x == 0) part[(size_t)blockIdx.y * nb_max + blockIdx.x] = red[0];
}

__global__ void batch_storage_final_kernel(const ScenDesc* __restrict__ desc, const double* __restrict__ part,
                                           int e0, int n, int nb_max, double area, double* __restrict__ out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int nb = (desc[e0 + i].ny + kRows - 1) / kRows;
    double acc = 0.0;
    for (int b = 0; b < nb; ++b) acc += part[(size_t)i * nb_max + b];
    out[e0 + i] = acc * area;
}

}  // namespace

bool pageable(const void* p)
{
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeUnregistered;
}

// An allocation of the current device (size 0: none).
struct Allocation {
    uintptr_t base = 0;
    size_t size = 0;
    bool holds(const void* p, size_t bytes) const
    {
        const uintptr_t q = reinterpret_cast<uintptr_t>(p);
        return q >= base && q - base <= size && bytes <= size - (q - base);
    }
};

static Allocation allocation_of(const void* p)
{
    Allocation r;
    cudaPointerAttributes at{};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return r;
    }
    if (at.type != cudaMemoryTypeDevice || at.device != dev) return r;
    static const PFN_cuMemGetAddressRange_v3020 range = [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuMemGetAddressRange", &fn, 3020, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            fn = nullptr;
        return reinterpret_cast<PFN_cuMemGetAddressRange_v3020>(fn);
    }();
    CUdeviceptr base = 0;
    size_t size = 0;
    if (range && range(&base, &size, reinterpret_cast<CUdeviceptr>(p)) == CUDA_SUCCESS) {
        r.base = (uintptr_t)base;
        r.size = size;
    }
    return r;
}

bool capturing(cudaStream_t s)
{
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &st) != cudaSuccess) {
        cudaGetLastError();
        return true;
    }
    return st != cudaStreamCaptureStatusNone;
}

bool read_by_kernel(const float* h, const float* qx, const float* qy, size_t n, cudaStream_t s)
{
    const float* out[3] = {h, qx, qy};
    bool any = false;
    Allocation in;
    for (int i = 0; i < 3; ++i) {
        if (!out[i]) continue;
        any = true;
        if ((reinterpret_cast<uintptr_t>(out[i]) & 3) != 0) return false;
        // the whole array inside one allocation (a copy refuses an array that
        // is too short, a kernel would write past it)
        if (!in.holds(out[i], sizeof(float) * n)) in = allocation_of(out[i]);
        if (!in.holds(out[i], sizeof(float) * n)) return false;
        for (int j = 0; j < i; ++j)
            if (out[j] && out[i] < out[j] + n && out[j] < out[i] + n) return false;
    }
    return any && !capturing(s);
}

void launch_read_state(const float* state, size_t buffer, const MemberClock* clk, int ny, int nx, int ld, size_t plane,
                       float* h, float* qx, float* qy, int n_sm, cudaStream_t s)
{
    auto aligned = [](const float* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
    const bool vec = nx % 4 == 0 && aligned(h) && aligned(qx) && aligned(qy);
    const dim3 block(64, 4), grid(std::min((ny + 3) / 4, n_sm * 8), 3);
    if (vec)
        read_state_kernel<true><<<grid, block, 0, s>>>(state, buffer, clk, ny, nx, ld, plane, h, qx, qy);
    else
        read_state_kernel<false><<<grid, block, 0, s>>>(state, buffer, clk, ny, nx, ld, plane, h, qx, qy);
}

void launch_pack_members(const MemberClock* clk, const float* rain, const float* scale, const double* w, int M,
                         MemberRow* out, cudaStream_t s)
{
    pack_members_kernel<<<(M + 127) / 128, 128, 0, s>>>(clk, rain, scale, w, M, out);
}

void launch_batch_storage(const ScenDesc* desc, const MemberClock* ms, int S, int ny_max, double* part, double area,
                          double* out, cudaStream_t s)
{
    const int nb = (ny_max + kRows - 1) / kRows;
    for (int e0 = 0; e0 < S; e0 += 65535) {
        const int n = std::min(65535, S - e0);
        batch_storage_partial_kernel<<<dim3(nb, n), 256, 0, s>>>(desc, ms, e0, part + (size_t)e0 * nb, nb);
        batch_storage_final_kernel<<<(n + 127) / 128, 128, 0, s>>>(desc, part + (size_t)e0 * nb, e0, n, nb, area, out);
    }
}

}  // namespace flood
