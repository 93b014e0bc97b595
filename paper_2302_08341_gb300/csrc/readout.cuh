// Launchers that read results out (readout.cu).
#pragma once

#include <algorithm>

#include "batch.cuh"

namespace flood {

// Ordinary host memory, which a copy on any stream has read or written by the
// time it returns.
bool pageable(const void* p);
// The stream records a graph (or cannot say): such calls keep to plain copies.
bool capturing(cudaStream_t s);
// The outputs that are not null are distinct arrays of n floats in memory of
// the current device, so that launch_read_state may write them.
bool read_by_kernel(const float* h, const float* qx, const float* qy, size_t n, cudaStream_t s);

// One member's scalars, as flood_get_members returns them.
struct MemberRow {
    double t;
    int64_t steps;
    double w;
    float rain, scale, hmax, pad;
};

// The current state (state + clk->cur * buffer: h, qx, qy planes of [ny][ld])
// into device arrays [ny][nx]; any may be null.
void launch_read_state(const float* state, size_t buffer, const MemberClock* clk, int ny, int nx, int ld, size_t plane,
                       float* h, float* qx, float* qy, int n_sm, cudaStream_t s);
void launch_pack_members(const MemberClock* clk, const float* rain, const float* scale, const double* w, int M,
                         MemberRow* out, cudaStream_t s);
// Stored volume (FP64, times area) of every entry of a batch into out [S].
// part: S * ceil(ny_max / 16) doubles.
void launch_batch_storage(const ScenDesc* desc, const MemberClock* ms, int S, int ny_max, double* part, double area,
                          double* out, cudaStream_t s);

}  // namespace flood
