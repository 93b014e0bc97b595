// Steps of ensembles that stay on the chip (step_resident.cu).
#pragma once

#include "flood_internal.cuh"

namespace flood {

struct ResidentShape {
    int bands;    // CTAs of a member (0: the state does not fit)
    int rows;     // rows of a band (the last may have fewer)
    size_t smem;  // dynamic shared memory of a CTA
};

struct ResidentArgs {
    StepArgs a;                 // ms_in: the clocks before the first step (plan, ms_out, ms_clr unused)
    MemberClock* ms_end;        // clock slot after the last step
    MemberClock* ms_next;       // the slot after that one
    unsigned long long* words;  // [2][M][bands] step number and maximum depth of a band
    unsigned long long* xch;    // [2][M][bands][2][ld] first and last row of a band's depths,
                                // each with the step number above it
    uint32_t* seq;              // [M] step numbers already used
    int bands, rows, n_steps;
};

ResidentShape resident_shape(int ny, int nx, int M, int n_sm, size_t smem_max, bool track, bool lc);
cudaError_t launch_resident(const ResidentArgs& t, const ResidentShape& sh, cudaStream_t s);

}  // namespace flood
