// The Yee update of one step as a kernel of its own (yee.cuh): after every push that is
// not followed by one fused with it.  (A version
// without shared memory and barriers, each thread recomputing the half-step B and
// new E it shares with its neighbours from global loads, ran at half the speed.)
#include "yee.cuh"

namespace picrr {

namespace {

template <bool PDL>
__global__ void __launch_bounds__(FIELD_T) k_field(const FieldParams P) {
    __shared__ FieldSmem S;
    pdl_release<PDL>();
    field_block<FIELD_T, PDL>(P, *P.phase + P.k, blockIdx.x, S);
}

__global__ void __launch_bounds__(FIELD_T) k_zero_current(const FieldParams P) {
    const RunDev& R = P.runs[P.blk_run[blockIdx.x]];
    if (!R.active) return;
    const int i0 = P.blk_i0[blockIdx.x];
    for (int p = i0 + threadIdx.x; p < min(i0 + FIELD_NODES + 2 * PADF, R.glen); p += FIELD_T)
        for (int set = 0; set < 3; ++set) R.J[set][0][p] = R.J[set][1][p] = R.J[set][2][p] = 0ull;
}

}  // namespace

// Zeroes every current set of the active runs.
void launch_zero_current(const FieldParams& P, cudaStream_t st) {
    if (P.nblk > 0) k_zero_current<<<P.nblk, FIELD_T, 0, st>>>(P);
}

void launch_field(const FieldParams& P, int grid, cudaStream_t st, bool pdl) {
    if (grid > 0) launch(pdl ? k_field<true> : k_field<false>, dim3(grid), FIELD_T, st, pdl, P);
}

}  // namespace picrr
