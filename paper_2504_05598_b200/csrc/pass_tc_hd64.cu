// The kernels of pass_tc.cuh for head dimension 64.
#include "pass_tc.cuh"

cudaError_t pass_tc_prepare_hd64() { return pass::prepare_hd<64>(); }

cudaError_t launch_pass_tc_hd64(const PassTcMaps &maps, const PassTcArgs &w, int np, int grid, cudaStream_t st, bool pdl) {
    return pass::launch_hd<64>(maps, w, np, grid, st, pdl);
}
