// The kernels of pass_tc.cuh for head dimension 128.
#include "pass_tc.cuh"

cudaError_t pass_tc_prepare_hd128() { return pass::prepare_hd<128>(); }

cudaError_t launch_pass_tc_hd128(const PassTcMaps &maps, const PassTcArgs &w, int np, int grid, cudaStream_t st, bool pdl) {
    return pass::launch_hd<128>(maps, w, np, grid, st, pdl);
}
