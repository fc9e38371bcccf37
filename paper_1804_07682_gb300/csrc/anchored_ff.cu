// anchored_ff.cu -- the chunk-anchored node kernels with anchors reduced in double-float.
#include "anchored_launch.cuh"
namespace gna {
cudaError_t dispatch_nodes_ph0(bool grad, const BinArgs& a, int grid, int block, cudaStream_t s) {
    return launch_nodes<0>(grad, a, grid, block, s);
}
int nodes_resident_ctas_ph0(int nL, bool grad, int block) { return resident_nodes<0>(nL, grad, block); }
}  // namespace gna
