// anchored_f64.cu -- the chunk-anchored node kernels with anchors reduced in double.
#include "anchored_launch.cuh"
namespace gna {
cudaError_t dispatch_nodes_ph1(bool grad, const BinArgs& a, int grid, int block, cudaStream_t s) {
    return launch_nodes<1>(grad, a, grid, block, s);
}
int nodes_resident_ctas_ph1(int nL, bool grad, int block) { return resident_nodes<1>(nL, grad, block); }
}  // namespace gna
