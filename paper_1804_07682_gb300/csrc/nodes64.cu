// nodes64.cu -- launchers of the double-precision node kernel (nodes64.cuh).
#include "nodes64.cuh"

#include <mutex>

#include "slices.cuh"

namespace gna {

cudaError_t launch_nodes64(bool gen, bool grad, const Args64& a, int grid, int block, cudaStream_t s) {
    if (gen)
        return grad ? launch_dependent(k_nodes64<true, true>, a, grid, block, s)
                    : launch_dependent(k_nodes64<true, false>, a, grid, block, s);
    return grad ? launch_dependent(k_nodes64<false, true>, a, grid, block, s)
                : launch_dependent(k_nodes64<false, false>, a, grid, block, s);
}

template <bool GEN, bool GRAD>
static cudaError_t launch_reduce64(const double* part, int S, int NV, const EpiArgs& ea, const PointConst* pcs,
                                   const GenConst* gc, int npts, cudaStream_t s) {
    constexpr int W = 16;
    constexpr int most = sums64(GEN, GRAD) + (GEN ? 0 : GNA_NLMAX);
    cudaError_t e = allow_smem<k_slices_reduce64<GEN, GRAD, W>>(sizeof(double) * W * most * 32);
    if (e != cudaSuccess) return e;
    return launch_blocks(k_slices_reduce64<GEN, GRAD, W>, (int64_t)npts * ea.ngroups, W * 32,
                         sizeof(double) * W * NV * 32, s, part, S, NV, ea, pcs, gc);
}

cudaError_t launch_slices_reduce64(bool gen, bool grad, const double* part, int S, int NV, const EpiArgs& ea,
                                   const PointConst* pcs, const GenConst* gc, int npts, cudaStream_t s) {
    if (gen)
        return grad ? launch_reduce64<true, true>(part, S, NV, ea, pcs, gc, npts, s)
                    : launch_reduce64<true, false>(part, S, NV, ea, pcs, gc, npts, s);
    return grad ? launch_reduce64<false, true>(part, S, NV, ea, pcs, gc, npts, s)
                : launch_reduce64<false, false>(part, S, NV, ea, pcs, gc, npts, s);
}

}  // namespace gna
