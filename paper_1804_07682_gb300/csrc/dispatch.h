// dispatch.h -- host-side selection of the fused-kernel instantiation.
#pragma once
#include <cuda_runtime.h>

struct PointConst;

namespace gna {
// ph: 0 = double-float phase, 1 = double phase (both FP32 + Kahan bulk), 2 = all double.
// nl: instantiated baseline count (1, 2, 4, 8 or 16).  args points to
// SplitArgs (ph 0, 1) or SplitArgs64 (ph 2).
cudaError_t dispatch_split(int ph, int nl, bool grad, bool spec, const void* args, int grid, int block, cudaStream_t s);
// registers per thread of the split kernel (for occupancy-aware grid sizing)
int split_regs(int ph, int nl, bool grad, bool spec);
// second step of the slice mapping (slices.cu): S slices of NV values per
// (point, group) in part [npts][ngroups][S][NV][32]; pcs: the points' constants
struct EpiArgs;
cudaError_t launch_slices_reduce(const float2* part, int S, int NV, const EpiArgs& ea, const PointConst* pcs, int npts,
                                 cudaStream_t s);
// node kernel of the mixed precisions, bin and slice mappings (anchored.cuh);
// ph 0 or 1.  Threads per block are at most 128 (nodes_block).
struct BinArgs;
struct FitArgs;
cudaError_t dispatch_fit(int ph, int nl, const FitArgs& a, int grid, int block, cudaStream_t s);
cudaError_t launch_fit_slices_reduce(const float2* part, int S, const EpiArgs& ea, int npts, cudaStream_t s);
cudaError_t launch_point_sums(int npar, const EpiArgs& ea, cudaStream_t s);  // npar: 4 or 6
cudaError_t launch_cached_terms(const float2* sums, const EpiArgs& ea, cudaStream_t s);
cudaError_t dispatch_nodes(int ph, bool grad, const BinArgs& a, int grid, int block, cudaStream_t s);
int nodes_block(int block);
int nodes_resident_ctas(int ph, int nL, bool grad, int block);  // per SM
// epilogue only, on kept node sums [npts][nbins][ea.NV] (slices.cu)
cudaError_t launch_cached_epilogue(const double* sums, const EpiArgs& ea, cudaStream_t s);
}  // namespace gna
