// slices.cu -- second step of the slice mapping: for each (point, group of
// 32 bins) the slices' values are summed in slice order (double-float, so the
// result does not depend on which warp computed which slice), then the bin
// epilogue runs for the group's bins and the group and point reductions
// follow (steps a7-a9 of the chain).
#include <mutex>

#include "anchored.cuh"
#include "dispatch.h"
#include "epilogue.cuh"
#include "slices.cuh"

namespace gna {

// One block of W warps per (point, group); warp 0 runs the epilogue of the
// group: 32 warps for up to 6 values, 24 for up to 14, 16 beyond.
template <int NVM, int W>
__global__ void __launch_bounds__(W * 32) k_slices_reduce(const float2* __restrict__ part, int S, int NV, EpiArgs ea,
                                                          const PointConst* __restrict__ pcs) {
    const int p = blockIdx.x / ea.ngroups, g = blockIdx.x - p * ea.ngroups;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // the epilogue's inputs do not depend on the node kernel: load them first
    const int i = g * 32 + lane;
    BinInput in;
    if (w == 0) in = bin_input(ea, p, min(i, ea.nbins - 1));
    // (and the point's constants, written before the node kernel began)
    if (w == 0 && lane < (int)(sizeof(PointConst) + 127) / 128)
        asm volatile("prefetch.global.L1 [%0];" ::"l"(reinterpret_cast<const char*>(pcs + p) + lane * 128));
    const float2* fin = sum_slices<NVM, W>(part, S, NV, w, lane);
    if (w == 0) {
        // the task sums T, N (anchored.cuh), then the per-baseline parts
        TaskSums q;
        float2 sp[GNA_NLMAX];
        for (int j = 0; j < 3; j++) q.T[j] = fin[j * 32 + lane];
        const int from = ea.has_grad ? 6 : 3;
        for (int r = 0; r < ea.nspec; r++) sp[r] = fin[(from + r) * 32 + lane];
        if (ea.has_grad) {
            for (int j = 0; j < 3; j++) q.N[j] = fin[(3 + j) * 32 + lane];
            float2 regs[5];
            if (i < ea.nbins) bin_terms<4>(ea, p, i, bin_sums<true>(pcs + p, in.sumw, q), sp, in, regs);
            group_done_terms<4>(ea, p, g, lane, regs);
        } else {
            float2 regs[1];
            if (i < ea.nbins) bin_terms<0>(ea, p, i, bin_sums<false>(pcs + p, in.sumw, q), sp, in, regs);
            group_done_terms<0>(ea, p, g, lane, regs);
        }
    }
}

template <int NVM, int W>
cudaError_t launch_reduce(const float2* part, int S, int NV, const EpiArgs& ea, const PointConst* pcs, int npts,
                          cudaStream_t s) {
    cudaError_t e = allow_smem<k_slices_reduce<NVM, W>>(sizeof(float2) * (W + 1) * NVM * 32);
    if (e != cudaSuccess) return e;
    return launch_blocks(k_slices_reduce<NVM, W>, (int64_t)npts * ea.ngroups, W * 32, sizeof(float2) * (W + 1) * NV * 32, s,
                         part, S, NV, ea, pcs);
}

cudaError_t launch_slices_reduce(const float2* part, int S, int NV, const EpiArgs& ea, const PointConst* pcs, int npts,
                                 cudaStream_t s) {
    if (NV < 1 || NV > 6 + GNA_NLMAX) return cudaErrorInvalidValue;
    if (NV <= 6) return launch_reduce<6, 32>(part, S, NV, ea, pcs, npts, s);
    if (NV <= 14) return launch_reduce<14, 24>(part, S, NV, ea, pcs, npts, s);
    return launch_reduce<6 + GNA_NLMAX, 16>(part, S, NV, ea, pcs, npts, s);
}

// The fits' slice sums (FitArgs: the five values of fused.cuh).
__global__ void __launch_bounds__(32 * 32) k_fit_slices_reduce(const float2* __restrict__ part, int S, int NV, EpiArgs ea) {
    constexpr int NVM = 5, W = 32;
    extern __shared__ float2 red[];  // [W][NV][32], then [NV][32] doubles
    double* fin = reinterpret_cast<double*>(red + W * NV * 32);
    const int pg = blockIdx.x;
    const int p = pg / ea.ngroups;
    const int g = pg - p * ea.ngroups;
    const int w = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    // the next evaluation's first kernel may be placed now; it waits for this
    // kernel to complete before it touches anything
    asm volatile("griddepcontrol.launch_dependents;");
    float2 acc[NVM];
#pragma unroll
    for (int v = 0; v < NVM; v++) acc[v] = make_float2(0.f, 0.f);
    // the epilogue's inputs do not depend on the node kernel: load them first
    const int i = g * 32 + lane;
    BinIn in{0.0, 0.0, 0.0};
    if (w == 0 && i < ea.nbins) in = bin_inputs(ea, p, i);
    // launched as a programmatic dependent of the node kernel: the blocks may
    // be resident before it ends; wait (in hardware) until it has completed
    // and its writes are visible
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const float2* base = part + (int64_t)pg * S * NV * 32 + lane;
    const int64_t stride = (int64_t)NV * 32;
    for (int sl = w; sl < S; sl += W) {
        const float2* src = base + sl * stride;
        float2 t[NVM];
#pragma unroll
        for (int v = 0; v < NVM; v++) t[v] = (v < NV) ? __ldg(src + v * 32) : make_float2(0.f, 0.f);
#pragma unroll
        for (int v = 0; v < NVM; v++)
            if (v < NV) acc[v] = ff_add(acc[v], t[v]);
    }
#pragma unroll
    for (int v = 0; v < NVM; v++)
        if (v < NV) red[(w * NV + v) * 32 + lane] = acc[v];
    __syncthreads();
    for (int v = w; v < NV; v += W) {
        float2 sum = red[v * 32 + lane];
        for (int k = 1; k < W; k++) sum = ff_add(sum, red[(k * NV + v) * 32 + lane]);
        fin[v * 32 + lane] = (double)sum.x + (double)sum.y;
    }
    __syncthreads();
    if (w == 0) {
        double vals[kMaxNV];
        for (int v = 0; v < NV; v++) vals[v] = fin[v * 32 + lane];
        float2 regs[15];  // this lane's per-bin values: the warp reduces its own group
        if (i < ea.nbins) bin_epilogue(ea, p, i, vals, in, regs);
        group_done(ea, p, g, lane, regs);
    }
}

cudaError_t launch_fit_slices_reduce(const float2* part, int S, const EpiArgs& ea, int npts, cudaStream_t s) {
    constexpr int NV = 5, W = 32;
    constexpr size_t smem = sizeof(float2) * W * NV * 32 + sizeof(double) * NV * 32;
    cudaError_t e = allow_smem<k_fit_slices_reduce>(smem);
    if (e != cudaSuccess) return e;
    return launch_blocks(k_fit_slices_reduce, (int64_t)npts * ea.ngroups, W * 32, smem, s, part, S, NV, ea);
}

// After whole-bin tasks of the anchored kernels: one warp per point sums its
// groups and writes its outputs.
template <int NG>
__global__ void __launch_bounds__(256) k_point_sums(EpiArgs ea) {
    asm volatile("griddepcontrol.launch_dependents;");
    const int p = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (p < ea.npts) point_reduce<8, NG>(ea, p, threadIdx.x & 31);
}

cudaError_t launch_point_sums(int npar, const EpiArgs& ea, cudaStream_t s) {
    return launch_blocks(npar == 6 ? k_point_sums<6> : k_point_sums<4>, ((int64_t)ea.npts * 32 + 255) / 256, 256, 0, s, ea);
}

// Epilogue-only evaluation (steps a7-a9) on the node sums an evaluation in
// the anchored kernels kept (as k_cached_epilogue below).
template <int NG>
__global__ void __launch_bounds__(256) k_cached_terms(const float2* __restrict__ sums, EpiArgs ea) {
    const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (wid >= (int64_t)ea.npts * ea.ngroups) return;
    const int p = (int)(wid / ea.ngroups);
    const int g = (int)(wid - (int64_t)p * ea.ngroups);
    const int i = g * 32 + lane;
    float2 regs[1 + NG];
    if (i < ea.nbins) {
        const float2* src = sums + ((int64_t)p * ea.nbins + i) * ea.NV;
        BinSums<NG> b;
        b.M = src[0];
#pragma unroll
        for (int q = 0; q < NG; q += 2) {
            b.d[q] = src[1 + q / 2].x;
            b.d[q + 1] = src[1 + q / 2].y;
        }
        bin_terms<NG>(ea, p, i, b, src + 1 + NG / 2, bin_input(ea, p, i), regs);
    }
    group_done_terms<NG>(ea, p, g, lane, regs);
}

cudaError_t launch_cached_terms(const float2* sums, const EpiArgs& ea, cudaStream_t s) {
    const unsigned blocks = (unsigned)(((int64_t)ea.npts * ea.ngroups * 32 + 255) / 256);
    if (ea.has_grad) k_cached_terms<4><<<blocks, 256, 0, s>>>(sums, ea);
    else k_cached_terms<0><<<blocks, 256, 0, s>>>(sums, ea);
    return cudaGetLastError();
}

// Epilogue-only evaluation (steps a7-a9) on the node sums a previous
// evaluation kept: one warp per (point, group of 32 bins), lane l bin 32 g + l.
__global__ void __launch_bounds__(256) k_cached_epilogue(const double* __restrict__ sums, EpiArgs ea) {
    const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (wid >= (int64_t)ea.npts * ea.ngroups) return;
    const int p = (int)(wid / ea.ngroups);
    const int g = (int)(wid - (int64_t)p * ea.ngroups);
    const int i = g * 32 + lane;
    float2 regs[15];
    if (i < ea.nbins) {
        double v[kMaxNV];
        const double* src = sums + ((int64_t)p * ea.nbins + i) * ea.NV;
        for (int j = 0; j < ea.NV; j++) v[j] = src[j];
        bin_epilogue(ea, p, i, v, bin_inputs(ea, p, i), regs);
    }
    group_done(ea, p, g, lane, regs);
}

cudaError_t launch_cached_epilogue(const double* sums, const EpiArgs& ea, cudaStream_t s) {
    const int64_t threads = (int64_t)ea.npts * ea.ngroups * 32;
    k_cached_epilogue<<<(unsigned)((threads + 255) / 256), 256, 0, s>>>(sums, ea);
    return cudaGetLastError();
}

}  // namespace gna
