// anchored_launch.cuh -- choice of the chunk-anchored node kernel: one baseline
// takes two nodes per packed value, more take 2, 4, 6 or 8 baselines at a time
// (beyond 8 the nodes are taken again).
#pragma once

#include <mutex>

#include "anchored.cuh"
#include "slices.cuh"

namespace gna {

template <int NP, bool GRAD>
size_t nodes_smem(int block) {
    return sizeof(f32x2p) * NP * (GRAD ? 6 : 3) * (size_t)block + (size_t)block / 32 * QuadRing<kRingMulti>::kWarpBytes;
}

constexpr size_t kNodesSmem = 72 * 1024;  // the most a block of 128 threads takes

inline size_t one_smem(int block) { return (size_t)block / 32 * QuadRing<kRingOne>::kWarpBytes; }

template <int PH, int NP, bool GRAD>
cudaError_t launch_multi(const BinArgs& a, int grid, int block, cudaStream_t s) {
    cudaError_t e = allow_smem<k_nodes_multi<PH, NP, GRAD>>(kNodesSmem);
    if (e != cudaSuccess) return e;
    return launch_dependent(k_nodes_multi<PH, NP, GRAD>, a, grid, block, s, nodes_smem<NP, GRAD>(block));
}

// Pairs of baselines taken at a time: up to four, the baselines spread evenly
// over the passes over the nodes that this takes.  GB300, twelve as 6 + 6
// instead of 8 + 4: 500 bins x 1000 nodes 43.8 -> 39.0 us, 127 x 67 41.0 -> 34.8.
inline int baseline_pairs(int nL) {
    const int passes = (nL + 7) / 8, per = (nL + passes - 1) / passes;
    return (per + 1) / 2;
}

template <int PH, bool GRAD>
cudaError_t launch_nodes_g(const BinArgs& a, int grid, int block, cudaStream_t s) {
    if (a.nL <= 1) return launch_dependent(k_nodes_one<PH, GRAD>, a, grid, block, s, one_smem(block));
    switch (baseline_pairs(a.nL)) {
        case 1: return launch_multi<PH, 1, GRAD>(a, grid, block, s);
        case 2: return launch_multi<PH, 2, GRAD>(a, grid, block, s);
        case 3: return launch_multi<PH, 3, GRAD>(a, grid, block, s);
        default: return launch_multi<PH, 4, GRAD>(a, grid, block, s);
    }
}

template <int PH>
cudaError_t launch_nodes(bool grad, const BinArgs& a, int grid, int block, cudaStream_t s) {
    return grad ? launch_nodes_g<PH, true>(a, grid, block, s) : launch_nodes_g<PH, false>(a, grid, block, s);
}

template <auto K>
int resident_of(int block, size_t smem) {
    int n = 0;
    if (allow_smem<K>(kNodesSmem) != cudaSuccess) return 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, K, block, smem) != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return n > 0 ? n : 1;
}

template <int PH, bool GRAD>
int resident_nodes_g(int nL, int block) {
    if (nL <= 1) return resident_of<k_nodes_one<PH, GRAD>>(block, one_smem(block));
    switch (baseline_pairs(nL)) {
        case 1: return resident_of<k_nodes_multi<PH, 1, GRAD>>(block, nodes_smem<1, GRAD>(block));
        case 2: return resident_of<k_nodes_multi<PH, 2, GRAD>>(block, nodes_smem<2, GRAD>(block));
        case 3: return resident_of<k_nodes_multi<PH, 3, GRAD>>(block, nodes_smem<3, GRAD>(block));
        default: return resident_of<k_nodes_multi<PH, 4, GRAD>>(block, nodes_smem<4, GRAD>(block));
    }
}

template <int PH>
int resident_nodes(int nL, bool grad, int block) {
    return grad ? resident_nodes_g<PH, true>(nL, block) : resident_nodes_g<PH, false>(nL, block);
}

}  // namespace gna
