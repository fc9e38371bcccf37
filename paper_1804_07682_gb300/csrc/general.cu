// general.cu -- the any-channel chain: per-point coefficients (step a0 for
// P(alpha -> beta)), the node and slice-reduction kernels of general.cuh and
// their launchers.
#include <algorithm>
#include <mutex>

#include "general.cuh"
#include "general_nodes.cuh"
#include "slices.cuh"

namespace gna {

// ------------------------------------------------------------ step a0 ----
// A real number with its derivative in one of (s2_12, s2_13, s2_23, delta):
// forward-mode differentiation of the written-out mixing matrix.
struct Dn {
    double v, d;
};

__device__ inline Dn dn_const(double v) { return Dn{v, 0.0}; }
__device__ inline Dn operator+(const Dn& a, const Dn& b) { return Dn{a.v + b.v, a.d + b.d}; }
__device__ inline Dn operator-(const Dn& a, const Dn& b) { return Dn{a.v - b.v, a.d - b.d}; }
__device__ inline Dn operator-(const Dn& a) { return dn_const(0.0) - a; }
__device__ inline Dn operator*(const Dn& a, const Dn& b) { return Dn{a.v * b.v, a.d * b.v + a.v * b.d}; }

// Complex number of such reals.
struct Cn {
    Dn re, im;
};
__device__ inline Cn cn(const Dn& re, const Dn& im) { return Cn{re, im}; }
__device__ inline Cn operator+(const Cn& a, const Cn& b) { return Cn{a.re + b.re, a.im + b.im}; }
__device__ inline Cn operator*(const Cn& a, const Cn& b) {
    return Cn{a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
__device__ inline Cn operator*(const Dn& a, const Cn& b) { return Cn{a * b.re, a * b.im}; }
__device__ inline Cn conjn(const Cn& a) { return Cn{a.re, -a.im}; }

// Sines and cosines of the mixing angles and e^{+-i delta}.
struct Angles {
    Dn s12, c12, s13, c13, s23, c23;
    Cn ep, em;
};

// Row `flavour` of the mixing matrix in the standard parameterisation (U = R23
// U13(delta) R12), written out element by element.
__device__ __forceinline__ void pmns_row(const Angles& t, int flavour, Cn (&U)[3]) {
    const Dn zero = dn_const(0.0);
    if (flavour == 0) {
        U[0] = cn(t.c12 * t.c13, zero);
        U[1] = cn(t.s12 * t.c13, zero);
        U[2] = t.s13 * t.em;
        return;
    }
    const Cn s13ep = t.s13 * t.ep;
    if (flavour == 1) {
        U[0] = cn(-(t.s12 * t.c23), zero) + (-(t.c12 * t.s23)) * s13ep;
        U[1] = cn(t.c12 * t.c23, zero) + (-(t.s12 * t.s23)) * s13ep;
        U[2] = cn(t.s23 * t.c13, zero);
    } else {
        U[0] = cn(t.s12 * t.s23, zero) + (-(t.c12 * t.c23)) * s13ep;
        U[1] = cn(-(t.c12 * t.s23), zero) + (-(t.s12 * t.c23)) * s13ep;
        U[2] = cn(t.c23 * t.c13, zero);
    }
}

__device__ __forceinline__ Cn pick(bool first, const Cn& a, const Cn& b) { return first ? a : b; }

// Sixteen threads per point, one per baseline slot for the phase constants (as
// for the survival chain).  The coefficients of P(alpha -> beta) --
// X_ij = U*_ai U_bi U_aj U*_bj for the pairs (21, 31, 32), a = -4 Re X,
// b = 4 Im X, and for antineutrinos (V = U*, so X -> X*) b -> -b -- are formed
// by twelve of them, thread 4 k + q the pair k and its derivative in parameter
// q, the roots and their reciprocals by six, one each.  A warp's FP64
// instruction takes its SM quarter's pipe for 64 cycles however many threads
// take part, so the number of instructions in the longest thread is the
// kernel's time: one thread with all four derivatives and nine matrix elements
// issued about 900.  GB300, whole evaluations: nu_mu disappearance at one point
// (400 bins x 513 nodes x 2) 42.6 -> 27 us, 1021 points of nu_mu -> nu_e 165 ->
// 132 us.  The first thread checks that the mixing parameters lie inside (0, 1)
// (the derivatives are singular on the boundary).  Zeroes the evaluation's
// counters.
__global__ void k_prepare_general(const gna_osc_full* __restrict__ prm, int npts, BaseConst bc, int alpha, int beta,
                                  int anti, PointConst* __restrict__ out, GenConst* __restrict__ gout,
                                  int* __restrict__ zero, int64_t nz, int* __restrict__ status) {
    asm volatile("griddepcontrol.launch_dependents;");
    // a programmatic dependent of the kernel before it: wait for it first
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t k = tid; k < nz; k += (int64_t)gridDim.x * blockDim.x) zero[k] = 0;
    static_assert(GNA_NLMAX == 16, "two points per warp");
    if (tid / 32 * 2 >= npts) return;  // the warp's first point: whole warps go on
    const int r = (int)(tid % GNA_NLMAX);
    const bool live = tid / GNA_NLMAX < npts;
    const int p = live ? (int)(tid / GNA_NLMAX) : npts - 1;
    const gna_osc_full o = prm[p];
    const double kl = (r < bc.nL) ? bc.kld[r] : 0.0;
    const double c21 = o.dm2_21 * kl, c32 = o.dm2_32 * kl;
    if (live) {
        PointConst& pc = out[p];
        pc.c21[r] = c21;
        pc.c32[r] = c32;
        split_ff(c21, pc.c21h[r], pc.c21l[r]);
        split_ff(c32, pc.c32h[r], pc.c32l[r]);
    }
    // roots of s2_12, 1 - s2_12, ... in threads 0 to 5, with 1 / (2 root):
    // d sin(theta) / d sin^2(theta) = 1 / (2 sin), d cos / d sin^2 = -1 / (2 cos)
    const double x2 = r < 2 ? o.s2_12 : r < 4 ? o.s2_13 : o.s2_23;
    const double root = sqrt((r & 1) ? 1.0 - x2 : x2), half = 0.5 / root;
    const int k = min(r >> 2, 2), q = r & 3;
    auto angle = [&](int j, int par, double sign) {
        const double v = __shfl_sync(0xffffffffu, root, j, 16), h = __shfl_sync(0xffffffffu, half, j, 16);
        return Dn{v, q == par ? sign * h : 0.0};
    };
    Angles t;
    t.s12 = angle(0, 0, 1.0);
    t.c12 = angle(1, 0, -1.0);
    t.s13 = angle(2, 1, 1.0);
    t.c13 = angle(3, 1, -1.0);
    t.s23 = angle(4, 2, 1.0);
    t.c23 = angle(5, 2, -1.0);
    if (!live) return;
    double sd, cd;
    sincos(o.delta_cp, &sd, &cd);
    const Dn cosd{cd, q == 3 ? -sd : 0.0}, sind{sd, q == 3 ? cd : 0.0};
    t.ep = cn(cosd, sind);
    t.em = cn(cosd, -sind);
    Cn Ua[3], Ub[3];
    pmns_row(t, alpha, Ua);
    pmns_row(t, beta, Ub);
    const bool i1 = k == 0, j0 = k != 2;  // (i, j) = (1, 0), (2, 0), (2, 1)
    const Cn X = conjn(pick(i1, Ua[1], Ua[2])) * pick(i1, Ub[1], Ub[2]) * pick(j0, Ua[0], Ua[1]) *
                 conjn(pick(j0, Ub[0], Ub[1]));
    const double sb = anti ? -4.0 : 4.0;
    GenConst& gc = gout[p];
    if (r < 12) {
        const double da = -4.0 * X.re.d, db = sb * X.im.d;
        gc.da[q][k] = da;
        gc.db[q][k] = db;
        gc.daf[q][k] = (float)da;
        gc.dbf[q][k] = (float)db;
        if (q == 0) {
            const double a = -4.0 * X.re.v, b = sb * X.im.v;
            const float af = (float)a, bf = (float)b;
            gc.a[k] = a;
            gc.b[k] = b;
            gc.af[k] = af;
            gc.bf[k] = bf;
            gc.alo[k] = (float)(a - (double)af);
            gc.blo[k] = (float)(b - (double)bf);
        }
    }
    if (r != 0) return;
    out[p].cmax = largest_phase(bc, o.dm2_21, o.dm2_32);
    gc.dab = (alpha == beta) ? 1.0 : 0.0;
    gc.wsum = bc.wsum_pair;
    const bool inside = o.s2_12 > 0.0 && o.s2_12 < 1.0 && o.s2_13 > 0.0 && o.s2_13 < 1.0 && o.s2_23 > 0.0 &&
                        o.s2_23 < 1.0 && isfinite(o.delta_cp) && isfinite(o.dm2_21) && isfinite(o.dm2_32);
    if (!inside && status) atomicExch(status, (int)GNA_EINVAL);
}

cudaError_t launch_prepare_general(const gna_osc_full* prm, int npts, const BaseConst& bc, int alpha, int beta,
                                   int anti, PointConst* out, GenConst* gout, int* zero, int64_t nz, int* status,
                                   cudaStream_t s) {
    const int64_t threads = std::max<int64_t>((int64_t)npts * GNA_NLMAX, std::min<int64_t>(nz, 1LL << 20));
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)((threads + 255) / 256));
    cfg.blockDim = dim3(256);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_prepare_general, prm, npts, bc, alpha, beta, anti, out, gout, zero, nz, status);
}

// ------------------------------------------------------------ launchers ----
// Fits.
template <int PH, int NL>
static cudaError_t launch_gen_fit(bool surv, const GenArgs& a, int grid, int block, cudaStream_t s) {
    return surv ? launch_dependent(k_fit_bins_gen<PH, NL, true>, a, grid, block, s)
                : launch_dependent(k_fit_bins_gen<PH, NL, false>, a, grid, block, s);
}

template <int PH>
static cudaError_t dispatch_gen_fit(int nl, bool surv, const GenArgs& a, int grid, int block, cudaStream_t s) {
    switch (nl) {
        case 1: return launch_gen_fit<PH, 1>(surv, a, grid, block, s);
        case 2: return launch_gen_fit<PH, 2>(surv, a, grid, block, s);
        case 4: return launch_gen_fit<PH, 4>(surv, a, grid, block, s);
        case 8: return launch_gen_fit<PH, 8>(surv, a, grid, block, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t dispatch_general_fit(int ph, int nl, bool surv, const GenArgs& a, int grid, int block, cudaStream_t s) {
    return ph == 0 ? dispatch_gen_fit<0>(nl, surv, a, grid, block, s) : dispatch_gen_fit<1>(nl, surv, a, grid, block, s);
}

template <typename Kernel>
static int occupancy(Kernel k, int block) {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, block, 0) != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return n > 0 ? n : 1;
}

template <int PH>
static int fit_ctas(int nl, bool surv, int block) {
    switch (nl) {
        case 1: return surv ? occupancy(k_fit_bins_gen<PH, 1, true>, block) : occupancy(k_fit_bins_gen<PH, 1, false>, block);
        case 2: return surv ? occupancy(k_fit_bins_gen<PH, 2, true>, block) : occupancy(k_fit_bins_gen<PH, 2, false>, block);
        case 4: return surv ? occupancy(k_fit_bins_gen<PH, 4, true>, block) : occupancy(k_fit_bins_gen<PH, 4, false>, block);
        case 8: return surv ? occupancy(k_fit_bins_gen<PH, 8, true>, block) : occupancy(k_fit_bins_gen<PH, 8, false>, block);
        default: return 1;
    }
}
int general_fit_ctas(int ph, int nl, bool surv, int block) {
    return ph == 0 ? fit_ctas<0>(nl, surv, block) : fit_ctas<1>(nl, surv, block);
}

// Evaluations: one baseline takes two nodes per packed value, more take two or
// four baselines at a time.
constexpr size_t kGenSmem = 72 * 1024;  // the most a block of 128 threads takes
template <int NP, bool GRAD>
static size_t gen_smem(int block) {
    return sizeof(f32x2p) * NP * gen_sums(GRAD) * (size_t)block + (size_t)block / 32 * QuadRing<kRingMulti>::kWarpBytes;
}
static size_t gen_one_smem(int block) { return (size_t)block / 32 * QuadRing<kRingOne>::kWarpBytes; }

template <int PH, int NP, bool GRAD>
static cudaError_t launch_gen_multi(const GenArgs& a, int grid, int block, cudaStream_t s) {
    cudaError_t e = allow_smem<k_gen_multi<PH, NP, GRAD>>(kGenSmem);
    if (e != cudaSuccess) return e;
    return launch_dependent(k_gen_multi<PH, NP, GRAD>, a, grid, block, s, gen_smem<NP, GRAD>(block));
}

template <int PH, bool GRAD>
static cudaError_t launch_gen(const GenArgs& a, int grid, int block, cudaStream_t s) {
    if (a.b.nL <= 1) return launch_dependent(k_gen_one<PH, GRAD>, a, grid, block, s, gen_one_smem(block));
    if (a.b.nL <= 2) return launch_gen_multi<PH, 1, GRAD>(a, grid, block, s);
    return launch_gen_multi<PH, 2, GRAD>(a, grid, block, s);
}

cudaError_t dispatch_general(int ph, bool grad, const GenArgs& a, int grid, int block, cudaStream_t s) {
    if (ph == 0) return grad ? launch_gen<0, true>(a, grid, block, s) : launch_gen<0, false>(a, grid, block, s);
    if (ph == 1) return grad ? launch_gen<1, true>(a, grid, block, s) : launch_gen<1, false>(a, grid, block, s);
    return cudaErrorInvalidValue;
}

template <auto K>
static int resident_of(int block, size_t smem) {
    int n = 0;
    if (allow_smem<K>(kGenSmem) != cudaSuccess) return 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, K, block, smem) != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return n > 0 ? n : 1;
}
template <int PH, bool GRAD>
static int resident_gen(int nL, int block) {
    if (nL <= 1) return resident_of<k_gen_one<PH, GRAD>>(block, gen_one_smem(block));
    if (nL <= 2) return resident_of<k_gen_multi<PH, 1, GRAD>>(block, gen_smem<1, GRAD>(block));
    return resident_of<k_gen_multi<PH, 2, GRAD>>(block, gen_smem<2, GRAD>(block));
}

int general_fit_ctas64(int nl, int block) {
    switch (nl) {
        case 1: return occupancy(k_fit64_bins_gen<1>, block);
        case 2: return occupancy(k_fit64_bins_gen<2>, block);
        case 4: return occupancy(k_fit64_bins_gen<4>, block);
        case 8: return occupancy(k_fit64_bins_gen<8>, block);
        default: return 1;
    }
}

int general_resident_ctas(int ph, int nL, bool grad, int block) {
    if (ph == 0) return grad ? resident_gen<0, true>(nL, block) : resident_gen<0, false>(nL, block);
    return grad ? resident_gen<1, true>(nL, block) : resident_gen<1, false>(nL, block);
}

template <int NL>
static cudaError_t launch_gen_fit64(const GenArgs64& a, int grid, int block, cudaStream_t s) {
    k_fit64_bins_gen<NL><<<grid, block, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t dispatch_general_fit64(int nl, const GenArgs64& a, int grid, int block, cudaStream_t s) {
    switch (nl) {
        case 1: return launch_gen_fit64<1>(a, grid, block, s);
        case 2: return launch_gen_fit64<2>(a, grid, block, s);
        case 4: return launch_gen_fit64<4>(a, grid, block, s);
        case 8: return launch_gen_fit64<8>(a, grid, block, s);
        default: return cudaErrorInvalidValue;
    }
}

template <int NVM, int W>
static cudaError_t launch_gen_reduce(const float2* part, int S, int NV, const EpiArgs& ea, const GenConst* gc, int npts,
                                     cudaStream_t s) {
    cudaError_t e = allow_smem<k_gen_slices_reduce<NVM, W>>(sizeof(float2) * (W + 1) * NVM * 32);
    if (e != cudaSuccess) return e;
    return launch_blocks(k_gen_slices_reduce<NVM, W>, (int64_t)npts * ea.ngroups, W * 32,
                         sizeof(float2) * (W + 1) * NV * 32, s, part, S, NV, ea, gc);
}

cudaError_t launch_slices_reduce_general(const float2* part, int S, int NV, const EpiArgs& ea, const GenConst* gc,
                                         int npts, cudaStream_t s) {
    if (NV == gen_sums(false)) return launch_gen_reduce<6, 32>(part, S, NV, ea, gc, npts, s);
    if (NV == gen_sums(true)) return launch_gen_reduce<12, 24>(part, S, NV, ea, gc, npts, s);
    return cudaErrorInvalidValue;
}

cudaError_t launch_fit_slices_reduce_general(const float2* part, int S, const EpiArgs& ea, const GenConst* gc, int npts,
                                             cudaStream_t s) {
    constexpr int W = 24, NV = gen_nv(true);
    constexpr size_t smem = sizeof(float2) * W * NV * 32 + sizeof(double) * NV * 32;
    cudaError_t e = allow_smem<k_fit_slices_reduce_gen<W>>(smem);
    if (e != cudaSuccess) return e;
    return launch_blocks(k_fit_slices_reduce_gen<W>, (int64_t)npts * ea.ngroups, W * 32, smem, s, part, S, NV, ea, gc);
}

}  // namespace gna
