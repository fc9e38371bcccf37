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
// A real number with its derivatives in (s2_12, s2_13, s2_23, delta):
// forward-mode differentiation of the written-out mixing matrix.
struct Dn {
    double v, d[4];
};

__device__ inline Dn dn_const(double v) {
    Dn x;
    x.v = v;
    for (int q = 0; q < 4; q++) x.d[q] = 0.0;
    return x;
}
__device__ inline Dn dn_var(double v, int q, double dq) {
    Dn x = dn_const(v);
    x.d[q] = dq;
    return x;
}
__device__ inline Dn operator+(const Dn& a, const Dn& b) {
    Dn x;
    x.v = a.v + b.v;
    for (int q = 0; q < 4; q++) x.d[q] = a.d[q] + b.d[q];
    return x;
}
__device__ inline Dn operator-(const Dn& a, const Dn& b) {
    Dn x;
    x.v = a.v - b.v;
    for (int q = 0; q < 4; q++) x.d[q] = a.d[q] - b.d[q];
    return x;
}
__device__ inline Dn operator-(const Dn& a) { return dn_const(0.0) - a; }
__device__ inline Dn operator*(const Dn& a, const Dn& b) {
    Dn x;
    x.v = a.v * b.v;
    for (int q = 0; q < 4; q++) x.d[q] = a.d[q] * b.v + a.v * b.d[q];
    return x;
}

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

// Coefficients of P(alpha -> beta) at one point: the mixing matrix in the
// standard parameterisation written out element by element (U = R23
// U13(delta) R12), X_ij = U*_ai U_bi U_aj U*_bj for the pairs (21, 31, 32),
// a = -4 Re X, b = 4 Im X, and for antineutrinos (V = U*, so X -> X*) b -> -b.
__device__ void general_coefficients(const gna_osc_full& o, int alpha, int beta, int anti, GenConst& gc) {
    const double s12v = sqrt(o.s2_12), c12v = sqrt(1.0 - o.s2_12);
    const double s13v = sqrt(o.s2_13), c13v = sqrt(1.0 - o.s2_13);
    const double s23v = sqrt(o.s2_23), c23v = sqrt(1.0 - o.s2_23);
    // d sin(theta) / d sin^2(theta) = 1 / (2 sin), d cos / d sin^2 = -1 / (2 cos)
    const Dn s12 = dn_var(s12v, 0, 0.5 / s12v), c12 = dn_var(c12v, 0, -0.5 / c12v);
    const Dn s13 = dn_var(s13v, 1, 0.5 / s13v), c13 = dn_var(c13v, 1, -0.5 / c13v);
    const Dn s23 = dn_var(s23v, 2, 0.5 / s23v), c23 = dn_var(c23v, 2, -0.5 / c23v);
    double sd, cd;
    sincos(o.delta_cp, &sd, &cd);
    const Dn cosd = dn_var(cd, 3, -sd), sind = dn_var(sd, 3, cd);
    const Cn ep = cn(cosd, sind);   // e^{+i delta}
    const Cn em = cn(cosd, -sind);  // e^{-i delta}
    const Dn zero = dn_const(0.0);
    const Cn s13ep = s13 * ep;
    Cn U[3][3];
    U[0][0] = cn(c12 * c13, zero);
    U[0][1] = cn(s12 * c13, zero);
    U[0][2] = s13 * em;
    U[1][0] = cn(-(s12 * c23), zero) + (-(c12 * s23)) * s13ep;
    U[1][1] = cn(c12 * c23, zero) + (-(s12 * s23)) * s13ep;
    U[1][2] = cn(s23 * c13, zero);
    U[2][0] = cn(s12 * s23, zero) + (-(c12 * c23)) * s13ep;
    U[2][1] = cn(-(c12 * s23), zero) + (-(s12 * c23)) * s13ep;
    U[2][2] = cn(c23 * c13, zero);
    const int pi_[3] = {1, 2, 2}, pj_[3] = {0, 0, 1};
    gc.dab = (alpha == beta) ? 1.0 : 0.0;
    for (int k = 0; k < 3; k++) {
        const int i = pi_[k], j = pj_[k];
        const Cn X = conjn(U[alpha][i]) * U[beta][i] * U[alpha][j] * conjn(U[beta][j]);
        const double sb = anti ? -4.0 : 4.0;
        gc.a[k] = -4.0 * X.re.v;
        gc.b[k] = sb * X.im.v;
        gc.af[k] = (float)gc.a[k];
        gc.bf[k] = (float)gc.b[k];
        gc.alo[k] = (float)(gc.a[k] - (double)gc.af[k]);
        gc.blo[k] = (float)(gc.b[k] - (double)gc.bf[k]);
        for (int q = 0; q < 4; q++) {
            gc.da[q][k] = -4.0 * X.re.d[q];
            gc.db[q][k] = sb * X.im.d[q];
            gc.daf[q][k] = (float)gc.da[q][k];
            gc.dbf[q][k] = (float)gc.db[q][k];
        }
    }
}

// One thread per (point, baseline slot): the phase constants as for the
// survival chain; the point's first thread also forms its coefficients and
// checks that the mixing parameters lie inside (0, 1) (the derivatives are
// singular on the boundary).  Zeroes the evaluation's counters.
__global__ void k_prepare_general(const gna_osc_full* __restrict__ prm, int npts, BaseConst bc, int alpha, int beta,
                                  int anti, PointConst* __restrict__ out, GenConst* __restrict__ gout,
                                  int* __restrict__ zero, int64_t nz, int* __restrict__ status) {
    asm volatile("griddepcontrol.launch_dependents;");
    // a programmatic dependent of the kernel before it: wait for it first
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t k = tid; k < nz; k += (int64_t)gridDim.x * blockDim.x) zero[k] = 0;
    const int p = (int)(tid / GNA_NLMAX), r = (int)(tid % GNA_NLMAX);
    if (p >= npts) return;
    const gna_osc_full o = prm[p];
    PointConst& pc = out[p];
    const double kl = (r < bc.nL) ? bc.kld[r] : 0.0;
    const double c21 = o.dm2_21 * kl, c32 = o.dm2_32 * kl;
    pc.c21[r] = c21;
    pc.c32[r] = c32;
    split_ff(c21, pc.c21h[r], pc.c21l[r]);
    split_ff(c32, pc.c32h[r], pc.c32l[r]);
    if (r != 0) return;
    pc.cmax = largest_phase(bc, o.dm2_21, o.dm2_32);
    const bool inside = o.s2_12 > 0.0 && o.s2_12 < 1.0 && o.s2_13 > 0.0 && o.s2_13 < 1.0 && o.s2_23 > 0.0 &&
                        o.s2_23 < 1.0 && isfinite(o.delta_cp) && isfinite(o.dm2_21) && isfinite(o.dm2_32);
    if (!inside && status) atomicExch(status, (int)GNA_EINVAL);
    general_coefficients(o, alpha, beta, anti, gout[p]);
    double w = 0.0;
    for (int q = 0; q < bc.nL; q++) w += (double)bc.om[q] + (double)bc.omlo[q];
    gout[p].wsum = w;
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
