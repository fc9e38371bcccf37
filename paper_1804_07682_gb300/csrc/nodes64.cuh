// nodes64.cuh -- GNA_FP64: node kernel of both chains with every step in
// double (the fits and the forced split mapping keep fused64.cuh, general.cuh).
//
// What bounds it: the FP64 pipe (two FMAs per clock and SM: a warp-wide
// instruction holds an SM quarter's pipe for 64 cycles).  Reducing two phases
// and taking their sincos per (node, baseline) costs about 90 FP64
// instructions.  Here a lane walks its bin's nodes in chunks (anchored.cuh):
// the doubled phase of the chunk's middle node is formed exactly (FMA
// residual), reduced and given to sincos once, and a node contributes through
// its small offset t = 2c (1/E - 1/E_anchor),
//   sin t and cos t - 1 by their Taylor polynomials, of pairs 21 and 32, the
//   third pair by the addition formulas,
// summed with the weights W and W/E; the anchor's rotation is applied to the
// chunk's sums.  Two lengths of polynomial: |t| <= 2^-6 (terms to t^5, t^6;
// the next ones are below 5e-17) and |t| <= 1/4 (t^11, t^12; below 3e-18):
// 36 or 48 instructions per (node, baseline) with the gradient.  Grids whose
// nodes lie further apart take sincos per node as before.  Measured (GB300):
// 1000 bins x 16384 nodes x 8 baselines with gradient 18.9 -> 12.1 ms, 1000 x
// 262 x 8 825 -> 435 us (the split mapping filled a sixth of the GPU), nu_mu
// disappearance 400 x 513 x 2 23.3 ms -> 102 us (whole bins: 13 warps); the
// FP64 pipe is 89 % busy with 16 warps per SM.
//
// Per baseline and pair (y = 2x):
//   T = sum W (1 - cos y), V = sum W sin y (any channel),
//   N = sum W/E sin y, Z = sum W/E cos y (any channel).
#pragma once

#include "common.cuh"
#include "epilogue.cuh"
#include "general.cuh"

namespace gna {

constexpr int kChunk64 = 32;

struct Args64 {
    const double2* grid;  // {1/E, W}, [group][node][lane]
    const int64_t* goff;  // [ngrids] first node of each grid
    const int* gn;        // [ngrids] order of each grid
    const int* gid;       // [npts] grid of each point, or NULL
    const int* tasks;     // [ntasks] p * ngroups + b (whole bins)
    int ntasks, ngroups, nbins;
    const PointConst* pcs;
    const GenConst* gc;   // any channel, or NULL
    BaseConst bc;
    int* counter;
    EpiArgs ea;
    int S, L;             // slices per group and nodes per slice (S = 1: whole bins)
    double* part;         // [ntasks][NVs][32] (S > 1)
    int NVs;
    int nL, spec;
    const float2* step;   // [ngrids][ngroups] .x: largest step of 1/E
};

// Values of a task: T(3), [V(3)], [N(3)], [Z(3)], sum W, [per-baseline parts].
__host__ __device__ constexpr int sums64(bool gen, bool grad) { return 3 + (gen ? 3 : 0) + (grad ? 3 : 0) + (gen && grad ? 3 : 0) + 1; }

template <bool GEN, bool GRAD>
struct Sums64 {
    double T[3], V[3], N[3], Z[3], W;
};

// sin t and cos t - 1 for |t| <= 2^-6 (SMALL) or 1/4.
template <bool SMALL>
__device__ __forceinline__ void small_angle(double t, double& s, double& h) {
    const double u = t * t;
    double p, c;
    if constexpr (SMALL) {
        p = fma(u, 1.0 / 120.0, -1.0 / 6.0);
        c = fma(u, -1.0 / 720.0, 1.0 / 24.0);
    } else {
        p = fma(u, -1.0 / 39916800.0, 1.0 / 362880.0);
        p = fma(p, u, -1.0 / 5040.0);
        p = fma(p, u, 1.0 / 120.0);
        p = fma(p, u, -1.0 / 6.0);
        c = fma(u, 1.0 / 479001600.0, -1.0 / 3628800.0);
        c = fma(c, u, 1.0 / 40320.0);
        c = fma(c, u, -1.0 / 720.0);
        c = fma(c, u, 1.0 / 24.0);
    }
    c = fma(c, u, -0.5);
    s = fma(t * u, p, t);
    h = u * c;
}

// sin and cos of the phase x = c e, reduced modulo pi from the exact product.
__device__ __forceinline__ void phase_sincos(double c, double e, double& s, double& co) {
    const double p = c * e;
    const double lo = fma(c, e, -p);
    const double q = rint(p * GNA_INV_PI_D);
    double r = fma(-q, GNA_PI_DA, p);
    r = fma(-q, GNA_PI_DB, r);
    r = fma(-q, GNA_PI_DC, r) + lo;
    sincos(r, &s, &co);
}

// One baseline's sums over a chunk of nodes k0 <= k < k1 around e0, without the anchor's rotation.
template <bool GRAD>
struct Chunk64 {
    double S[3], H[3], SE[3], HE[3];
};
template <bool GRAD, bool SMALL>
__device__ __forceinline__ void chunk_sums(const double2* g, int k0, int k1, double e0, double c21, double c32,
                                           Chunk64<GRAD>& x) {
#pragma unroll
    for (int j = 0; j < 3; j++) x.S[j] = x.H[j] = x.SE[j] = x.HE[j] = 0.0;
    double2 nx = g[(int64_t)k0 * 32];
#pragma unroll 1
    for (int k = k0; k < k1; k++) {
        const double2 n = nx;
        if (k + 1 < k1) nx = g[(int64_t)(k + 1) * 32];
        const double d = n.x - e0;
        double s1, h1, s2, h2;
        small_angle<SMALL>(c21 * d, s1, h1);
        small_angle<SMALL>(c32 * d, s2, h2);
        const double s3 = fma(h1, s2, fma(s1, h2, s1 + s2)), h3 = fma(-s1, s2, fma(h1, h2, h1 + h2));
        x.S[0] = fma(n.y, s1, x.S[0]);
        x.S[1] = fma(n.y, s3, x.S[1]);
        x.S[2] = fma(n.y, s2, x.S[2]);
        x.H[0] = fma(n.y, h1, x.H[0]);
        x.H[1] = fma(n.y, h3, x.H[1]);
        x.H[2] = fma(n.y, h2, x.H[2]);
        if constexpr (GRAD) {
            const double we = n.y * n.x;
            x.SE[0] = fma(we, s1, x.SE[0]);
            x.SE[1] = fma(we, s3, x.SE[1]);
            x.SE[2] = fma(we, s2, x.SE[2]);
            x.HE[0] = fma(we, h1, x.HE[0]);
            x.HE[1] = fma(we, h3, x.HE[1]);
            x.HE[2] = fma(we, h2, x.HE[2]);
        }
    }
}

// sum_ij A_ij/2 T_ij
__device__ __forceinline__ double spectrum_part64(const PointConst* pc, const double (&T)[3]) {
    return 0.5 * (pc->A[0] * T[0] + pc->A[1] * T[1] + pc->A[2] * T[2]);
}

// The values the epilogues take (fused64.cuh, general.cuh), from the sums.
template <bool GEN, bool GRAD>
__device__ __forceinline__ void values64(const PointConst* pc, const Sums64<GEN, GRAD>& q, double* v) {
    if constexpr (GEN) {
#pragma unroll
        for (int j = 0; j < 3; j++) {
            v[j] = 0.5 * q.T[j];
            v[3 + j] = 0.5 * q.V[j];
            if constexpr (GRAD) {
                v[6 + j] = q.N[j];
                v[9 + j] = 2.0 * q.Z[j];
            }
        }
        v[GRAD ? 12 : 6] = q.W;
    } else {
        v[0] = q.W - spectrum_part64(pc, q.T);
        if constexpr (GRAD) {
            v[1] = 0.5 * (pc->dA12[0] * q.T[0] + pc->dA12[1] * q.T[1] + pc->dA12[2] * q.T[2]);
            v[2] = 0.5 * (pc->dA13[0] * q.T[0] + pc->dA13[1] * q.T[1] + pc->dA13[2] * q.T[2]);
            v[3] = pc->A[0] * q.N[0] + pc->A[1] * q.N[1];
            v[4] = pc->A[1] * q.N[1] + pc->A[2] * q.N[2];
        }
    }
}

template <bool GEN, bool GRAD>
__device__ __forceinline__ void finish64(const EpiArgs& ea, const PointConst* pcs, const GenConst* gc, int p, int b, int lane,
                                         const Sums64<GEN, GRAD>& q, const double* sp) {
    const int i = b * 32 + lane;
    if constexpr (GEN) {
        float2 regs[kGenNBVFit];
        double v[13];
        values64<GEN, GRAD>(nullptr, q, v);
        if (i < ea.nbins) gen_bin_epilogue64(ea, gc[p], p, i, v, GRAD ? 13 : 7, bin_inputs(ea, p, i), regs);
        gen_group_done(ea, p, b, lane, regs);
    } else {
        float2 regs[15];
        double v[kMaxNV];
        values64<GEN, GRAD>(pcs + p, q, v);
        for (int r = 0; r < ea.nspec; r++) v[(GRAD ? 5 : 1) + r] = q.W - sp[r];
        if (i < ea.nbins) bin_epilogue(ea, p, i, v, bin_inputs(ea, p, i), regs);
        group_done(ea, p, b, lane, regs);
    }
}

template <bool GEN, bool GRAD>
__global__ void __launch_bounds__(128) k_nodes64(Args64 a) {
    const int lane = threadIdx.x & 31;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // slices take the same time each: static; whole bins from the counter, longest first
    const int warps = gridDim.x * (blockDim.x >> 5);
    int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    while (true) {
        if (a.S <= 1) {
            if (lane == 0) t = atomicAdd(a.counter, 1);
            t = __shfl_sync(0xffffffffu, t, 0);
        }
        if (t >= a.ntasks) break;
        int p, b, k0 = 0;
        if (a.S > 1) {
            const int per_point = a.ngroups * a.S;
            p = t / per_point;
            const int rem = t - p * per_point;
            b = rem / a.S;
            k0 = (rem - b * a.S) * a.L;
        } else {
            const int task = a.tasks[t];
            p = task / a.ngroups;
            b = task - p * a.ngroups;
        }
        const int gi = a.gid ? a.gid[p] : 0;
        const int n = a.gn[gi];
        const int kn = min(n, k0 + (a.S > 1 ? a.L : n)) - k0;
        const double2* g = a.grid + a.goff[gi] + ((int64_t)b * n + k0) * 32 + lane;
        const PointConst* pc = a.pcs + p;
        // nodes per chunk: the anchor is node m / 2, at most m / 2 steps from the others
        const float per = 2.0f * pc->cmax * a.step[(int64_t)gi * a.ngroups + b].x;
        const float ms = 2.0f * 0.015625f / per, ml = 2.0f * 0.25f / per;
        // below eight nodes the anchors cost more than the longer polynomials
        const bool small = ms >= 8.0f;
        const float mf = small ? ms : ml;
        const bool direct = !(mf >= 4.0f);
        int m = direct || mf >= (float)kChunk64 ? kChunk64 : (int)mf;
        const int nch = (kn + m - 1) / m;
        m = (kn + nch - 1) / nch;
        Sums64<GEN, GRAD> q;
        q.W = 0.0;
#pragma unroll
        for (int j = 0; j < 3; j++) q.T[j] = q.V[j] = q.N[j] = q.Z[j] = 0.0;
        double sp[GNA_NLMAX];
        if (a.spec)
            for (int r = 0; r < a.nL; r++) sp[r] = 0.0;
        for (int ka = 0; ka < kn; ka += m) {
            const int kb = min(kn, ka + m);
            double cw = 0.0, ce = 0.0;
            for (int k = ka; k < kb; k++) {
                const double2 nd = g[(int64_t)k * 32];
                cw += nd.y;
                if constexpr (GEN || GRAD) ce = fma(nd.y, nd.x, ce);
            }
            q.W += cw;
            const double e0 = g[(int64_t)(ka + ((kb - ka) >> 1)) * 32].x;
#pragma unroll 1
            for (int r = 0; r < a.nL; r++) {
                const double c21 = pc->c21[r], c32 = pc->c32[r], om = a.bc.omd[r], kl = a.bc.kld[r];
                double T[3], V[3], N[3], Z[3];
                if (!direct) {
                    Chunk64<GRAD> x;
                    if (small) chunk_sums<GRAD, true>(g, ka, kb, e0, 2.0 * c21, 2.0 * c32, x);
                    else chunk_sums<GRAD, false>(g, ka, kb, e0, 2.0 * c21, 2.0 * c32, x);
                    double s[3], c[3];  // of the anchor's x
                    phase_sincos(c21, e0, s[0], c[0]);
                    phase_sincos(c32, e0, s[2], c[2]);
                    s[1] = s[0] * c[2] + c[0] * s[2];
                    c[1] = c[0] * c[2] - s[0] * s[2];
#pragma unroll
                    for (int j = 0; j < 3; j++) {
                        const double v = 2.0 * s[j] * s[j], sy = 2.0 * s[j] * c[j], cy = 1.0 - v;  // 1 - cos y, sin y, cos y
                        T[j] = fma(v, cw, fma(sy, x.S[j], -cy * x.H[j]));
                        if constexpr (GEN) V[j] = fma(sy, cw + x.H[j], cy * x.S[j]);
                        if constexpr (GRAD) N[j] = fma(sy, ce + x.HE[j], cy * x.SE[j]);
                        if constexpr (GEN && GRAD) Z[j] = fma(cy, ce + x.HE[j], -sy * x.SE[j]);
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < 3; j++) T[j] = V[j] = N[j] = Z[j] = 0.0;
#pragma unroll 1
                    for (int k = ka; k < kb; k++) {
                        const double2 nd = g[(int64_t)k * 32];
                        double s[3], c[3];
                        phase_sincos(c21, nd.x, s[0], c[0]);
                        phase_sincos(c32, nd.x, s[2], c[2]);
                        s[1] = s[0] * c[2] + c[0] * s[2];
                        c[1] = c[0] * c[2] - s[0] * s[2];
                        const double w2 = 2.0 * nd.y;
#pragma unroll
                        for (int j = 0; j < 3; j++) {
                            T[j] = fma(w2 * s[j], s[j], T[j]);
                            const double sc = w2 * s[j] * c[j];
                            if constexpr (GEN) V[j] += sc;
                            if constexpr (GRAD) N[j] = fma(sc, nd.x, N[j]);
                            if constexpr (GEN && GRAD) Z[j] = fma(nd.y * nd.x, fma(c[j], c[j], -s[j] * s[j]), Z[j]);
                        }
                    }
                }
                const double ok = om * kl;
#pragma unroll
                for (int j = 0; j < 3; j++) {
                    q.T[j] = fma(om, T[j], q.T[j]);
                    if constexpr (GEN) q.V[j] = fma(om, V[j], q.V[j]);
                    if constexpr (GRAD) q.N[j] = fma(ok, N[j], q.N[j]);
                    if constexpr (GEN && GRAD) q.Z[j] = fma(ok, Z[j], q.Z[j]);
                }
                if (!GEN && a.spec) sp[r] += spectrum_part64(pc, T);
            }
        }
        if (a.S > 1) {
            double* pp = a.part + (int64_t)t * a.NVs * 32 + lane;
            int v = 0;
#pragma unroll
            for (int j = 0; j < 3; j++) pp[32 * v++] = q.T[j];
            if constexpr (GEN) {
#pragma unroll
                for (int j = 0; j < 3; j++) pp[32 * v++] = q.V[j];
            }
            if constexpr (GRAD) {
#pragma unroll
                for (int j = 0; j < 3; j++) pp[32 * v++] = q.N[j];
            }
            if constexpr (GEN && GRAD) {
#pragma unroll
                for (int j = 0; j < 3; j++) pp[32 * v++] = q.Z[j];
            }
            pp[32 * v++] = q.W;
            if (!GEN && a.spec)
                for (int r = 0; r < a.nL; r++) pp[32 * v++] = sp[r];
            t += warps;
        } else {
            finish64<GEN, GRAD>(a.ea, a.pcs, a.gc, p, b, lane, q, sp);
        }
    }
    asm volatile("griddepcontrol.launch_dependents;");
}

// Slice sums (in slice order per warp, the warps' sums in warp order), then the
// epilogue: one block of W warps per (point, group).
template <bool GEN, bool GRAD, int W>
__global__ void __launch_bounds__(W * 32) k_slices_reduce64(const double* __restrict__ part, int S, int NV, EpiArgs ea,
                                                            const PointConst* __restrict__ pcs, const GenConst* __restrict__ gc) {
    extern __shared__ double red64[];  // [W][NV][32]
    const int p = blockIdx.x / ea.ngroups, b = blockIdx.x - p * ea.ngroups;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    asm volatile("griddepcontrol.launch_dependents;");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const double* base = part + (int64_t)blockIdx.x * S * NV * 32 + lane;
    for (int v = 0; v < NV; v++) {
        double s = 0.0;
        for (int sl = w; sl < S; sl += W) s += base[((int64_t)sl * NV + v) * 32];
        red64[(w * NV + v) * 32 + lane] = s;
    }
    __syncthreads();
    const int used = min(W, S);
    for (int v = w; v < NV; v += W) {
        double s = red64[v * 32 + lane];
        for (int k = 1; k < used; k++) s += red64[(k * NV + v) * 32 + lane];
        red64[v * 32 + lane] = s;
    }
    __syncthreads();
    if (w == 0) {
        Sums64<GEN, GRAD> q;
        int v = 0;
#pragma unroll
        for (int j = 0; j < 3; j++) q.T[j] = red64[32 * v++ + lane];
        if constexpr (GEN) {
#pragma unroll
            for (int j = 0; j < 3; j++) q.V[j] = red64[32 * v++ + lane];
        }
        if constexpr (GRAD) {
#pragma unroll
            for (int j = 0; j < 3; j++) q.N[j] = red64[32 * v++ + lane];
        }
        if constexpr (GEN && GRAD) {
#pragma unroll
            for (int j = 0; j < 3; j++) q.Z[j] = red64[32 * v++ + lane];
        }
        q.W = red64[32 * v++ + lane];
        double sp[GNA_NLMAX];
        if (!GEN)
            for (int r = 0; r < ea.nspec; r++) sp[r] = red64[32 * v++ + lane];
        finish64<GEN, GRAD>(ea, pcs, gc, p, b, lane, q, sp);
    }
}

// Launchers (nodes64.cu).
cudaError_t launch_nodes64(bool gen, bool grad, const Args64& a, int grid, int block, cudaStream_t s);
cudaError_t launch_slices_reduce64(bool gen, bool grad, const double* part, int S, int NV, const EpiArgs& ea,
                                   const PointConst* pcs, const GenConst* gc, int npts, cudaStream_t s);

}  // namespace gna
