// general_nodes.cuh -- chunk-anchored node kernels of the any-channel chain in
// the mixed precisions (the fits' node kernel is in general.cuh).
//
// As in anchored.cuh the phases y_ij = 2 c_ij,r / E are carried from a chunk's
// anchor.  The channel's coefficients a_ij, b_ij are not known to the node
// pass; per baseline and pair it sums
//   T = sum_k W_k (1 - cos y),  V = sum_k W_k sin y,
//   Y = sum_k W_k/E_k sin y,    Z = sum_k W_k/E_k cos y   (gradient),
// and the epilogue forms (sin^2 x = (1 - cos y) / 2, 2 sin x cos x = sin y)
//   M = delta_ab sum_k W_k + sum_ij (a_ij T_ij + b_ij V_ij) / 2
// and its six derivatives.  Near the zeros of P M is a small difference:
// survival channels have sum a_ij ~ -1 where T -> 2 sum W, appearance
// channels small T.  So the anchor is reduced modulo pi/2, |r0| <= pi/4, and
// with s = sin r, h = cos r - 1 (never formed as a difference) a chunk in
// quadrant q adds to
//   T: -H, C + S, 2C + H, C - S     V: S, C + H, -S, -(C + H)     (q = 0, 1, 2, 3)
//   Y: as V with the weights W/E    Z: C + H, -S, -(C + H), S
// where H = sum W h, S = sum W s, C = sum W: the large part is C, summed with
// compensation, and the rest carries an error relative to itself.
//
// The CP terms cancel further: b_21 = b_32 = -b_31, and V_21 + V_32 - V_31 is a
// product of three sines.  So of the third pair a node adds only what
// s_31 = s_21 + s_32 + (s_21 h_32 + h_21 s_32) and
// h_31 = h_21 + h_32 + (h_21 h_32 - s_21 s_32) have beyond the other two, and
// a chunk's sums S, H of pair 31 are put together from the three in float
// pairs: the roundings of S_21 and S_32 drop out (P(e -> tau), 5.8 MeV at 4.2
// GeV, 810 and 295 km: 8.2e-8 of the prediction with s_31 summed by itself,
// 1.1e-8 so).
//
// What bounds it: the FP32 pipe.  Operations per (node, baseline), gradient
// on: phases 2, sines and cosines 20, addition 4, sums 12 = 38, two more with
// one baseline (reducing each node's phases, with sin^2, cos^2 and sin cos of
// three phases: 120-150).
#pragma once

#include "anchored.cuh"
#include "general.cuh"
#include "slices.cuh"

namespace gna {

constexpr float kSwingQ = 0.4f;  // the polynomials (ff_consts.h) cover pi/4 + this
constexpr int gen_sums(bool grad) { return grad ? 12 : 6; }  // T, V, [Y, Z] of three pairs

// s = sin r, h = cos r - 1 on |r| <= pi/4 + kSwingQ (see sinh2).
template <int N>
__device__ __forceinline__ void sinhq2(const f32x2 (&r)[N], f32x2 (&s)[N], f32x2 (&h)[N]) {
    f32x2 u[N], p[N], c[N];
#define GNA_STEP(expr)                 \
    _Pragma("unroll") for (int i = 0; i < N; i++) { \
        expr;                          \
    }
    GNA_STEP(u[i] = mul2(r[i], r[i]))
    GNA_STEP(p[i] = fma2(dup2(GNA_SINQ_C4), u[i], dup2(GNA_SINQ_C3)))
    GNA_STEP(c[i] = fma2(dup2(GNA_COSQ_C4), u[i], dup2(GNA_COSQ_C3)))
    GNA_STEP(p[i] = fma2(p[i], u[i], dup2(GNA_SINQ_C2)))
    GNA_STEP(c[i] = fma2(c[i], u[i], dup2(GNA_COSQ_C2)))
    GNA_STEP(p[i] = fma2(p[i], u[i], dup2(GNA_SINQ_C1)))
    GNA_STEP(c[i] = fma2(c[i], u[i], dup2(GNA_COSQ_C1)))
    GNA_STEP(s[i] = mul2(r[i], u[i]))
    GNA_STEP(h[i] = mul2(c[i], u[i]))
    GNA_STEP(s[i] = fma2(s[i], p[i], r[i]))
#undef GNA_STEP
}

// What sin and cos - 1 of r1 + r2 have beyond those of r1 and r2.
__device__ __forceinline__ void angle_rest2(f32x2 s1, f32x2 h1, f32x2 s2, f32x2 h2, f32x2& s, f32x2& h) {
    s = fma2(h1, s2, mul2(s1, h2));
    h = fma2(neg2(s1), s2, mul2(h1, h2));
}

// Doubled phase of baseline r's pair 21 or 32 modulo pi/2, and the quadrant
// (mod 4).  The quotient's steps q PI_A / 2 and q PI_B / 2 are exact (12-bit
// parts); r is rounded once, when the small part is added.
// FAR: as reduce_sign_ff; low: what that rounding dropped
template <int PH, bool FAR>
__device__ __forceinline__ float phase_q(const PointConst* pc, int r, bool p32, float eh, float el, unsigned& quad,
                                         float& low) {
    if constexpr (PH == 0) {
        const float ch = 2.0f * (p32 ? pc->c32h[r] : pc->c21h[r]), cl = 2.0f * (p32 ? pc->c32l[r] : pc->c21l[r]);
        const float p = __fmul_rn(ch, eh);
        const float e = __fmaf_rn(ch, eh, -p);
        const float lo = __fmaf_rn(ch, el, __fmaf_rn(cl, eh, e));
        const float qm = __fmaf_rn(p, 2.0f * GNA_INV_PI_F, GNA_ROUND_MAGIC);
        quad = __float_as_uint(qm) & 3u;
        float q = __fsub_rn(qm, GNA_ROUND_MAGIC);
        if (FAR && fabsf(p) > kFarPhase) {
            q = far_quotient(p, lo, 2.0f * GNA_INV_PI_F, 0.5f * GNA_PI_A, 0.5f * GNA_PI_B);
            quad = (unsigned)__float2int_rn(q) & 3u;
        }
        float x = __fmaf_rn(-q, 0.5f * GNA_PI_A, p);
        x = __fmaf_rn(-q, 0.5f * GNA_PI_B, x);
        const float y = __fmaf_rn(-q, 0.5f * GNA_PI_C, lo), s = __fadd_rn(x, y);
        low = __fadd_rn(__fsub_rn(x, s), y);  // (|x| >= |y|, or both are tiny)
        return s;
    } else {
        const double p = 2.0 * (p32 ? pc->c32[r] : pc->c21[r]) * ((double)eh + (double)el);
        const double qm = fma(p, 2.0 * GNA_INV_PI_D, 6755399441055744.0);
        quad = (unsigned)__double2loint(qm) & 3u;
        const double q = qm - 6755399441055744.0;
        double x = fma(-q, 0.5 * GNA_PI_DA, p);
        x = fma(-q, 0.5 * GNA_PI_DB, x);
        x = fma(-q, 0.5 * GNA_PI_DC, x);
        const float s = (float)x;
        low = (float)(x - (double)s);
        return s;
    }
}
template <int PH, bool FAR>
__device__ __forceinline__ float phase_q(const PointConst* pc, int r, bool p32, float eh, float el, unsigned& quad) {
    float low;
    return phase_q<PH, FAR>(pc, r, p32, eh, el, quad, low);
}

// What a chunk in quadrant q adds, as big + part (T, V: |big| >= |part| or
// big = 0; c: 2 * float pair sum W) or one float (Y, Z; e: sum W/E).
struct QuadrantSums {
    float2 T, V;  // {big, part} with the pair's low part of C apart
    float Tl, Vl;
};
__device__ __forceinline__ QuadrantSums quadrant_sums(unsigned q, float2 S, float2 H, float2 c) {
    QuadrantSums r;
    const bool odd = q & 1u;
    const float k = odd ? 1.0f : (q & 2u) ? 2.0f : 0.0f;
    const float st = ((q + 1u) & 2u) ? 1.0f : -1.0f;  // T: -H, +S, +H, -S
    const float sv = (q & 2u) ? -1.0f : 1.0f;         // V: S, C + H, -S, -(C + H)
    r.T = make_float2(k * c.x, st * (odd ? S.x : H.x));
    r.Tl = fmaf(k, c.y, st * (odd ? S.y : H.y));
    r.V = make_float2(odd ? sv * c.x : 0.f, sv * (odd ? H.x : S.x));
    r.Vl = sv * (odd ? c.y + H.y : S.y);
    return r;
}
__device__ __forceinline__ float quadrant_Y(unsigned q, float SE, float HE, float e) {
    const float x = (q & 1u) ? e + HE : SE;
    return (q & 2u) ? -x : x;
}
__device__ __forceinline__ float quadrant_Z(unsigned q, float SE, float HE, float e) {
    const float x = (q & 1u) ? SE : e + HE;
    return ((q + 1u) & 2u) ? -x : x;
}
// big + part + lo as a float pair (see QuadrantSums)
__device__ __forceinline__ float2 big_sum(float2 v, float lo) {
    const float hi = __fadd_rn(v.x, v.y);
    return make_float2(hi, __fadd_rn(__fadd_rn(v.y, __fsub_rn(v.x, hi)), lo));
}

// One baseline's running sums of a task.
template <bool GRAD>
struct GenSums {
    float2 T[3], V[3];
    KahanF Y[3], Z[3];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int j = 0; j < 3; j++) {
            T[j] = V[j] = make_float2(0.f, 0.f);
            kzero(Y[j]);
            kzero(Z[j]);
        }
    }
    // a chunk's sums of the three pairs, [1] the third's beyond the other two,
    // S, H of pair 32 as pairs; q21, q32: quadrants
    __device__ __forceinline__ void add(unsigned q21, unsigned q32, const float (&S)[2], const float (&H)[2], float2 S32,
                                        float2 H32, const float (&SE)[3], const float (&HE)[3], float2 c, float e) {
        const float2 s = make_float2(S[0], 0.f), h = make_float2(H[0], 0.f);
        add(0, q21, s, h, SE[0], HE[0], c, e);
        add(1, (q21 + q32) & 3u, ff_add(ff_add(s, S32), make_float2(S[1], 0.f)),
            ff_add(ff_add(h, H32), make_float2(H[1], 0.f)), SE[0] + SE[2] + SE[1], HE[0] + HE[2] + HE[1], c, e);
        add(2, q32, S32, H32, SE[2], HE[2], c, e);
    }
    // a chunk's sums of pair j
    __device__ __forceinline__ void add(int j, unsigned q, float2 S, float2 H, float SE, float HE, float2 c, float e) {
        const QuadrantSums r = quadrant_sums(q, S, H, c);
        T[j] = ff_add(T[j], big_sum(r.T, r.Tl));
        V[j] = ff_add(V[j], big_sum(r.V, r.Vl));
        if constexpr (GRAD) {
            kadd_prod(Y[j], 1.0f, quadrant_Y(q, SE, HE, e));
            kadd_prod(Z[j], 1.0f, quadrant_Z(q, SE, HE, e));
        }
    }
};

// Sums over the baselines: T, V weighted by omega_r, Y by omega_r K L_r, Z by
// 2 omega_r K L_r.
struct GenTaskSums {
    float2 T[3], V[3], Y[3], Z[3];
};

template <bool GRAD>
__device__ __forceinline__ void store_gen_sums(const GenTaskSums& q, float2* pp) {
#pragma unroll
    for (int j = 0; j < 3; j++) {
        pp[j * 32] = q.T[j];
        pp[(3 + j) * 32] = q.V[j];
        if constexpr (GRAD) {
            pp[(6 + j) * 32] = q.Y[j];
            pp[(9 + j) * 32] = q.Z[j];
        }
    }
}

// A bin's prediction (in float pairs: its terms may cancel) and derivatives.
template <bool GRAD>
__device__ __forceinline__ BinSums<GRAD ? 6 : 0> gen_bin_sums(const GenConst& c, float2 sumw, const GenTaskSums& q) {
    BinSums<GRAD ? 6 : 0> b;
    float2 M = c.dab != 0.0 ? sumw : make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < 3; j++) {
        M = ff_add(M, ff_mul(0.5f * c.af[j], 0.5f * c.alo[j], q.T[j]));
        M = ff_add(M, ff_mul(0.5f * c.bf[j], 0.5f * c.blo[j], q.V[j]));
    }
    b.M = M;
    if constexpr (GRAD) {
        float U[3], C[3], Y[3], Z[3];
#pragma unroll
        for (int j = 0; j < 3; j++) {
            U[j] = 0.5f * (q.T[j].x + q.T[j].y);
            C[j] = 0.5f * (q.V[j].x + q.V[j].y);
            Y[j] = q.Y[j].x + q.Y[j].y;
            Z[j] = q.Z[j].x + q.Z[j].y;
        }
#pragma unroll
        for (int p = 0; p < 4; p++) {
            b.d[p] = 0.f;
#pragma unroll
            for (int j = 0; j < 3; j++) b.d[p] = fmaf(c.daf[p][j], U[j], fmaf(c.dbf[p][j], C[j], b.d[p]));
        }
        // pairs 0 = 21, 1 = 31, 2 = 32; x31 moves with both splittings
        const float t31 = fmaf(c.af[1], Y[1], 0.5f * c.bf[1] * Z[1]);
        b.d[4] = fmaf(c.af[0], Y[0], fmaf(0.5f * c.bf[0], Z[0], t31));
        b.d[5] = fmaf(c.af[2], Y[2], fmaf(0.5f * c.bf[2], Z[2], t31));
    }
    return b;
}

template <bool GRAD>
__device__ __forceinline__ void finish_gen_bins(const GenArgs& ga, int p, int b, const GenTaskSums& q, const BinInput& in,
                                                int lane) {
    constexpr int NG = GRAD ? 6 : 0;
    const int i = b * 32 + lane;
    float2 regs[1 + NG];
    if (i < ga.b.nbins) bin_terms<NG>(ga.b.ea, p, i, gen_bin_sums<GRAD>(ga.gc[p], in.sumw, q), nullptr, in, regs);
    group_terms<NG>(ga.b.ea, p, b, lane, regs);
}

// One node on its own (grids too coarse for chunks): its phases reduced, its
// terms added to baseline r's sums as a chunk of one.
template <int PH, bool GRAD>
__device__ __forceinline__ void gen_single(const PointConst* pc, int r, float eh, float el, float W, GenSums<GRAD>& g) {
    unsigned q21, q32;
    const f32x2 y[1] = {pack2(phase_q<PH, true>(pc, r, false, eh, el, q21), phase_q<PH, true>(pc, r, true, eh, el, q32))};
    f32x2 s[1], h[1], s3, h3;
    sinhq2(y, s, h);
    angle_rest2(dup2(s[0].x), dup2(h[0].x), dup2(s[0].y), dup2(h[0].y), s3, h3);
    const float We = W * eh;
    const float S[2] = {W * s[0].x, W * s3.x}, H[2] = {W * h[0].x, W * h3.x};
    const float SE[3] = {We * s[0].x, We * s3.x, We * s[0].y}, HE[3] = {We * h[0].x, We * h3.x, We * h[0].y};
    g.add(q21, q32, S, H, make_float2(W * s[0].y, 0.f), make_float2(W * h[0].y, 0.f), SE, HE, make_float2(W, 0.f), We);
}

// ---------------------------------------------------- one baseline -------
// S and H of pair 32 are summed as differences from their values s0, h0 at the
// anchor, which enter with the chunk's weight: FP32 sums of up to 32 terms near
// 0.7 (the quadrants' edges) were the largest error of a bin that is one chunk
// (nu_mu disappearance in 40 - 500 bins of 4 - 2400 nodes, largest error of a
// bin: 1.8e-7 of mu, 6.0e-8 so; a reduction and a compensated sum per node
// 7.5e-8; scan of 1021 points 135 -> 138 us).
template <int PH, bool GRAD>
struct GenOneMath {
    f32x2 c21, c32, a21, a32;
    f32x2 S[3], H[3], SE[3], HE[3];
    float s0, h0;

    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int j = 0; j < 3; j++) S[j] = H[j] = SE[j] = HE[j] = f32x2{0.f, 0.f};
    }
    // s0, h0: at a32
    __device__ __forceinline__ void base() {
        const f32x2 y[1] = {a32};
        f32x2 s[1], h[1];
        sinhq2(y, s, h);
        s0 = s[0].x;
        h0 = h[0].x;
    }
    __device__ __forceinline__ void pair(const NodePair& n, f32x2 nah, f32x2 nal, f32x2 we) {
        const f32x2 d = add2(add2(n.e, nah), add2(n.l, nal));
        const f32x2 r[2] = {fma2(c21, d, a21), fma2(c32, d, a32)};
        f32x2 s[2], h[2], s3, h3;
        sinhq2(r, s, h);
        angle_rest2(s[0], h[0], s[1], h[1], s3, h3);
        H[0] = fma2(n.w, h[0], H[0]);
        H[1] = fma2(n.w, h3, H[1]);
        H[2] = fma2(n.w, add2(h[1], dup2(-h0)), H[2]);
        S[0] = fma2(n.w, s[0], S[0]);
        S[1] = fma2(n.w, s3, S[1]);
        S[2] = fma2(n.w, add2(s[1], dup2(-s0)), S[2]);
        if constexpr (GRAD) {
            HE[0] = fma2(we, h[0], HE[0]);
            HE[1] = fma2(we, h3, HE[1]);
            HE[2] = fma2(we, h[1], HE[2]);
            SE[0] = fma2(we, s[0], SE[0]);
            SE[1] = fma2(we, s3, SE[1]);
            SE[2] = fma2(we, s[1], SE[2]);
        }
    }
};

template <int PH, bool GRAD>
__global__ void __maxnreg__(128) k_gen_one(GenArgs ga) {
    const BinArgs& a = ga.b;
    const int lane = threadIdx.x & 31;
    extern __shared__ f32x2p rings[];
    QuadRing<kRingOne> in(rings);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const bool whole = a.S <= 1;
    TaskQueue queue(a);
    for (int t = queue.take(); t < a.ntasks; t = queue.take()) {
        queue.prefetch();
        const NodeTask k = node_task(a, t);
        in.start(k);
        const PointConst* pc = a.pcs + k.p;
        BinInput bin;
        if (whole) bin = bin_input(a.ea, k.p, min(k.b * 32 + lane, a.nbins - 1));
        const int len = chunk_quads<PH>(pc->cmax, k.step, k.nq, kSwingQ);
        const bool direct = len == 0;
        const int step = direct ? 1 : len;
        GenOneMath<PH, GRAD> x;
        x.c21 = dup2(2.0f * pc->c21h[0]);
        x.c32 = dup2(2.0f * pc->c32h[0]);
        x.zero();
        GenSums<GRAD> g;
        g.zero();
        float2 an = load_anchor(k, 0, min(step, k.nq));
        for (int ka = 0; ka < k.nq; ka += step) {
            const int kb = min(k.nq, ka + step);
            if (!direct) {
                unsigned q21, q32;
                float low;
                x.a32 = dup2(phase_q<PH, false>(pc, 0, true, an.x, an.y, q32, low));
                // the anchor moves to where pair 32's phase is that float: its
                // rounding would be common to the chunk (nu_mu disappearance, eight
                // spectra of 4 - 1000 nodes per bin, largest error of a bin: 7.3e-8
                // -> 6.4e-8 of mu, with a reduction per node 6.7e-8)
                const float shift = low != 0.f ? __fdividef(-low, x.c32.x) : 0.f;
                x.a21 = dup2(fmaf(x.c21.x, shift, phase_q<PH, false>(pc, 0, false, an.x, an.y, q21)));
                const f32x2 nah = dup2(-an.x), nal = dup2(-an.y - shift);
                x.base();
                if (kb < k.nq) an = load_anchor(k, kb, min(step, k.nq - kb));
                WeightSum w;
                in.wait();
                w.start(in.pair(0).w);
                f32x2 e = f32x2{0.f, 0.f};
#pragma unroll 1
                for (int j = ka; j < kb; j++) {
                    in.wait();
                    const NodePair n0 = in.pair(0), n1 = in.pair(1);
                    const f32x2 we0 = mul2(n0.w, n0.e), we1 = mul2(n1.w, n1.e);
                    w.add(n0.w);
                    w.add(n1.w);
                    if constexpr (GRAD) e = add2(e, add2(we0, we1));
                    x.pair(n0, nah, nal, we0);
                    x.pair(n1, nah, nal, we1);
                    in.done();
                }
                const float2 c = w.total();
                const float es = e.x + e.y;
                float S[3], H[3], SE[3], HE[3];
#pragma unroll
                for (int v = 0; v < 3; v++) {
                    S[v] = x.S[v].x + x.S[v].y;
                    H[v] = x.H[v].x + x.H[v].y;
                    SE[v] = x.SE[v].x + x.SE[v].y;
                    HE[v] = x.HE[v].x + x.HE[v].y;
                }
                g.add(q21, q32, {S[0], S[1]}, {H[0], H[1]}, ff_add(ff_mul(x.s0, 0.f, c), make_float2(S[2], 0.f)),
                      ff_add(ff_mul(x.h0, 0.f, c), make_float2(H[2], 0.f)), SE, HE, c, es);
                x.zero();
            } else {
                in.wait();
#pragma unroll 1
                for (int u = 0; u < 4; u++) {
                    const NodePair n = in.pair(u >> 1);
                    gen_single<PH, GRAD>(pc, 0, (u & 1) ? n.e.y : n.e.x, (u & 1) ? n.l.y : n.l.x, (u & 1) ? n.w.y : n.w.x, g);
                }
                in.done();
            }
        }
        GenTaskSums q;
#pragma unroll
        for (int v = 0; v < 3; v++) {
            q.T[v] = g.T[v];
            q.V[v] = g.V[v];
            // omega = 1 for one baseline: wkl = 2 K L
            q.Y[v] = ff_mul(0.5f * a.bc.wkl[0], 0.5f * a.bc.wkllo[0], kahan_to_ff(g.Y[v]));
            q.Z[v] = ff_mul(a.bc.wkl[0], a.bc.wkllo[0], kahan_to_ff(g.Z[v]));
        }
        if (!whole) store_gen_sums<GRAD>(q, a.part + (int64_t)t * a.NVs * 32 + lane);
        else finish_gen_bins<GRAD>(ga, k.p, k.b, q, bin, lane);
    }
    asm volatile("griddepcontrol.launch_dependents;");
}

// ------------------------------------------------ several baselines ------
// 2 NP baselines at a time, two per packed value (MultiMath): the chunk's sums
// in registers, the task's in shared memory.
template <int PH, int NP, bool GRAD>
struct GenMultiMath {
    static constexpr int NS = gen_sums(GRAD);
    f32x2 c[2 * NP], a[2 * NP];
    f32x2 S[NP][3], H[NP][3], SE[NP][3], HE[NP][3];

    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int i = 0; i < NP; i++)
#pragma unroll
            for (int j = 0; j < 3; j++) S[i][j] = H[i][j] = SE[i][j] = HE[i][j] = f32x2{0.f, 0.f};
    }
    __device__ __forceinline__ void load(const PointConst* pc, int r0) {
#pragma unroll
        for (int i = 0; i < NP; i++) {
            const float2 x = *reinterpret_cast<const float2*>(pc->c21h + r0 + 2 * i);
            const float2 y = *reinterpret_cast<const float2*>(pc->c32h + r0 + 2 * i);
            c[2 * i] = pack2(2.0f * x.x, 2.0f * x.y);
            c[2 * i + 1] = pack2(2.0f * y.x, 2.0f * y.y);
        }
    }
    // quadrants: four bits per baseline (pair 21, pair 32)
    __device__ __forceinline__ unsigned anchor(const PointConst* pc, int r0, float eh, float el) {
        unsigned quads = 0;
#pragma unroll
        for (int i = 0; i < NP; i++) {
            unsigned q[4];
            float x[4];
#pragma unroll
            for (int j = 0; j < 4; j++) x[j] = phase_q<PH, false>(pc, r0 + 2 * i + (j & 1), j >= 2, eh, el, q[j]);
            a[2 * i] = pack2(x[0], x[1]);
            a[2 * i + 1] = pack2(x[2], x[3]);
            quads |= (q[0] | q[2] << 2 | q[1] << 4 | q[3] << 6) << (8 * i);
        }
        return quads;
    }
    __device__ __forceinline__ void node(float d, float W, float We) {
        const f32x2 d2 = dup2(d), W2 = dup2(W), We2 = dup2(We);
        f32x2 r[2 * NP], s[2 * NP], h[2 * NP];
#pragma unroll
        for (int i = 0; i < 2 * NP; i++) r[i] = fma2(c[i], d2, a[i]);
        sinhq2(r, s, h);
#pragma unroll
        for (int i = 0; i < NP; i++) {
            f32x2 s3, h3;
            angle_rest2(s[2 * i], h[2 * i], s[2 * i + 1], h[2 * i + 1], s3, h3);
            const f32x2 sj[3] = {s[2 * i], s3, s[2 * i + 1]}, hj[3] = {h[2 * i], h3, h[2 * i + 1]};
#pragma unroll
            for (int j = 0; j < 3; j++) {
                S[i][j] = fma2(W2, sj[j], S[i][j]);
                H[i][j] = fma2(W2, hj[j], H[i][j]);
                if constexpr (GRAD) {
                    SE[i][j] = fma2(We2, sj[j], SE[i][j]);
                    HE[i][j] = fma2(We2, hj[j], HE[i][j]);
                }
            }
        }
    }
};

// A baseline's running sums in shared memory: value v (T, V, Y, Z of the three
// pairs) of packed baseline i at comp[(i NS + v) stride], lane half `half`.
template <int NS, bool GRAD>
__device__ __forceinline__ GenSums<GRAD> load_gen(const f32x2p* comp, int stride, int i, int half) {
    GenSums<GRAD> g;
    const float* f = reinterpret_cast<const float*>(comp + i * NS * stride) + half;
    const int w = stride * 4;
#pragma unroll
    for (int j = 0; j < 3; j++) {
        g.T[j] = make_float2(f[j * w], f[j * w + 2]);
        g.V[j] = make_float2(f[(3 + j) * w], f[(3 + j) * w + 2]);
        if constexpr (GRAD) {
            g.Y[j].s = f[(6 + j) * w];
            g.Y[j].c = f[(6 + j) * w + 2];
            g.Z[j].s = f[(9 + j) * w];
            g.Z[j].c = f[(9 + j) * w + 2];
        }
    }
    return g;
}
template <int NS, bool GRAD>
__device__ __forceinline__ void save_gen(f32x2p* comp, int stride, int i, int half, const GenSums<GRAD>& g) {
    float* f = reinterpret_cast<float*>(comp + i * NS * stride) + half;
    const int w = stride * 4;
#pragma unroll
    for (int j = 0; j < 3; j++) {
        f[j * w] = g.T[j].x;
        f[j * w + 2] = g.T[j].y;
        f[(3 + j) * w] = g.V[j].x;
        f[(3 + j) * w + 2] = g.V[j].y;
        if constexpr (GRAD) {
            f[(6 + j) * w] = g.Y[j].s;
            f[(6 + j) * w + 2] = g.Y[j].c;
            f[(9 + j) * w] = g.Z[j].s;
            f[(9 + j) * w + 2] = g.Z[j].c;
        }
    }
}

template <int PH, int NP, bool GRAD>
__global__ void __maxnreg__(NP == 2 ? 168 : 128) k_gen_multi(GenArgs ga) {
    using M = GenMultiMath<PH, NP, GRAD>;
    constexpr int NS = M::NS;
    const BinArgs& a = ga.b;
    extern __shared__ f32x2p comp_all[];  // [NP * NS][blockDim], then the rings
    f32x2p* comp = comp_all + threadIdx.x;
    const int stride = blockDim.x;
    const int lane = threadIdx.x & 31;
    QuadRing<kRingMulti> in(comp_all + NP * NS * stride);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const bool whole = a.S <= 1;
    TaskQueue queue(a);
    for (int t = queue.take(); t < a.ntasks; t = queue.take()) {
        queue.prefetch();
        const NodeTask k = node_task(a, t);
        const PointConst* pc = a.pcs + k.p;
        BinInput bin;
        if (whole) bin = bin_input(a.ea, k.p, min(k.b * 32 + lane, a.nbins - 1));
        const int len = chunk_quads<PH>(pc->cmax, k.step, k.nq, kSwingQ);
        const bool direct = len == 0;
        const int step = direct ? 1 : len;
        GenTaskSums q;
#pragma unroll
        for (int j = 0; j < 3; j++) {
            q.T[j] = q.V[j] = q.Y[j] = q.Z[j] = make_float2(0.f, 0.f);
        }
        for (int r0 = 0; r0 < a.nL; r0 += 2 * NP) {
            M x;
            in.start(k);
            x.load(pc, r0);
            x.zero();
            float2 an = load_anchor(k, 0, min(step, k.nq));
            for (int ka = 0; ka < k.nq; ka += step) {
                const int kb = min(k.nq, ka + step);
                if (!direct) {
                    const unsigned quads = x.anchor(pc, r0, an.x, an.y);
                    const f32x2 nah = dup2(-an.x), nal = dup2(-an.y);
                    if (kb < k.nq) an = load_anchor(k, kb, min(step, k.nq - kb));
                    WeightSum w;
                    in.wait();
                    w.start(in.pair(0).w);
                    f32x2 e = f32x2{0.f, 0.f};
#pragma unroll 1
                    for (int j = ka; j < kb; j++) {
                        in.wait();
#pragma unroll 1
                        for (int u = 0; u < 2; u++) {
                            const NodePair n = in.pair(u);
                            const f32x2 d = add2(add2(n.e, nah), add2(n.l, nal)), we = mul2(n.w, n.e);
                            w.add(n.w);
                            if constexpr (GRAD) e = add2(e, we);
                            x.node(d.x, n.w.x, we.x);
                            x.node(d.y, n.w.y, we.y);
                        }
                        in.done();
                    }
                    const float2 c = w.total();
                    const float es = e.x + e.y;
#pragma unroll
                    for (int i = 0; i < NP; i++)
#pragma unroll
                        for (int half = 0; half < 2; half++) {
                            const unsigned b = quads >> (8 * i + 4 * half), q21 = b & 3u, q32 = (b >> 2) & 3u;
                            GenSums<GRAD> g;
                            if (ka == 0) g.zero();
                            else g = load_gen<NS, GRAD>(comp, stride, i, half);
                            float S[3], H[3], SE[3], HE[3];
#pragma unroll
                            for (int j = 0; j < 3; j++) {
                                S[j] = half ? x.S[i][j].y : x.S[i][j].x;
                                H[j] = half ? x.H[i][j].y : x.H[i][j].x;
                                SE[j] = half ? x.SE[i][j].y : x.SE[i][j].x;
                                HE[j] = half ? x.HE[i][j].y : x.HE[i][j].x;
                            }
                            g.add(q21, q32, {S[0], S[1]}, {H[0], H[1]}, make_float2(S[2], 0.f), make_float2(H[2], 0.f), SE,
                                  HE, c, es);
                            save_gen<NS, GRAD>(comp, stride, i, half, g);
                        }
                    x.zero();
                } else {
                    in.wait();
#pragma unroll 1
                    for (int r = 0; r < 2 * NP; r++) {
                        GenSums<GRAD> g;
                        if (ka == 0) g.zero();
                        else g = load_gen<NS, GRAD>(comp, stride, r >> 1, r & 1);
#pragma unroll 1
                        for (int u = 0; u < 4; u++) {
                            const NodePair n = in.pair(u >> 1);
                            gen_single<PH, GRAD>(pc, r0 + r, (u & 1) ? n.e.y : n.e.x, (u & 1) ? n.l.y : n.l.x,
                                                 (u & 1) ? n.w.y : n.w.x, g);
                        }
                        save_gen<NS, GRAD>(comp, stride, r >> 1, r & 1, g);
                    }
                    in.done();
                }
            }
#pragma unroll 1
            for (int i = 0; i < 2 * NP && r0 + i < a.nL; i++) {
                const int r = r0 + i;
                const GenSums<GRAD> g = load_gen<NS, GRAD>(comp, stride, i >> 1, i & 1);
#pragma unroll
                for (int j = 0; j < 3; j++) {
                    q.T[j] = ff_add(q.T[j], ff_mul(a.bc.om[r], a.bc.omlo[r], g.T[j]));
                    q.V[j] = ff_add(q.V[j], ff_mul(a.bc.om[r], a.bc.omlo[r], g.V[j]));
                    if constexpr (GRAD) {
                        q.Y[j] = ff_add(q.Y[j], ff_mul(0.5f * a.bc.wkl[r], 0.5f * a.bc.wkllo[r], kahan_to_ff(g.Y[j])));
                        q.Z[j] = ff_add(q.Z[j], ff_mul(a.bc.wkl[r], a.bc.wkllo[r], kahan_to_ff(g.Z[j])));
                    }
                }
            }
        }
        if (!whole) store_gen_sums<GRAD>(q, a.part + (int64_t)t * a.NVs * 32 + lane);
        else finish_gen_bins<GRAD>(ga, k.p, k.b, q, bin, lane);
    }
    asm volatile("griddepcontrol.launch_dependents;");
}

// Slice sums, then the epilogue and the group and point reductions.
template <int NVM, int W>
__global__ void __launch_bounds__(W * 32) k_gen_slices_reduce(const float2* __restrict__ part, int S, int NV, EpiArgs ea,
                                                              const GenConst* __restrict__ gc) {
    const int p = blockIdx.x / ea.ngroups, g = blockIdx.x - p * ea.ngroups;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = g * 32 + lane;
    BinInput in;
    if (w == 0) in = bin_input(ea, p, min(i, ea.nbins - 1));
    const float2* fin = sum_slices<NVM, W>(part, S, NV, w, lane);
    if (w == 0) {
        GenTaskSums q;
        for (int j = 0; j < 3; j++) {
            q.T[j] = fin[j * 32 + lane];
            q.V[j] = fin[(3 + j) * 32 + lane];
        }
        if (ea.has_grad) {
            for (int j = 0; j < 3; j++) {
                q.Y[j] = fin[(6 + j) * 32 + lane];
                q.Z[j] = fin[(9 + j) * 32 + lane];
            }
            float2 regs[7];
            if (i < ea.nbins) bin_terms<6>(ea, p, i, gen_bin_sums<true>(gc[p], in.sumw, q), nullptr, in, regs);
            group_done_terms<6>(ea, p, g, lane, regs);
        } else {
            float2 regs[1];
            if (i < ea.nbins) bin_terms<0>(ea, p, i, gen_bin_sums<false>(gc[p], in.sumw, q), nullptr, in, regs);
            group_done_terms<0>(ea, p, g, lane, regs);
        }
    }
}

}  // namespace gna
