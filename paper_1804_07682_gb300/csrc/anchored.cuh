// anchored.cuh -- node pass of the mixed precisions, bin and slice mappings:
// phases carried from chunk anchors, two FP32 lanes per instruction.
//
// Per energy node and baseline the pass needs cos and sin of the doubled
// phases y_ij = 2 c_ij,r / E (c = K dm2 L), since sin^2 x = (1 - cos 2x) / 2
// and 2 sin x cos x = sin 2x.  It accumulates per baseline r
//   T_ij,r = sum_k W_k (1 - cos y_ij),   N_ij,r = sum_k W_k/E_k sin y_ij,
// from which (P_r = 1 - sum_ij A_ij sin^2 x_ij, omega_r the baseline weights)
//   sum_k W_k P_r = sum_k W_k - sum_ij A_ij/2 T_ij,r,
//   d/d s2   = -sum_ij dA_ij/2 sum_r omega_r T_ij,r,
//   d/d dm2_21 = -sum_r omega_r K L_r (A21 N21 + A31 N31), d/d dm2_32 likewise with 31, 32.
//
// Anchors.  A lane walks the nodes of one bin in order, so 1/E moves by small
// steps.  The nodes are taken in chunks of at most kChunkQuads quads; the phase
// of a node in the chunk's middle is formed and reduced modulo pi exactly
// (double-float, or in double), y = q pi + r0, and a node's argument is
// r = r0 + 2c d with d = 1/E - 1/E_anchor (the float pairs' high parts subtract
// exactly): one FMA instead of the nine operations of a reduction.  The chunk
// length is chosen per task so that |2c d| <= kSwing for every phase (c from
// the point's constants, the largest step of 1/E from the plan), which bounds
// the offset's rounding to that of r0 and keeps r inside the polynomials'
// range.  The sign (-1)^q is common to the chunk and applied when its sums are
// added: with s = sin r, h = cos r - 1
//   q even: 1 - cos y = -h,     sin y =  s,
//   q odd:  1 - cos y = 2 + h,  sin y = -s,
// so an odd chunk adds 2 sum W.  h is formed without the 1, and the third pair
// by the addition formulas in (s, h), so small phases keep their relative
// accuracy, and so does P where 1 - cos y is close to 2.  Grids whose
// neighbouring nodes lie too far apart for chunks of one quad reduce every
// node's phases instead (direct).
//
// The chunk sums are plain FP32 sums of at most 32 terms; they are added to the
// task's sums in double-float (T) or with Kahan compensation (N).
//
// What bounds it: the FP32 pipe.  Operations per (node, baseline), gradient
// on: phases 2, sines and cosines 22, addition 6, sums 6 = 36 (reducing each
// node's phases: 61).  fma.rn.f32x2 runs at the plain FMA rate per lane but
// takes half the issue slots, so the loads, address arithmetic and loop
// control no longer compete with the arithmetic.  An FMA (packed or not) that
// reads three registers no neighbouring instruction reads runs at two thirds
// of the rate (26 against 39 T lane operations/s measured): the polynomials
// of all phases in hand are stepped together, so that neighbours share a
// coefficient.  Nodes come through a ring in shared memory (cp.async): with
// loads into registers the warps spent half their time waiting for them.
#pragma once

#include "common.cuh"
#include "epilogue.cuh"
#include "fused.cuh"

namespace gna {

constexpr int kChunkQuads = 8;
constexpr float kSwing = 0.25f;  // the polynomials (ff_consts.h) cover pi/2 + this
constexpr int kRingOne = 4, kRingMulti = 3;  // quads per lane in shared memory

// ------------------------------------------------------- packed floats --
struct __align__(8) f32x2 {
    float x, y;
};
struct __align__(16) f32x2p {  // two packed values: high and low parts
    f32x2 x, y;
};

__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("{\n\t.reg .b64 p, q, s, t;\n\tmov.b64 p, {%2, %3};\n\tmov.b64 q, {%4, %5};\n\tmov.b64 s, {%6, %7};\n\t"
        "fma.rn.f32x2 t, p, q, s;\n\tmov.b64 {%0, %1}, t;\n\t}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("{\n\t.reg .b64 p, q, t;\n\tmov.b64 p, {%2, %3};\n\tmov.b64 q, {%4, %5};\n\t"
        "mul.rn.f32x2 t, p, q;\n\tmov.b64 {%0, %1}, t;\n\t}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("{\n\t.reg .b64 p, q, t;\n\tmov.b64 p, {%2, %3};\n\tmov.b64 q, {%4, %5};\n\t"
        "add.rn.f32x2 t, p, q;\n\tmov.b64 {%0, %1}, t;\n\t}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ f32x2 pack2(float a, float b) { return f32x2{a, b}; }
__device__ __forceinline__ f32x2 dup2(float a) { return f32x2{a, a}; }
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) { return fma2(b, dup2(-1.0f), a); }
__device__ __forceinline__ f32x2 neg2(f32x2 a) { return f32x2{-a.x, -a.y}; }

// Sum of two pairs of floats per lane (x + y, error-free in the high parts, not normalised).
__device__ __forceinline__ f32x2p ff_add2(f32x2p a, f32x2p b) {
    const f32x2 s = add2(a.x, b.x), t = sub2(s, a.x);
    const f32x2 e = add2(sub2(a.x, sub2(s, t)), sub2(b.x, t));
    return f32x2p{s, add2(add2(a.y, b.y), e)};
}

// Compensated sum of the two lanes' values (s + n).
struct Kahan2 {
    f32x2 s, n;
    __device__ __forceinline__ void add(f32x2 x) {
        const f32x2 y = add2(x, n);
        const f32x2 t = add2(s, y);
        n = add2(y, sub2(s, t));
        s = t;
    }
};

// Sum of a chunk's weights to about 2^-40 of itself, four operations a value:
// s starts at a bias far above the weights, so that the fast form of the
// error-free sum holds from the first one on (weights grow along a bin's
// start), and the errors are summed in n.
struct WeightSum {
    float bias;
    f32x2 s, n;
    __device__ __forceinline__ void start(f32x2 w) {
        bias = 4096.0f * w.x;
        s = dup2(bias);
        n = f32x2{0.f, 0.f};
    }
    __device__ __forceinline__ void add(f32x2 x) {
        const f32x2 t = add2(s, x);
        n = add2(n, add2(sub2(s, t), x));
        s = t;
    }
    // both lanes, as a float pair
    __device__ __forceinline__ float2 total() const {
        return ff_add(make_float2(__fsub_rn(s.x, bias), n.x), make_float2(__fsub_rn(s.y, bias), n.y));
    }
};

// s = sin r, h = cos r - 1 on |r| <= pi/2 + kSwing, for N packed arguments
// stepped together (neighbouring instructions share a coefficient).
template <int N>
__device__ __forceinline__ void sinh2(const f32x2 (&r)[N], f32x2 (&s)[N], f32x2 (&h)[N]) {
    f32x2 u[N], p[N], c[N];
#define GNA_STEP(expr)                 \
    _Pragma("unroll") for (int i = 0; i < N; i++) { \
        expr;                          \
    }
    GNA_STEP(u[i] = mul2(r[i], r[i]))
    GNA_STEP(p[i] = fma2(dup2(GNA_SINA_C4), u[i], dup2(GNA_SINA_C3)))
    GNA_STEP(c[i] = fma2(dup2(GNA_COSA_C5), u[i], dup2(GNA_COSA_C4)))
    GNA_STEP(p[i] = fma2(p[i], u[i], dup2(GNA_SINA_C2)))
    GNA_STEP(c[i] = fma2(c[i], u[i], dup2(GNA_COSA_C3)))
    GNA_STEP(p[i] = fma2(p[i], u[i], dup2(GNA_SINA_C1)))
    GNA_STEP(c[i] = fma2(c[i], u[i], dup2(GNA_COSA_C2)))
    GNA_STEP(s[i] = mul2(r[i], u[i]))
    GNA_STEP(c[i] = fma2(c[i], u[i], dup2(GNA_COSA_C1)))
    GNA_STEP(s[i] = fma2(s[i], p[i], r[i]))
    GNA_STEP(h[i] = mul2(c[i], u[i]))
#undef GNA_STEP
}

// (s, h) of r1 + r2: sin = s1 + s2 + s1 h2 + h1 s2, cos - 1 = h1 + h2 + h1 h2 - s1 s2.
template <bool SIN>
__device__ __forceinline__ void angle_add2(f32x2 s1, f32x2 h1, f32x2 s2, f32x2 h2, f32x2& s, f32x2& h) {
    if constexpr (SIN) s = fma2(h1, s2, fma2(s1, h2, add2(s1, s2)));
    h = fma2(neg2(s1), s2, fma2(h1, h2, add2(h1, h2)));
}

// Multiple q of the unit 1 / inv = a + b (a of 8 bits) nearest to a phase p + lo
// beyond kFarPhase, where one rounding of p inv no longer gives it: the rounding
// of p inv and lo are no longer small against the polynomials' range, and the
// magic number ends at 2^22 (the quotients are doubled phases': twice those of
// reduce_pi_ff).  Its integer, then the rest's.  Good to q < 2^24.
constexpr float kFarPhase = 1e5f;
__device__ __forceinline__ float far_quotient(float p, float lo, float inv, float a, float b) {
    const float q = rintf(__fmul_rn(p, inv));
    return q + rintf(__fmul_rn(__fadd_rn(__fmaf_rn(-q, b, __fmaf_rn(-q, a, p)), lo), inv));
}

// Phase c * e reduced modulo pi (as reduce_pi_ff / reduce_pi_f64) and the
// parity of the multiple of pi as a float's sign bit.  FAR: of any size
// (anchors lie below kFarPhase, chunk_quads).
template <bool FAR>
__device__ __forceinline__ float reduce_sign_ff(float ch, float cl, float eh, float el, unsigned& sign) {
    const float p = __fmul_rn(ch, eh);
    const float e = __fmaf_rn(ch, eh, -p);
    const float lo = __fmaf_rn(ch, el, __fmaf_rn(cl, eh, e));
    const float qm = __fmaf_rn(p, GNA_INV_PI_F, GNA_ROUND_MAGIC);
    sign = __float_as_uint(qm) << 31;
    float q = __fsub_rn(qm, GNA_ROUND_MAGIC);
    if (FAR && fabsf(p) > kFarPhase) {
        q = far_quotient(p, lo, GNA_INV_PI_F, GNA_PI_A, GNA_PI_B2);
        sign = (unsigned)__float2int_rn(q) << 31;
    }
    float r = __fmaf_rn(-q, GNA_PI_A, p);
    r = __fmaf_rn(-q, GNA_PI_B2, r);
    return __fadd_rn(r, lo);
}
__device__ __forceinline__ float reduce_sign_f64(double c, double e, unsigned& sign) {
    const double p = c * e;
    const double qm = fma(p, GNA_INV_PI_D, 6755399441055744.0);  // 1.5 2^52 rounds to an integer
    sign = (unsigned)__double2loint(qm) << 31;
    const double q = qm - 6755399441055744.0;
    double r = fma(-q, GNA_PI_DA, p);
    r = fma(-q, GNA_PI_DB, r);
    return (float)fma(-q, GNA_PI_DC, r);
}

// The doubled phase of baseline r's pair 21 or 32 at 1/E = eh + el.
template <int PH, bool FAR>
__device__ __forceinline__ float phase(const PointConst* pc, int r, bool p32, float eh, float el, unsigned& sign) {
    if constexpr (PH == 0) {
        const float ch = p32 ? pc->c32h[r] : pc->c21h[r], cl = p32 ? pc->c32l[r] : pc->c21l[r];
        return reduce_sign_ff<FAR>(2.0f * ch, 2.0f * cl, eh, el, sign);
    } else {
        return reduce_sign_f64(2.0 * (p32 ? pc->c32[r] : pc->c21[r]), (double)eh + (double)el, sign);
    }
}

// Quads per chunk of a task of nq quads: at most kChunkQuads, and few enough
// that no node lies further than `swing` from the anchor; 0: a quad's own
// nodes already do, or (double-float phases) phases exceed kFarPhase, which
// the anchors' reduction does not take.  Chunks of a task are made about
// equally long.
template <int PH>
__device__ __forceinline__ int chunk_quads(float cmax, float2 step, int nq, float swing) {
    if (PH == 0 && 2.0f * cmax * step.y > kFarPhase) return 0;
    // the anchor is node 2 len of the chunk: a node lies at most 2 len steps from it
    const float lf = swing / (4.0f * cmax * step.x);
    if (!(lf >= 1.0f)) return 0;
    const int most = lf >= (float)kChunkQuads ? kChunkQuads : (int)lf;
    const int nch = (nq + most - 1) / most;
    return (nq + nch - 1) / nch;
}

// ---------------------------------------------------------------- tasks --
// A task's nodes: nq quads of neighbouring nodes per lane.  The plan stores,
// per group of 32 bins and quad, three rows of 32 float4 (one per bin): the
// high parts of 1/E, W, the low parts of 1/E; quads past an odd order's end
// repeat its last node with W = 0.
constexpr int kQuadBytes = 3 * 512;

struct NodeTask {
    int p, b, nq;     // point, group of 32 bins, quads
    const char* rec;  // first quad
    float2 step;      // largest step of 1/E between neighbouring nodes of the group's bins, and largest 1/E
};

__device__ __forceinline__ NodeTask node_task(const BinArgs& a, int t) {
    NodeTask k;
    if (a.S > 1) {
        const int per_point = a.ngroups * a.S;
        k.p = t / per_point;
        const int rem = t - k.p * per_point;
        k.b = rem / a.S;
        const int k0 = (rem - k.b * a.S) * a.L;
        const int n = (a.gn[0] + 3) >> 2;
        k.nq = min(n, k0 + a.L) - k0;
        k.rec = a.rec + ((int64_t)k.b * n + k0) * kQuadBytes;
        k.step = a.step[k.b];
    } else {
        const BinTask d = a.desc[t];
        k.p = d.p;
        k.b = d.b;
        k.nq = d.nq;
        k.rec = a.rec + d.quad * kQuadBytes;
        k.step = d.step;
    }
    return k;
}

struct NodePair {
    f32x2 e, w, l;  // 1/E (high parts), W, 1/E (low parts) of two neighbouring nodes
};

// The task's quads in order, through a ring of R quads per lane in shared
// memory: R - 1 quads are on their way while one is used.  Each lane copies
// and reads its own slots only, so waiting for its own copies suffices.
template <int R>
struct QuadRing {
    static constexpr unsigned kWarpBytes = R * kQuadBytes;
    unsigned base, put, get;  // shared addresses: ring, next slot to fill, next to use
    const char* src;          // this lane's next quad to copy
    int left;                 // quads not yet copied

    __device__ __forceinline__ QuadRing(void* rings) {
        base = put = get = (unsigned)__cvta_generic_to_shared(rings) + (threadIdx.x >> 5) * kWarpBytes +
                           (threadIdx.x & 31) * 16;
    }
    __device__ __forceinline__ void copy() {
        if (left > 0) {
            asm volatile(
                "cp.async.cg.shared.global [%0], [%1], 16;\n\tcp.async.cg.shared.global [%0 + 512], [%1 + 512], 16;\n\t"
                "cp.async.cg.shared.global [%0 + 1024], [%1 + 1024], 16;" ::"r"(put), "l"(src) : "memory");
            src += kQuadBytes;
            left--;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        put += kQuadBytes;
        if (put == base + kWarpBytes) put = base;
    }
    __device__ __forceinline__ void start(const NodeTask& k) {
        src = k.rec + (threadIdx.x & 31) * 16;
        left = k.nq;
        put = get = base;
#pragma unroll
        for (int u = 0; u < R - 1; u++) copy();
    }
    // wait() makes the next quad readable, pair(u) reads its half u, done()
    // gives its slot back.
    __device__ __forceinline__ void wait() { asm volatile("cp.async.wait_group %0;" ::"n"(R - 2) : "memory"); }
    __device__ __forceinline__ NodePair pair(int u) const {
        NodePair n;
        const unsigned at = get + u * 8;
        asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(n.e.x), "=f"(n.e.y) : "r"(at) : "memory");
        asm volatile("ld.shared.v2.f32 {%0, %1}, [%2 + 512];" : "=f"(n.w.x), "=f"(n.w.y) : "r"(at) : "memory");
        asm volatile("ld.shared.v2.f32 {%0, %1}, [%2 + 1024];" : "=f"(n.l.x), "=f"(n.l.y) : "r"(at) : "memory");
        return n;
    }
    __device__ __forceinline__ void done() {
        get += kQuadBytes;
        if (get == base + kWarpBytes) get = base;
        copy();
    }
};

// 1/E of the anchor of a chunk of len quads from quad j on: its node 2 len.
__device__ __forceinline__ float2 load_anchor(const NodeTask& k, int j, int len) {
    const char* at = k.rec + (int64_t)(j + (len >> 1)) * kQuadBytes + (threadIdx.x & 31) * 16 + (len & 1) * 8;
    return make_float2(__ldg(reinterpret_cast<const float*>(at)), __ldg(reinterpret_cast<const float*>(at + 1024)));
}

// Warp tasks.  Slices all take the same time and are about as many as the
// resident warps: warp w takes tasks w, w + warps, ....  Whole bins come from
// the counter (uneven grids, longest first); where there are many per warp
// the next one is asked for while the present one runs (the answer takes as
// long as a dozen nodes; with few per warp the early ones would take them all).
struct TaskQueue {
    int* counter;  // NULL: static
    int asked;     // dynamic: lane 0 holds the next task; static: the next task
    int warps;
    bool ahead;
    __device__ __forceinline__ explicit TaskQueue(const BinArgs& a) {
        warps = gridDim.x * (blockDim.x >> 5);
        counter = a.S > 1 ? nullptr : a.counter;
        ahead = a.ntasks > 8 * warps;
        asked = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5) - (counter ? 0 : warps);
        if (ahead) ask();
    }
    __device__ __forceinline__ void ask() {
        if (counter && (threadIdx.x & 31) == 0) asked = atomicAdd(counter, 1);
    }
    // the next task; call prefetch() when it is taken on
    __device__ __forceinline__ int take() {
        if (!counter) return asked += warps;
        if (!ahead) ask();
        return __shfl_sync(0xffffffffu, asked, 0);
    }
    __device__ __forceinline__ void prefetch() {
        if (ahead) ask();
    }
    // whether the next task may be fixed before the present one ends
    __device__ __forceinline__ bool early() const { return ahead || !counter; }
};

// Task sums over the baselines: T and N of the three pairs weighted by
// omega_r (N by omega_r K L_r).
struct TaskSums {
    float2 T[3], N[3];
};

// Unevaluated product of two float pairs (not normalised).
__device__ __forceinline__ float2 ff_mul(float ah, float al, float2 b) {
    const float p = __fmul_rn(ah, b.x);
    const float e = __fmaf_rn(ah, b.x, -p);
    return make_float2(p, __fmaf_rn(ah, b.y, __fmaf_rn(al, b.x, e)));
}

// sum_ij A_ij/2 T_ij
__device__ __forceinline__ float2 spectrum_part(const PointConst* pc, const float2 (&T)[3]) {
    float2 s = ff_mul(0.5f * pc->Af[0], 0.5f * pc->Alo[0], T[0]);
    s = ff_add(s, ff_mul(0.5f * pc->Af[1], 0.5f * pc->Alo[1], T[1]));
    return ff_add(s, ff_mul(0.5f * pc->Af[2], 0.5f * pc->Alo[2], T[2]));
}

// a . t: products and sums in FP32, the low parts of the factors added first.
template <int N>
__device__ __forceinline__ float dot_pairs(const float* hi, const float* lo, const float2* t) {
    float s = 0.f;
#pragma unroll
    for (int j = 0; j < N; j++) s = fmaf(hi[j], t[j].y, fmaf(lo[j], t[j].x, s));
#pragma unroll
    for (int j = N - 1; j >= 0; j--) s = fmaf(hi[j], t[j].x, s);
    return s;
}

// A bin's prediction and its derivatives from its sums.
template <bool GRAD>
__device__ __forceinline__ BinSums<GRAD ? 4 : 0> bin_sums(const PointConst* pc, float2 sumw, const TaskSums& q) {
    BinSums<GRAD ? 4 : 0> b;
    const float2 x = spectrum_part(pc, q.T);
    b.M = ff_add(sumw, make_float2(-x.x, -x.y));
    if constexpr (GRAD) {
        // dA12's last two are opposite: their sums' difference first (one bin of
        // 50 nodes at 3 MeV, eight baselines of 0.9 - 45 km, error of dM / d s2_12
        // in units of its rms: 5.4e-7 with three terms in FP32, 6.6e-8 so)
        const float2 D = make_float2((q.T[1].x - q.T[2].x) + (q.T[1].y - q.T[2].y), 0.f), TD[2] = {q.T[0], D};
        b.d[0] = -0.5f * dot_pairs<2>(pc->dA12f, pc->dA12lo, TD);
        b.d[1] = -0.5f * dot_pairs<3>(pc->dA13f, pc->dA13lo, q.T);
        b.d[2] = -dot_pairs<2>(pc->Af, pc->Alo, q.N);
        b.d[3] = -dot_pairs<2>(pc->Af + 1, pc->Alo + 1, q.N + 1);
    }
    return b;
}

// Stores the task sums for the slice reduction: T (3 pairs), N (3), as float pairs.
template <bool GRAD>
__device__ __forceinline__ void store_sums(const TaskSums& q, float2* pp) {
#pragma unroll
    for (int j = 0; j < 3; j++) pp[j * 32] = q.T[j];
    if constexpr (GRAD) {
#pragma unroll
        for (int j = 0; j < 3; j++) pp[(3 + j) * 32] = q.N[j];
    }
}

// A whole-bin task's end: this lane's bin through the epilogue, then the
// sums of the warp's group (a kernel after this one sums the groups: counting
// them here, as the split mapping does, would cost every task a fence and the
// answer to an atomic).  sp: sum_ij A_ij/2 T_ij,r per baseline (spectra).
template <bool GRAD>
__device__ __forceinline__ void finish_bins(const BinArgs& a, int p, int b, const TaskSums& q, const float2* sp,
                                            const BinInput& in, int lane) {
    const int i = b * 32 + lane;
    constexpr int NG = GRAD ? 4 : 0;
    float2 regs[1 + NG];
    if (i < a.nbins) bin_terms<NG>(a.ea, p, i, bin_sums<GRAD>(a.pcs + p, in.sumw, q), sp, in, regs);
    group_terms<NG>(a.ea, p, b, lane, regs);
}

// ------------------------------------------------ several baselines ------
// 2 NP baselines at a time, two per packed value; a plan with more takes the
// nodes again for the next ones.  The task's compensated sums live in shared
// memory (touched once per chunk), so the registers hold the chunk's sums,
// the anchors and the constants of all 2 NP baselines: 168 registers, three
// blocks of 128 threads per SM.
template <int PH, int NP, bool GRAD>
struct MultiMath {
    static constexpr int NS = GRAD ? 6 : 3;  // sums per baseline: T, N of three pairs
    f32x2 c[2 * NP];         // 2c of pairs 21, 32
    f32x2 a[2 * NP];         // anchors' reduced phases
    f32x2 acc[NP][NS];

    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int i = 0; i < NP; i++)
#pragma unroll
            for (int v = 0; v < NS; v++) acc[i][v] = f32x2{0.f, 0.f};
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

    // Anchors at 1/E = (eh, el); bit 4i + h (+ 2) of the result: parity of
    // pair 21 (32) of baseline 2i + h.
    __device__ __forceinline__ unsigned anchor(const PointConst* pc, int r0, float eh, float el) {
        unsigned par = 0;
#pragma unroll
        for (int i = 0; i < NP; i++) {
            const int r = r0 + 2 * i;
            unsigned s[4];
            float x[4];
            if constexpr (PH == 0) {
                const float2 l = *reinterpret_cast<const float2*>(pc->c21l + r);
                const float2 m = *reinterpret_cast<const float2*>(pc->c32l + r);
                x[0] = reduce_sign_ff<false>(c[2 * i].x, 2.0f * l.x, eh, el, s[0]);
                x[1] = reduce_sign_ff<false>(c[2 * i].y, 2.0f * l.y, eh, el, s[1]);
                x[2] = reduce_sign_ff<false>(c[2 * i + 1].x, 2.0f * m.x, eh, el, s[2]);
                x[3] = reduce_sign_ff<false>(c[2 * i + 1].y, 2.0f * m.y, eh, el, s[3]);
            } else {
#pragma unroll
                for (int j = 0; j < 4; j++) x[j] = phase<PH, false>(pc, r + (j & 1), j >= 2, eh, el, s[j]);
            }
            a[2 * i] = pack2(x[0], x[1]);
            a[2 * i + 1] = pack2(x[2], x[3]);
            par |= ((s[0] >> 31) | (s[1] >> 30) | (s[2] >> 29) | (s[3] >> 28)) << (4 * i);
        }
        return par;
    }

    // One node: offset d from the anchor, weights W and W/E.
    __device__ __forceinline__ void node(float d, float W, float We) {
        const f32x2 d2 = dup2(d), W2 = dup2(W), We2 = dup2(We);
        f32x2 r[2 * NP], s[2 * NP], h[2 * NP];
#pragma unroll
        for (int i = 0; i < 2 * NP; i++) r[i] = fma2(c[i], d2, a[i]);
        sinh2(r, s, h);
#pragma unroll
        for (int i = 0; i < NP; i++) {
            f32x2 s3, h3;
            angle_add2<GRAD>(s[2 * i], h[2 * i], s[2 * i + 1], h[2 * i + 1], s3, h3);
            acc[i][0] = fma2(W2, h[2 * i], acc[i][0]);
            acc[i][1] = fma2(W2, h3, acc[i][1]);
            acc[i][2] = fma2(W2, h[2 * i + 1], acc[i][2]);
            if constexpr (GRAD) {
                acc[i][3] = fma2(We2, s[2 * i], acc[i][3]);
                acc[i][4] = fma2(We2, s3, acc[i][4]);
                acc[i][5] = fma2(We2, s[2 * i + 1], acc[i][5]);
            }
        }
    }

    __device__ __forceinline__ void pair(const NodePair& n, f32x2 nah, f32x2 nal) {
        const f32x2 d = add2(add2(n.e, nah), add2(n.l, nal)), we = mul2(n.w, n.e);
        node(d.x, n.w.x, we.x);
        node(d.y, n.w.y, we.y);
    }

    // A node with its phases reduced.  T is summed as if q were even, with
    // -h for odd q, and the odd weights apart (in odd).
    __device__ __forceinline__ void node_direct(const PointConst* pc, int r0, float eh, float el, float W,
                                                f32x2 (&odd)[NP][3]) {
        const f32x2 W2 = dup2(W), We2 = dup2(W * eh);
#pragma unroll
        for (int i = 0; i < NP; i++) {
            unsigned q[4];
            f32x2 r[2], s[2], h[2], s3, h3;
#pragma unroll
            for (int j = 0; j < 2; j++)
                r[j] = pack2(phase<PH, true>(pc, r0 + 2 * i, j == 1, eh, el, q[2 * j]),
                             phase<PH, true>(pc, r0 + 2 * i + 1, j == 1, eh, el, q[2 * j + 1]));
            sinh2(r, s, h);
            angle_add2<true>(s[0], h[0], s[1], h[1], s3, h3);
            const f32x2 S[3] = {s[0], s3, s[1]}, H[3] = {h[0], h3, h[1]};
#pragma unroll
            for (int j = 0; j < 3; j++) {
                const unsigned x = j == 0 ? q[0] : j == 2 ? q[2] : q[0] ^ q[2];
                const unsigned y = j == 0 ? q[1] : j == 2 ? q[3] : q[1] ^ q[3];
                const f32x2 sg = pack2(__uint_as_float(0x3f800000u ^ x), __uint_as_float(0x3f800000u ^ y));
                acc[i][j] = fma2(mul2(sg, W2), H[j], acc[i][j]);
                odd[i][j] = pack2(x ? W : 0.f, y ? W : 0.f);
                if constexpr (GRAD) acc[i][3 + j] = fma2(mul2(sg, We2), S[j], acc[i][3 + j]);
            }
        }
    }

    // Adds to T (pair j of i) the value sg * acc + big + lo.
    static __device__ __forceinline__ void add_T(f32x2p* at, f32x2 sg, f32x2 x, f32x2 big, f32x2 lo, bool first) {
        const f32x2 hi = fma2(sg, x, big);
        // what the rounding to hi dropped (|big| >= |x|, or big = 0)
        f32x2p t{hi, add2(fma2(sg, x, sub2(big, hi)), lo)};
        if (!first) t = ff_add2(*at, t);
        *at = t;
    }
    static __device__ __forceinline__ void add_N(f32x2p* at, f32x2 x, bool first) {
        Kahan2 k{x, f32x2{0.f, 0.f}};
        if (!first) {
            const f32x2p y = *at;
            k.s = y.x;
            k.n = y.y;
            k.add(x);
        }
        *at = f32x2p{k.s, k.n};
    }

    // Adds the chunk's sums to the task's (in shared memory); par: parities,
    // cw: 2 sum W of the chunk.
    __device__ __forceinline__ void flush(f32x2p* comp, int stride, unsigned par, float2 cw, bool first) {
#pragma unroll
        for (int i = 0; i < NP; i++) {
            const unsigned b = par >> (4 * i);
            const unsigned o[3] = {b & 3u, (b ^ (b >> 2)) & 3u, (b >> 2) & 3u};
#pragma unroll
            for (int j = 0; j < 3; j++) {
                const unsigned x0 = o[j] << 31, x1 = (o[j] >> 1) << 31;
                // T: -acc (even) or 2 sum W + acc (odd); N: acc (even) or -acc
                const f32x2 sg = pack2(__uint_as_float(0xbf800000u ^ x0), __uint_as_float(0xbf800000u ^ x1));
                add_T(comp + (i * NS + j) * stride, sg, acc[i][j], pack2(x0 ? cw.x : 0.f, x1 ? cw.x : 0.f),
                      pack2(x0 ? cw.y : 0.f, x1 ? cw.y : 0.f), first);
                if constexpr (GRAD) add_N(comp + (i * NS + 3 + j) * stride, mul2(neg2(sg), acc[i][3 + j]), first);
            }
        }
        zero();
    }
    __device__ __forceinline__ void flush_direct(f32x2p* comp, int stride, const f32x2 (&odd)[NP][3], bool first) {
#pragma unroll
        for (int i = 0; i < NP; i++)
#pragma unroll
            for (int j = 0; j < 3; j++) {
                f32x2p t = ff_add2(f32x2p{mul2(dup2(2.0f), odd[i][j]), f32x2{0.f, 0.f}},
                                   f32x2p{neg2(acc[i][j]), f32x2{0.f, 0.f}});
                f32x2p* at = comp + (i * NS + j) * stride;
                if (!first) t = ff_add2(*at, t);
                *at = t;
                if constexpr (GRAD) add_N(comp + (i * NS + 3 + j) * stride, acc[i][3 + j], first);
            }
        zero();
    }
};

template <int PH, int NP, bool GRAD>
__global__ void __maxnreg__(NP >= 3 ? 168 : 128) k_nodes_multi(BinArgs a) {
    using M = MultiMath<PH, NP, GRAD>;
    extern __shared__ f32x2p comp_all[];  // [NP * NS][blockDim], then the rings
    f32x2p* comp = comp_all + threadIdx.x;
    const int stride = blockDim.x;
    const int lane = threadIdx.x & 31;
    QuadRing<kRingMulti> in(comp_all + NP * M::NS * stride);
    // a programmatic dependent of the kernel that prepares the per-point
    // constants and zeroes the counters: wait (in hardware) for it here
    asm volatile("griddepcontrol.wait;" ::: "memory");
    TaskQueue queue(a);
    for (int t = queue.take(); t < a.ntasks; t = queue.take()) {
        queue.prefetch();
        const NodeTask k = node_task(a, t);
        const PointConst* pc = a.pcs + k.p;
        const bool whole = a.S <= 1;
        BinInput bin;
        if (whole) bin = bin_input(a.ea, k.p, min(k.b * 32 + lane, a.nbins - 1));
        const int len = chunk_quads<PH>(pc->cmax, k.step, k.nq, kSwing);
        const bool direct = len == 0;
        const int step = direct ? 1 : len;
        // the spectra's parts, and the sums q between two passes over the nodes
        // (in local memory: the node loop needs the registers)
        float2 sp[GNA_NLMAX + 6];
        float2* pp = whole ? nullptr : a.part + (int64_t)t * a.NVs * 32 + lane;
        for (int r0 = 0; r0 < a.nL; r0 += 2 * NP) {
            M x;
            in.start(k);
            x.load(pc, r0);
            x.zero();
            float2 an = load_anchor(k, 0, min(step, k.nq));
            for (int ka = 0; ka < k.nq; ka += step) {
                const int kb = min(k.nq, ka + step);
                if (!direct) {
                    const unsigned par = x.anchor(pc, r0, an.x, an.y);
                    const f32x2 nah = dup2(-an.x), nal = dup2(-an.y);
                    if (kb < k.nq) an = load_anchor(k, kb, min(step, k.nq - kb));
                    WeightSum w;
                    in.wait();
                    w.start(in.pair(0).w);
#pragma unroll 1
                    for (int j = ka; j < kb; j++) {
                        in.wait();
#pragma unroll 1
                        for (int u = 0; u < 2; u++) {
                            const NodePair n = in.pair(u);
                            w.add(n.w);
                            x.pair(n, nah, nal);
                        }
                        in.done();
                    }
                    float2 cw = w.total();
                    cw.x *= 2.0f;
                    cw.y *= 2.0f;
                    x.flush(comp, stride, par, cw, ka == 0);
                } else {
                    // each node is added to the compensated sums by itself: few
                    // nodes do not average the roundings of a quad's FP32 sums
                    // (20 bins x 14 nodes x 12, median of 24 inputs against 64 bits:
                    // chi^2 5.5e-7 -> 7.0e-8, gradient 3.7e-7 -> 5.3e-8; no time)
                    f32x2 odd[NP][3];
                    in.wait();
#pragma unroll 1
                    for (int u = 0; u < 4; u++) {
                        const NodePair n = in.pair(u >> 1);
                        x.node_direct(pc, r0, (u & 1) ? n.e.y : n.e.x, (u & 1) ? n.l.y : n.l.x, (u & 1) ? n.w.y : n.w.x, odd);
                        x.flush_direct(comp, stride, odd, ka == 0 && u == 0);
                    }
                    in.done();
                }
            }
            TaskSums q;
#pragma unroll
            for (int j = 0; j < 3; j++) {
                q.T[j] = r0 ? sp[GNA_NLMAX + j] : make_float2(0.f, 0.f);
                q.N[j] = r0 ? sp[GNA_NLMAX + 3 + j] : make_float2(0.f, 0.f);
            }
            // (a loop: eight baselines' code would be fetched for one use a task)
#pragma unroll 1
            for (int i = 0; i < 2 * NP && r0 + i < a.nL; i++) {
                const int r = r0 + i;
                const float* f = reinterpret_cast<const float*>(comp + (i >> 1) * M::NS * stride) + (i & 1);
                const int w = stride * 4;
                float2 T[3];
#pragma unroll
                for (int j = 0; j < 3; j++) {
                    T[j] = make_float2(f[j * w], f[j * w + 2]);
                    q.T[j] = ff_add(q.T[j], ff_mul(a.bc.om[r], a.bc.omlo[r], T[j]));
                    if constexpr (GRAD) {
                        const float2 n = make_float2(f[(3 + j) * w], f[(3 + j) * w + 2]);
                        q.N[j] = ff_add(q.N[j], ff_mul(0.5f * a.bc.wkl[r], 0.5f * a.bc.wkllo[r], n));
                    }
                }
                if (a.spec) {
                    const float2 part = spectrum_part(pc, T);
                    if (pp) pp[(M::NS + r) * 32] = part;
                    else sp[r] = part;
                }
            }
            if (r0 + 2 * NP < a.nL) {
#pragma unroll
                for (int j = 0; j < 3; j++) {
                    sp[GNA_NLMAX + j] = q.T[j];
                    sp[GNA_NLMAX + 3 + j] = q.N[j];
                }
            } else if (pp) store_sums<GRAD>(q, pp);
            else finish_bins<GRAD>(a, k.p, k.b, q, sp, bin, lane);
        }
    }
    asm volatile("griddepcontrol.launch_dependents;");
}

// ---------------------------------------------------- one baseline -------
// Two neighbouring nodes per packed value; the sums stay in registers.
template <int PH, bool GRAD>
struct OneMath {
    static constexpr int NS = GRAD ? 6 : 3;
    f32x2 c21, c32, a21, a32;
    f32x2 acc[NS];

    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int v = 0; v < NS; v++) acc[v] = f32x2{0.f, 0.f};
    }

    // NU pairs together.
    template <int NU>
    __device__ __forceinline__ void pairs(const NodePair (&n)[NU], f32x2 nah, f32x2 nal) {
        f32x2 r[2 * NU], s[2 * NU], h[2 * NU];
#pragma unroll
        for (int u = 0; u < NU; u++) {
            const f32x2 d = add2(add2(n[u].e, nah), add2(n[u].l, nal));
            r[u] = fma2(c21, d, a21);
            r[NU + u] = fma2(c32, d, a32);
        }
        sinh2(r, s, h);
#pragma unroll
        for (int u = 0; u < NU; u++) {
            f32x2 s3, h3;
            angle_add2<GRAD>(s[u], h[u], s[NU + u], h[NU + u], s3, h3);
            acc[0] = fma2(n[u].w, h[u], acc[0]);
            acc[1] = fma2(n[u].w, h3, acc[1]);
            acc[2] = fma2(n[u].w, h[NU + u], acc[2]);
            if constexpr (GRAD) {
                const f32x2 we = mul2(n[u].w, n[u].e);
                acc[3] = fma2(we, s[u], acc[3]);
                acc[4] = fma2(we, s3, acc[4]);
                acc[5] = fma2(we, s[NU + u], acc[5]);
            }
        }
    }

    // As MultiMath::node_direct, for the two nodes of a pair.
    __device__ __forceinline__ void pair_direct(const PointConst* pc, f32x2 e, f32x2 l, f32x2 w, f32x2 (&odd)[3]) {
        unsigned q[4];
        f32x2 r[2], s[2], h[2], s3, h3;
#pragma unroll
        for (int j = 0; j < 2; j++)
            r[j] = pack2(phase<PH, true>(pc, 0, j == 1, e.x, l.x, q[2 * j]),
                         phase<PH, true>(pc, 0, j == 1, e.y, l.y, q[2 * j + 1]));
        sinh2(r, s, h);
        angle_add2<true>(s[0], h[0], s[1], h[1], s3, h3);
        const f32x2 we = mul2(w, e), S[3] = {s[0], s3, s[1]}, H[3] = {h[0], h3, h[1]};
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const unsigned x = j == 0 ? q[0] : j == 2 ? q[2] : q[0] ^ q[2];
            const unsigned y = j == 0 ? q[1] : j == 2 ? q[3] : q[1] ^ q[3];
            const f32x2 sg = pack2(__uint_as_float(0x3f800000u ^ x), __uint_as_float(0x3f800000u ^ y));
            acc[j] = fma2(mul2(sg, w), H[j], acc[j]);
            odd[j] = pack2(x ? w.x : 0.f, y ? w.y : 0.f);
            if constexpr (GRAD) acc[3 + j] = fma2(mul2(sg, we), S[j], acc[3 + j]);
        }
    }
};

// The next task is prepared while the present one runs, so that nothing of it
// has to be waited for: its number is asked for a task ahead, its description
// loaded at the present task's start, the point's constant at its end, and its
// first nodes and anchor are on their way during the present task's epilogue.
// 128 registers: four blocks of 128 threads per SM (112 hold no more of them
// and spill; scan of 4096 points 654 -> 640 us).
template <int PH, bool GRAD>
__global__ void __maxnreg__(128) k_nodes_one(BinArgs a) {
    using M = OneMath<PH, GRAD>;
    constexpr int NS = M::NS;
    const int lane = threadIdx.x & 31;
    extern __shared__ f32x2p rings[];
    QuadRing<kRingOne> in(rings);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const bool whole = a.S <= 1;
    TaskQueue queue(a);
    int t = queue.take();
    if (t < a.ntasks) {
        queue.prefetch();
        NodeTask k = node_task(a, t);
        in.start(k);
        int len = chunk_quads<PH>(a.pcs[k.p].cmax, k.step, k.nq, kSwing);
        float2 an = load_anchor(k, 0, min(max(len, 1), k.nq));
        while (true) {
            int tn = a.ntasks;
            NodeTask kn = k;
            if (queue.early()) {
                tn = queue.take();
                if (tn < a.ntasks) {
                    kn = node_task(a, tn);
                    queue.prefetch();
                }
            }
            const PointConst* pc = a.pcs + k.p;
            BinInput bin;
            if (whole) bin = bin_input(a.ea, k.p, min(k.b * 32 + lane, a.nbins - 1));
            const bool direct = len == 0;
            const int step = direct ? 1 : len;
            M x;
            x.c21 = dup2(2.0f * pc->c21h[0]);
            x.c32 = dup2(2.0f * pc->c32h[0]);
            x.zero();
            TaskSums q;
            KahanF N[3];
#pragma unroll
            for (int v = 0; v < 3; v++) {
                q.T[v] = make_float2(0.f, 0.f);
                kzero(N[v]);
            }
            for (int ka = 0; ka < k.nq; ka += step) {
                const int kb = min(k.nq, ka + step);
                if (!direct) {
                    unsigned q21, q32;
                    x.a21 = dup2(phase<PH, false>(pc, 0, false, an.x, an.y, q21));
                    x.a32 = dup2(phase<PH, false>(pc, 0, true, an.x, an.y, q32));
                    const f32x2 nah = dup2(-an.x), nal = dup2(-an.y);
                    if (kb < k.nq) an = load_anchor(k, kb, min(step, k.nq - kb));
                    WeightSum w;
                    in.wait();
                    w.start(in.pair(0).w);
#pragma unroll 1
                    for (int j = ka; j < kb; j++) {
                        in.wait();
                        const NodePair n[2] = {in.pair(0), in.pair(1)};
                        w.add(n[0].w);
                        w.add(n[1].w);
                        x.pairs(n, nah, nal);
                        in.done();
                    }
                    const float2 cw = w.total();
                    const unsigned o[3] = {q21, q21 ^ q32, q32};
#pragma unroll
                    for (int v = 0; v < 3; v++) {
                        // T: -acc (even) or 2 sum W + acc (odd); N: acc (even) or -acc
                        const float c = __uint_as_float(0xbf800000u ^ o[v]) * (x.acc[v].x + x.acc[v].y);
                        const float2 big = o[v] ? make_float2(2.0f * cw.x, 2.0f * cw.y) : make_float2(0.f, 0.f);
                        // (|big| >= |c| or big = 0)
                        const float hi = __fadd_rn(big.x, c);
                        q.T[v] = ff_add(q.T[v], make_float2(hi, __fadd_rn(__fadd_rn(c, __fsub_rn(big.x, hi)), big.y)));
                        if constexpr (GRAD)
                            kadd_prod(N[v], __uint_as_float(0x3f800000u ^ o[v]), x.acc[3 + v].x + x.acc[3 + v].y);
                    }
                } else {
                    in.wait();
#pragma unroll 1
                    for (int u = 0; u < 2; u++) {
                        f32x2 odd[3];
                        const NodePair n = in.pair(u);
                        x.pair_direct(pc, n.e, n.l, n.w, odd);
                        // each node by itself, as k_nodes_multi
#pragma unroll
                        for (int v = 0; v < 3; v++) {
                            auto node = [](float o, float h) { return ff_add(make_float2(2.0f * o, 0.f), make_float2(-h, 0.f)); };
                            q.T[v] = ff_add(q.T[v], ff_add(node(odd[v].x, x.acc[v].x), node(odd[v].y, x.acc[v].y)));
                            if constexpr (GRAD) {
                                kadd_prod(N[v], 1.0f, x.acc[3 + v].x);
                                kadd_prod(N[v], 1.0f, x.acc[3 + v].y);
                            }
                        }
                        x.zero();
                    }
                    in.done();
                }
                x.zero();
            }
            // omega = 1 for one baseline: wkl = 2 K L
#pragma unroll
            for (int v = 0; v < 3; v++) q.N[v] = ff_mul(0.5f * a.bc.wkl[0], 0.5f * a.bc.wkllo[0], kahan_to_ff(N[v]));
            const int t0 = t, p0 = k.p, b0 = k.b;
            if (!queue.early()) {
                tn = queue.take();
                if (tn < a.ntasks) kn = node_task(a, tn);
            }
            const bool more = tn < a.ntasks;
            if (more) {
                t = tn;
                k = kn;
                in.start(k);
                len = chunk_quads<PH>(a.pcs[k.p].cmax, k.step, k.nq, kSwing);
                an = load_anchor(k, 0, min(max(len, 1), k.nq));
            }
            float2 sp[1];
            if (a.spec) sp[0] = spectrum_part(pc, q.T);
            if (!whole) {
                float2* pp = a.part + (int64_t)t0 * a.NVs * 32 + lane;
                store_sums<GRAD>(q, pp);
                if (a.spec) pp[NS * 32] = sp[0];
            } else {
                finish_bins<GRAD>(a, p0, b0, q, sp, bin, lane);
            }
            if (!more) break;
        }
    }
    asm volatile("griddepcontrol.launch_dependents;");
}

}  // namespace gna
