// oscprob.cu -- element-wise OscProb (paper Sec. 4.1): the nu_e survival
// probability
//   P = 1 - sum_ij A_ij sin^2 x_ij,
// and the general vacuum formula for any channel, neutrinos and
// antineutrinos, with theta23 and the CP phase:
//   P(a -> b) = delta_ab + sum_{i>j} [ -4 Re X_ij sin^2 x_ij + 2 Im X_ij sin 2x_ij ],
//   X_ij = V*_ai V_bi V_aj V*_bj,  V = U (neutrinos) or U* (antineutrinos),
//   x_ij = K dm2_ij L / E.
// The host folds U into the six real coefficients (cr = -4 Re X, ci = 2 Im X)
// per channel; the kernels evaluate three phases per (baseline, energy).
#include <algorithm>
#include <cmath>
#include <mutex>
#include <type_traits>

#include "oscprob.h"

namespace gna {

void turn_constants(const double* c21, const double* c32, int nL, double dab, const double* cr, const double* ci,
                    TurnConst& t) {
    t = TurnConst{};
    double bound = dab;
    for (int q = 0; q < 3; q++) bound += std::fabs(cr[q]) + std::fabs(ci[q]);
    // the bound covers |K| + sum |a| + sum |b|; delta_ab = 1 leaves it below 4,
    // without delta_ab it is brought to 1 .. 2 so that small coefficients keep
    // their leading bits
    int g = 0;
    if (dab == 0.0 && bound > 0.0) {
        std::frexp(bound, &g);
        g = 1 - g;
    }
    if (!(bound < 4.0) || g > 900) return;
    t.scale = g;
    t.K = std::llrint(std::ldexp(dab, 61));
    for (int q = 0; q < 3; q++) {
        const double a = std::ldexp(cr[q], g - 1), b = std::ldexp(ci[q], g);
        if (!(std::fabs(a) < 1.0) || !(std::fabs(b) < 1.0)) return;
        t.a[q] = -std::llrint(std::ldexp(a, 63));
        t.b[q] = std::llrint(std::ldexp(b, 63));
        t.K += std::llrint(std::ldexp(a, 61));
    }
    for (int r = 0; r < nL; r++) {
        TurnCoef &p = t.ph21[r], &q = t.ph32[r];
        if (!turn_coef(c21[r], p) || !turn_coef(c32[r], q)) return;
        if (p.m == 0 && q.m == 0) p.e = q.e = -4096;  // no phase: the double path, P = delta_ab exactly
        if (p.m == 0) p.e = q.e;                       // one zero phase is in range wherever the other one is
        if (q.m == 0) q.e = p.e;
    }
    // Without delta_ab P falls with the square of the phases: an element whose
    // phases are below pi / 32 keeps its relative precision in the double path.
    t.min_shift = dab == 0.0 ? -2 : -32;
    t.ok = 1;
}

namespace {

// ------------------------------------------------------------------ FP64 --
// The double path, for the elements outside turns.cuh's range: energies that
// are not positive normal numbers, phases of more than 2^30 half-turns or next
// to zero, and probabilities next to zero.
__device__ __noinline__ double osc_double(const OscConst& oc, int r, double E) {
    const double e = 1.0 / E;
    const double s21 = sin(oc.c21[r] * e), s32 = sin(oc.c32[r] * e), s31 = sin((oc.c21[r] + oc.c32[r]) * e);
    return 1.0 - oc.A[0] * s21 * s21 - oc.A[1] * s31 * s31 - oc.A[2] * s32 * s32;
}

__device__ __noinline__ double osc_double(const OscGenConst& oc, int r, double E) {
    const double inv = 1.0 / E;
    double p = oc.dab;
#pragma unroll
    for (int q = 0; q < 3; q++) {
        double s, c;
        sincos(oc.c[q][r] * inv, &s, &c);
        p = fma(oc.cr[q], s * s, fma(oc.ci[q], 2.0 * s * c, p));
    }
    return p;
}

__device__ const longlong2 g_turn_table[512] = {GNA_TURN_TABLE};

// Per-element state of the fixed-point phases.
struct ElemTurns {
    TurnRecip rc;
    bool ok;
    __device__ __forceinline__ ElemTurns(const TurnConst& t, double E) {
        const uint32_t hi = (uint32_t)__double2hiint(E), lo = (uint32_t)__double2loint(E);
        rc = turn_recip(hi, lo);
        ok = t.ok && (hi >> 20) - 1u < 2046u;  // positive, neither subnormal nor infinite nor NaN
    }
    // phases 21 and 32 of baseline r (the third is their sum); false: out of range
    __device__ __forceinline__ bool phases(const TurnConst& t, int r, uint64_t& f21, uint64_t& f32) const {
        const int s21 = turn_shift(t.ph21[r].e, rc.e), s32 = turn_shift(t.ph32[r].e, rc.e);
        f21 = turn_phase(t.ph21[r].m, t.ph21[r].neg, rc.y, s21);
        f32 = turn_phase(t.ph32[r].m, t.ph32[r].neg, rc.y, s32);
        return ok && turn_shift_ok(s21) && turn_shift_ok(s32) && max(s21, s32) >= t.min_shift;
    }
};

// The integers carry P to a few units of 2^-61 of its largest value, whatever
// its own size is.  The formula in double is a sum of squares where P has a
// zero (two equal splittings or one that vanishes, maximal mixing): it stays
// at or above zero there and its error, about 2^-50 sqrt(P), falls with P.
// The two errors meet at 2^-16; below it P is taken from the formula.
constexpr int64_t kSmallTurns = 1ll << (61 - 16);

// Everything in 64-bit integers (turns.cuh): what bounds it is the issue of
// some eighty wide integer multiplies and their shifts and additions per
// probability, in place of three double sines (27 FP64 instructions each, at
// 64 cycles a warp).  The table is read from shared memory with its cosine and
// sine side by side; a limited number of blocks walk over the energies, so that
// it is loaded once each.  GB300: 4,000,000 energies at one baseline 529 -> 88 us,
// 3,000,017 at two (mu -> e) 1032 -> 156 us.  Largest error against 113-bit
// arithmetic, 1.8-12 MeV at 52.5 km: 1.5e-15 -> 5.2e-16; 0.5-5 GeV at 810 km,
// mu -> e: 1.9e-16 -> 8.2e-17.
template <class C>
__global__ void __launch_bounds__(256) k_osc_fp64(const double* __restrict__ E, int64_t n, const __grid_constant__ C oc,
                                                  double* __restrict__ P) {
    constexpr bool GEN = std::is_same<C, OscGenConst>::value;
    __shared__ longlong2 tab[512];
    tab[threadIdx.x] = g_turn_table[threadIdx.x];
    tab[threadIdx.x + 256] = g_turn_table[threadIdx.x + 256];
    __syncthreads();
    const int64_t step = (int64_t)gridDim.x * 256;
    for (int64_t k = (int64_t)blockIdx.x * 256 + threadIdx.x; k < n; k += step) {
        const double e = E[k];
        const ElemTurns el(oc.t, e);
        for (int r = 0; r < oc.nL; r++) {
            uint64_t f[3];
            const bool in = el.phases(oc.t, r, f[0], f[2]);
            f[1] = f[0] + f[2];
            int64_t v = oc.t.K;
#pragma unroll
            for (int q = 0; q < 3; q++) {
                int64_t dd, g, s;
                const longlong2 cz = tab[turn_split(f[q], dd)];
                turn_small(dd, g, s);
                const int64_t c = turn_cos(cz.x, cz.y, g, s);
                v += GEN ? mul_hi2(oc.t.a[q], c, oc.t.b[q], turn_sin(cz.x, cz.y, g, s)) : mul_hi(oc.t.a[q], c);
            }
            double p = __ll2double_rn(v);  // P 2^(61 + scale)
            if (v != 0) p = __hiloint2double(__double2hiint(p) - ((61 + oc.t.scale) << 20), __double2loint(p));
            if (!in || v < kSmallTurns) p = osc_double(oc, r, e);
            P[(int64_t)r * n + k] = p;
        }
    }
}

// ----------------------------------------------------------------- mixed --
// 1 / E as a float pair.  E is split by its bits (a conversion from double
// occupies the FP64 unit) while its exponent leaves both halves normal floats;
// the reciprocal is common.cuh's with one more term, r (e + e^2).
__device__ __forceinline__ void elem_recip(double E, float& rh, float& rl) {
    const uint32_t hi = (uint32_t)__double2hiint(E), lo = (uint32_t)__double2loint(E);
    if ((hi >> 20) - (1023u - 64u) > 128u) {
        ff_recip(E, rh, rl);
        return;
    }
    const uint32_t ex = (hi >> 20) - (1023u - 127u);  // float exponent
    const float eh = __uint_as_float(__funnelshift_l(lo, hi, 3) - (896u << 23));
    const float el = __uint2float_rn(lo & 0x1fffffffu) * __uint_as_float((ex - 52u) << 23);
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(eh));
    const float e = fmaf(-el, r, fmaf(-eh, r, 1.0f));
    const float d = r * fmaf(e, e, e);
    rh = r + d;
    rl = d - (rh - r);
}

// Radians of a signed fraction of pi in units of 2^-64, rounded to float: the
// leading 24 bits exactly, the following 32 rounded.
__device__ __forceinline__ float turn_radians(int64_t d) {
    const uint32_t h = (uint32_t)(d >> 32), l = (uint32_t)d;
    const float a = __int2float_rn((int)(h & ~0xffu));
    const float b = __uint2float_rn((h << 24) | (l >> 8));
    constexpr float A = 0x1p-32f * 3.14159274101257324f;  // pi = 3.14159274... - 8.7422777e-8
    constexpr float B = 0x1p-32f * -8.74227765734758577e-8f;
    constexpr float C = 0x1p-56f * 3.14159274101257324f;
    return fmaf(a, A, fmaf(a, B, b * C));
}

// A phase reduced modulo pi/2 with the quadrant's parity, and modulo pi.
__device__ __forceinline__ float turn_half(uint64_t f, int& odd) {
    const uint32_t k = ((uint32_t)(f >> 32) + (1u << 30)) >> 31;
    odd = (int)(k & 1u);
    return turn_radians((int64_t)(f - ((uint64_t)k << 63)));
}

// Survival: each phase reduced modulo pi/2 (quadrant parity q), sin r by the
// FP32 polynomial; sin^2(phase) = s^2 for even q, 1 - s^2 for odd q.  The
// dominant term is written as (1 - A21) + A21 s^2 for odd q so that P stays
// accurate to a few ulp where it is smallest.
__device__ __forceinline__ float reduce_half_pi(float ch, float cl, float eh, float el, int& odd) {
    float p = __fmul_rn(ch, eh);
    float e = __fmaf_rn(ch, eh, -p);
    float lo = __fmaf_rn(ch, el, __fmaf_rn(cl, eh, e));
    float qm = __fmaf_rn(p, 2.0f * GNA_INV_PI_F, GNA_ROUND_MAGIC);
    odd = __float_as_int(qm) & 1;
    float q = __fsub_rn(qm, GNA_ROUND_MAGIC);
    float r = __fmaf_rn(-q, 0.5f * GNA_PI_A, p);
    r = __fmaf_rn(-q, 0.5f * GNA_PI_B, r);
    r = __fmaf_rn(-q, 0.5f * GNA_PI_C, r);
    return __fadd_rn(r, lo);
}

__device__ __forceinline__ float reduce_half_pi_f64(double c, double e, int& odd) {
    double p = c * e;
    double q = rint(p * (2.0 * GNA_INV_PI_D));
    odd = ((long long)q) & 1;
    double r = fma(-q, 0.5 * GNA_PI_DA, p);
    r = fma(-q, 0.5 * GNA_PI_DB, r);
    r = fma(-q, 0.5 * GNA_PI_DC, r);
    return (float)r;
}

__device__ __forceinline__ float mixed_prob(const OscConst& oc, const float (&x)[3], const int (&odd)[3]) {
    const float s21 = sin_poly(x[0]), s31 = sin_poly(x[1]), s32 = sin_poly(x[2]);
    const float q21 = s21 * s21, q31 = s31 * s31, q32 = s32 * s32;
    const float S31 = odd[1] ? 1.0f - q31 : q31;
    const float S32 = odd[2] ? 1.0f - q32 : q32;
    const float base = odd[0] ? fmaf(oc.Af[0], q21, oc.one_minus_A21f) : fmaf(-oc.Af[0], q21, 1.0f);
    return fmaf(-oc.Af[2], S32, fmaf(-oc.Af[1], S31, base));
}

// Any channel: each phase reduced modulo pi (sin^2 x and sin 2x have period
// pi), FP32 polynomials.
__device__ __forceinline__ float mixed_prob(const OscGenConst& oc, const float (&x)[3], const int (&)[3]) {
    float p = 0.f;
#pragma unroll
    for (int q = 0; q < 3; q++) {
        float s, c;
        sincos_poly(x[q], s, c);
        p = fmaf(oc.crf[q], s * s, fmaf(oc.cif[q], 2.0f * s * c, p));
    }
    return p + (float)oc.dab;  // exact for delta_ab = 1 when p <= -1/2 (Sterbenz)
}

// Double-float phases.
__device__ __forceinline__ float mixed_ff(const OscConst& oc, int r, float eh, float el) {
    float x[3];
    int odd[3];
    x[0] = reduce_half_pi(oc.c21h[r], oc.c21l[r], eh, el, odd[0]);
    x[1] = reduce_half_pi(oc.c31h[r], oc.c31l[r], eh, el, odd[1]);
    x[2] = reduce_half_pi(oc.c32h[r], oc.c32l[r], eh, el, odd[2]);
    return mixed_prob(oc, x, odd);
}

__device__ __forceinline__ float mixed_ff(const OscGenConst& oc, int r, float eh, float el) {
    float x[3];
    int odd[3];
#pragma unroll
    for (int q = 0; q < 3; q++) x[q] = reduce_pi_ff(oc.ch[q][r], oc.cl[q][r], eh, el);
    return mixed_prob(oc, x, odd);
}

// Phases in double, for what turns.cuh does not take (see osc_double).
__device__ __noinline__ float mixed_double(const OscConst& oc, int r, double E) {
    float eh, el, x[3];
    int odd[3];
    ff_recip(E, eh, el);
    const double e = (double)eh + (double)el;
    x[0] = reduce_half_pi_f64(oc.c21[r], e, odd[0]);
    x[1] = reduce_half_pi_f64(oc.c21[r] + oc.c32[r], e, odd[1]);
    x[2] = reduce_half_pi_f64(oc.c32[r], e, odd[2]);
    return mixed_prob(oc, x, odd);
}

__device__ __noinline__ float mixed_double(const OscGenConst& oc, int r, double E) {
    float eh, el, x[3];
    int odd[3];
    ff_recip(E, eh, el);
    const double e = (double)eh + (double)el;
#pragma unroll
    for (int q = 0; q < 3; q++) x[q] = reduce_pi_f64(oc.c[q][r], e);
    return mixed_prob(oc, x, odd);
}

template <class C>
__global__ void __launch_bounds__(256) k_osc_ff(const double* __restrict__ E, int64_t n, const __grid_constant__ C oc,
                                                float* __restrict__ P) {
    const int64_t k = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (k >= n) return;
    float eh, el;
    elem_recip(E[k], eh, el);
    for (int r = 0; r < oc.nL; r++) P[(int64_t)r * n + k] = mixed_ff(oc, r, eh, el);
}

// Phases of turns.cuh: no FP64 instruction (three phases formed and reduced in
// double take 27).  GB300: 3,000,017 energies at two baselines (mu -> e) 39 us,
// 281 with phases in double.
template <class C>
__global__ void __launch_bounds__(256) k_osc_f64phase(const double* __restrict__ E, int64_t n,
                                                      const __grid_constant__ C oc, float* __restrict__ P) {
    constexpr bool GEN = std::is_same<C, OscGenConst>::value;
    const int64_t k = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (k >= n) return;
    const double e = E[k];
    const ElemTurns el(oc.t, e);
    for (int r = 0; r < oc.nL; r++) {
        uint64_t f[3];
        const bool in = el.phases(oc.t, r, f[0], f[2]);
        f[1] = f[0] + f[2];
        float x[3];
        int odd[3];
#pragma unroll
        for (int q = 0; q < 3; q++) x[q] = GEN ? turn_radians((int64_t)f[q]) : turn_half(f[q], odd[q]);
        float p = mixed_prob(oc, x, odd);
        if (!in) p = mixed_double(oc, r, e);
        P[(int64_t)r * n + k] = p;
    }
}

// Most blocks of k_osc_fp64: twice what the current device holds at a time
// (asked once per device).  The second half starts as blocks of the first end
// and evens them out: 4,000,000 energies 88.2 us, with one wave 90.3; a table
// load per block is what more of them would cost.
template <class C>
cudaError_t osc_blocks(int64_t& blocks) {
    static std::once_flag once[64];
    static int count[64];
    static cudaError_t err[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::call_once(once[dev], [&] {
        int sms = 0, per_sm = 0;
        err[dev] = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (err[dev] == cudaSuccess) err[dev] = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_osc_fp64<C>, 256, 0);
        count[dev] = 2 * sms * std::max(per_sm, 1);
    });
    blocks = count[dev];
    return err[dev];
}

template <class C>
cudaError_t launch(const double* E, int64_t n, const C& oc, int prec, void* P, cudaStream_t s) {
    const int64_t blocks = (n + 255) / 256;
    if (prec == GNA_FP64) {
        int64_t most = 0;
        const cudaError_t e = osc_blocks<C>(most);
        if (e != cudaSuccess) return e;
        k_osc_fp64<C><<<(unsigned)std::min(blocks, most), 256, 0, s>>>(E, n, oc, (double*)P);
    } else if (prec == GNA_MIXED_F64PHASE)
        k_osc_f64phase<C><<<(unsigned)blocks, 256, 0, s>>>(E, n, oc, (float*)P);
    else
        k_osc_ff<C><<<(unsigned)blocks, 256, 0, s>>>(E, n, oc, (float*)P);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_oscprob(const double* E, int64_t n, const OscConst& oc, int prec, void* P, cudaStream_t s) {
    return launch(E, n, oc, prec, P, s);
}

cudaError_t launch_oscgen(const double* E, int64_t n, const OscGenConst& oc, int prec, void* P, cudaStream_t s) {
    return launch(E, n, oc, prec, P, s);
}

}  // namespace gna
