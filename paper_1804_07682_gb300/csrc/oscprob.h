// oscprob.h -- constants and launchers of the element-wise OscProb (oscprob.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"
#include "gnaosc.h"
#include "turns.cuh"

namespace gna {

// Constants of the fixed-point evaluation (turns.cuh) for
//   P = K + sum_q (a_q cos 2x_q + b_q sin 2x_q),
// K = delta + sum_q cr_q / 2, a_q = -cr_q / 2, b_q = ci_q, times 2^scale:
// integers with 61 bits after the point (K) and 63 (a, b).
struct TurnConst {
    TurnCoef ph21[GNA_NLMAX], ph32[GNA_NLMAX];
    int64_t K, a[3], b[3];
    int scale;
    int min_shift;  // smallest turn_shift() of the larger phase taken here
    int ok;         // 0: constants outside the integers' range, every element takes the double path
};

void turn_constants(const double* c21, const double* c32, int nL, double dab, const double* cr, const double* ci,
                    TurnConst& t);

// Survival probability: amplitudes A_ij and the phase coefficients K dm2 L.
struct OscConst {
    double c21[GNA_NLMAX], c32[GNA_NLMAX];
    float c21h[GNA_NLMAX], c21l[GNA_NLMAX], c32h[GNA_NLMAX], c32l[GNA_NLMAX], c31h[GNA_NLMAX], c31l[GNA_NLMAX];
    double A[3];
    float Af[3];
    float one_minus_A21f;
    int nL;
    TurnConst t;
};
cudaError_t launch_oscprob(const double* E, int64_t n, const OscConst& oc, int prec, void* P, cudaStream_t s);

// Any channel: phases q = (21, 31, 32) per baseline (double and hi + lo
// floats), coefficients -4 Re X and 2 Im X.
struct OscGenConst {
    double c[3][GNA_NLMAX];
    float ch[3][GNA_NLMAX], cl[3][GNA_NLMAX];
    double cr[3], ci[3];
    float crf[3], cif[3];
    double dab;  // delta_ab
    int nL;
    TurnConst t;
};
cudaError_t launch_oscgen(const double* E, int64_t n, const OscGenConst& oc, int prec, void* P, cudaStream_t s);

}  // namespace gna
