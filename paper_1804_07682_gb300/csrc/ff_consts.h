// Generated by fit_sincos.py -- do not edit.
// FP32 minimax-style polynomials on |r| <= 1.572796 (Lawson-weighted least squares).
// Polynomial error (double evaluation): sin 4.87e-09, cos 5.36e-08.
// Float32 Horner evaluation error (sampled): sin 8.25e-08, cos 1.57e-07.
#pragma once
#define GNA_SIN_C1 (-1.666665673e-01f)
#define GNA_SIN_C2 (8.333008736e-03f)
#define GNA_SIN_C3 (-1.980601664e-04f)
#define GNA_SIN_C4 (2.598767651e-06f)
#define GNA_COS_C1 (-4.999993145e-01f)
#define GNA_COS_C2 (4.166396707e-02f)
#define GNA_COS_C3 (-1.385575277e-03f)
#define GNA_COS_C4 (2.319028135e-05f)
// Chunk-anchored loops, |r| <= 1.821796: polynomial error sin 2.33e-08, cos 5.25e-09 (cos - 1: 4.22e-09 of itself).
#define GNA_SINA_C1 (-1.666663587e-01f)
#define GNA_SINA_C2 (8.332575671e-03f)
#define GNA_SINA_C3 (-1.977937063e-04f)
#define GNA_SINA_C4 (2.548287284e-06f)
#define GNA_COSA_C1 (-5.000000000e-01f)
#define GNA_COSA_C2 (4.166664928e-02f)
#define GNA_COSA_C3 (-1.388838165e-03f)
#define GNA_COSA_C4 (2.475560905e-05f)
#define GNA_COSA_C5 (-2.590579697e-07f)
// Chunk-anchored loops, |r| <= 1.186398: polynomial error sin 2.28e-10, cos 1.14e-08 (cos - 1: 2.08e-08 of itself).
#define GNA_SINQ_C1 (-1.666666567e-01f)
#define GNA_SINQ_C2 (8.333275095e-03f)
#define GNA_SINQ_C3 (-1.982997928e-04f)
#define GNA_SINQ_C4 (2.666453838e-06f)
#define GNA_COSQ_C1 (-5.000000000e-01f)
#define GNA_COSQ_C2 (4.166652262e-02f)
#define GNA_COSQ_C3 (-1.388277742e-03f)
#define GNA_COSQ_C4 (2.405918167e-05f)
// pi = PI_A + PI_B + PI_C; PI_A and PI_B have 12 significant bits.
#define GNA_PI_A (3.140625f)
#define GNA_PI_B (0.00096750259399414062f)
#define GNA_PI_C (1.509958025e-07f)
// pi = PI_A + PI_B2 + e2 with PI_B2 the float32 rounding of pi - PI_A, |e2| = 5.13e-12.
#define GNA_PI_B2 (9.676535847e-04f)
#define GNA_PI_E2 (5.127e-12)
#define GNA_INV_PI_F (3.183098733e-01f)
// pi = PI_DA + PI_DB + PI_DC in double; PI_DA, PI_DB have 26 significant bits.
#define GNA_PI_DA (3.1415926218032837)
#define GNA_PI_DB (3.1786509424591713e-08)
#define GNA_PI_DC (1.2246467991473532e-16)
#define GNA_INV_PI_D (0.31830988618379069)
