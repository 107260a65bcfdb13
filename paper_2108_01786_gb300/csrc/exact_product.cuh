// The full-accuracy (hi + lo) operator times a block of columns by exact
// integer slices on the tensor cores (exact_product.cu).
#pragma once
#include "common.cuh"

#define OZ_BITS 5
#define OZ_S 10
#define OZ_KMAX 16384   // largest row length: the integer sums of a level stay below 2^31
#define OZ_MIN_RHS 8    // solves: below this many columns the double-float GEMV is faster

// Y[c ys + m] = sum_l B_ml x_cl w_l (+ sgn_m x_cm where sgn is given), c < nrhs <= 64,
// for the matrix `which` (0: A, N rows; 1: the surface U-matrix, M_0 rows), w_l = 1/M_l
// when apply_w, else 1, with the first S slices of each operand (S = OZ_S: full accuracy).
// Enqueued on the context's stream; *err (device, zeroed by the caller) becomes 1
// when a wait inside the product ran out.
bie_status oz_product(bie_ctx* c, int which, int nrhs, const double* X, long long xs, int apply_w,
                      int S, double* Y, long long ys, const float* sgn, int* err);
