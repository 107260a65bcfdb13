// FP64 discrete Fourier transforms of the boundaries' node vectors (dft.cu).
#pragma once
#include "common.cuh"

struct DftJob {
  int M, M1;
  int off_in;    // input offset (real omega for mode 0, spectrum for modes 1/2)
  int off_out;   // output offset in the complex work array
  int off_tw;    // offset of the boundary's nodes (its tables: e^{-2 pi i j / M}, j < M)
  int mode;      // 0: real input; 1: conj(i k X); 2: conj(|k| X); 3: complex input;
                 // 4: conj(-i sgn(k) X) (Hilbert transform); 5: conj(-k^2 X)
                 // (second derivative); 6: conj(rho(k) X) (filter of eq. filter);
                 // 7: conj(X/(ik)), zero at k = 0 (zero-mean antiderivative);
                 // 8: real input from the second input array
};
struct DftJobs {
  int n;
  DftJob j[2 * BIE_MAXB + 2];
};

// The transforms of the jobs: inputs xr (modes 0, 8: xr2) or xc, outputs in X
// (off_out of each job), Y a work array of the outputs' size.  nvec independent
// vectors: vector v reads at v in_stride and writes at v stride.  X may be xc.
bie_status dft_run(bie_ctx* c, const DftJobs& J, const double* xr, const double2* xc, double2* Y,
                   double2* X, int nvec = 1, long long in_stride = 0, long long stride = 0,
                   const double* xr2 = nullptr);
// The same from bare tables (e^{-2 pi i j / M} at off_tw), without a context.
cudaError_t dft_run_plain(cudaStream_t st, const DftJobs& J, const double* xr, const double2* xc,
                          const double2* tw, double2* Y, double2* X);
// Which boundaries take Bluestein's form and its tables (after the node counts changed).
bie_status dft_tables(bie_ctx* c);
