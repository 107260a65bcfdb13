// FP64 discrete Fourier transforms of any length, for the spectral derivative,
// the Hilbert transform, the filter and the antiderivative of every boundary.
//
// For M = M1 M2 (M1 the largest divisor <= sqrt(M)),
//   X[k1 + M1 k2] = sum_{n2} W^{M1 n2 k2} [W^{n2 k1} sum_{n1} x[M2 n1 + n2] W^{M2 n1 k1}],
// W = e^{-2 pi i / M}: pass A the inner transforms of length M1 with the twiddle,
// pass B the outer ones of length M2, one launch each over all jobs and vectors.
// FP64 issue bounds them (an SM retires two FP64 lanes a cycle), so the terms per
// output count: a pass of length L = La Lb takes La + Lb terms in two steps through
// shared memory instead of L (8192 points: 16 + 24 instead of 64 + 128), and many
// small CTAs spread the columns over the chip.  A prime L (or one with a prime
// factor above 64) is summed directly, its outputs shared by several CTAs and its
// input staged DFT_CHUNK elements at a time: with all of it staged, 131 KB at 8179
// (a length the context-free velocity takes), one CTA of four warps had an SM to
// itself and waited for its own sums (8179 + 13 nodes: 5365 us, in pieces 2650).
// Lengths with a large prime factor P, where that still means P terms per output
// (M P > 2^20), take Bluestein's form (L. Bluestein, "A linear filtering approach to
// the computation of discrete Fourier transform", 1970): with c_n = e^{-i pi n^2 / M},
// X_k = c_k sum_n (x_n c_n) conj(c_{k - n}), a convolution by two transforms of
// length Q = 2^q >= 2 M - 1 against the tabulated transform of conj(c).
// Measured: velocity weights at 16383 unknowns (four passes) 88 -> 43 us; a
// derivative of 3001 (prime) points 249 -> 67 us.
//
// Modes other than plain input scale the spectrum on the way in; the inverse is
// conj(DFT(conj(.)))/M, the division left to the caller.  A direct circulant
// convolution with the derivative kernel (entries up to M / 2 pi of alternating
// sign) loses too many digits; the DFT keeps FP64 accuracy in every mode.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "dft.cuh"

#define DFT_THREADS 128
#define DFT_TW_SMEM 1024   // transforms up to this length keep their twiddles in shared memory
#define DFT_CHUNK 512      // input elements of a longer direct pass staged at a time

namespace {

enum { PA_IN = 0, PA_BL = 1, PA_MID = 2, PB_OUT = 3, PB_MID = 4, PB_BL = 5 };

struct DftP {
  int T, L, La, cols;      // transform length, this pass's length and first factor (1: direct), columns T / L
  int C, KC, nch;          // columns per CTA, outputs per CTA and chunks per column (direct)
  int sp;                  // lanes per output
  int cta0;                // first CTA
  int in, out, work;       // offsets: input, output, Bluestein work
  int tw;                  // twiddle table offset
  int mode, kind, Mt;      // input mode; pass kind; true length (Bluestein)
  int chirp, bhat;         // table offsets
};
struct DftArgs {
  int n;
  DftP p[2 * BIE_MAXB + 2];
  const double *xr, *xr2;
  const double2 *xc, *tw, *twq, *chirp, *bhat;
  double2 *Y, *X, *bly, *blf;
  long long in_stride, stride, bl_stride;
};

__device__ __forceinline__ double2 zmul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -(a.y * b.y)), fma(a.x, b.y, a.y * b.x));
}

__device__ __forceinline__ double signed_k(int i, int M) {
  if (2 * i == M) return 0.0;           // Nyquist mode set to zero (even M)
  return (double)(2 * i < M ? i : i - M);
}

__device__ __forceinline__ double2 dft_input(int mode, int M, int off, const double* __restrict__ xr,
                                             const double* __restrict__ xr2,
                                             const double2* __restrict__ xc, int i) {
  if (mode == 0) return make_double2(xr[off + i], 0.0);
  if (mode == 8) return make_double2(xr2[off + i], 0.0);
  const double2 X = xc[off + i];
  if (mode == 3) return X;                                       // complex input as is
  if (mode == 6) {                                               // conj(rho(k) X), eq. filter
    const int ka = (2 * i <= M) ? i : M - i;                     // |k|, Nyquist at M/2
    const double r = (double)ka / (0.5 * (double)M);
    const double rho = exp(-36.0 * pow(r, 36.0));
    return make_double2(rho * X.x, -rho * X.y);
  }
  const double k = signed_k(i, M);
  if (mode == 5) return make_double2(-k * k * X.x, k * k * X.y);      // conj(-k^2 X)
  if (mode == 7) {                                               // conj(X/(ik)), 0 at k = 0
    if (k == 0.0) return make_double2(0.0, 0.0);
    return make_double2(X.y / k, X.x / k);
  }
  if (mode == 4) {                                               // conj(-i sgn(k) X)
    const double sg = (k > 0.0) ? 1.0 : (k < 0.0 ? -1.0 : 0.0);
    return make_double2(sg * X.y, sg * X.x);
  }
  if (mode == 1) return make_double2(-k * X.y, -k * X.x);        // conj(i k X)
  const double ak = fabs(k);
  return make_double2(ak * X.x, -ak * X.y);                      // conj(|k| X)
}

// four independent sums: the products of a complex term do not wait for one another
struct ZAcc {
  double a, b, c, d;
  __device__ __forceinline__ void zero() { a = b = c = d = 0.0; }
  __device__ __forceinline__ void add(double2 x, double2 w) {
    a = fma(x.x, w.x, a);
    b = fma(x.y, w.y, b);
    c = fma(x.x, w.y, c);
    d = fma(x.y, w.x, d);
  }
  __device__ __forceinline__ double2 value() const { return make_double2(a - b, c + d); }
};

__global__ void __launch_bounds__(DFT_THREADS) k_dft(const __grid_constant__ DftArgs a) {
  extern __shared__ __align__(16) double2 zs[];
  int q = 0;
  while (q + 1 < a.n && (int)blockIdx.x >= a.p[q + 1].cta0) ++q;
  const DftP& p = a.p[q];
  const int L = p.L, cols = p.cols, C = p.C;
  const int b = (int)blockIdx.x - p.cta0;
  const int col0 = (b / p.nch) * C, chunk = b % p.nch;
  const int nc = min(C, cols - col0);
  const long long v = blockIdx.y;
  const bool bl = p.kind == PA_BL || p.kind == PA_MID || p.kind == PB_MID || p.kind == PB_BL;
  const int sp = p.sp, sub = threadIdx.x % sp;   // sp: a power of two <= 32
  auto lanes = [&](double2 x) -> double2 {       // sum over the output's lanes
    for (int o = sp >> 1; o > 0; o >>= 1) {
      x.x += __shfl_xor_sync(0xffffffffu, x.x, o);
      x.y += __shfl_xor_sync(0xffffffffu, x.y, o);
    }
    return x;
  };
  const double2* tw = (bl ? a.twq : a.tw) + p.tw;
  double2* sx = zs;                      // input, element n of column c at n C + c
  double2* st = sx + C * L;              // twiddles e^{-2 pi i j / L}, j < L (L <= DFT_TW_SMEM)
  double2* sm = st + (L <= DFT_TW_SMEM ? L : 0);   // first step's result (two-step form)
  if (L <= DFT_TW_SMEM)
    for (int j = threadIdx.x; j < L; j += DFT_THREADS) st[j] = tw[(size_t)j * cols];
  // elements n0 .. n0 + len - 1 of every column into sx (all of them, but for a long direct pass)
  const int chunk_len = p.La == 1 && L > DFT_TW_SMEM ? DFT_CHUNK : L;
  auto stage = [&](int n0, int len) {
    for (int e = threadIdx.x; e < nc * len; e += DFT_THREADS) {
      const int n = e / nc, c = e - n * nc;
      const int i = (n0 + n) * cols + col0 + c;
      double2 x;
      switch (p.kind) {
        case PA_IN:
          x = dft_input(p.mode, p.T, p.in, a.xr + v * a.in_stride, a.xr2, a.xc + v * a.in_stride, i);
          break;
        case PA_BL:
          x = make_double2(0.0, 0.0);
          if (i < p.Mt)
            x = zmul(dft_input(p.mode, p.Mt, p.in, a.xr + v * a.in_stride, a.xr2, a.xc + v * a.in_stride, i),
                     a.chirp[p.chirp + i]);
          break;
        case PA_MID:
          x = zmul(a.blf[v * a.bl_stride + p.work + i], a.bhat[p.bhat + i]);
          x.y = -x.y;
          break;
        case PB_OUT:
          x = a.Y[v * a.stride + p.out + i];
          break;
        default:
          x = a.bly[v * a.bl_stride + p.work + i];
      }
      sx[n * C + c] = x;
    }
  };
  stage(0, min(L, chunk_len));
  __syncthreads();
  auto W = [&](int j) -> double2 { return L <= DFT_TW_SMEM ? st[j] : tw[(size_t)j * cols]; };
  auto store = [&](int c, int k, double2 x) {
    const int col = col0 + c;
    if (p.kind <= PA_MID) {              // pass A: twiddle, column-major work array
      x = zmul(x, tw[(size_t)col * k]);
      const size_t o = (size_t)col * L + k;
      if (p.kind == PA_IN) a.Y[v * a.stride + p.out + o] = x;
      else a.bly[v * a.bl_stride + p.work + o] = x;
      return;
    }
    const int o = col + cols * k;
    if (p.kind == PB_OUT) a.X[v * a.stride + p.out + o] = x;
    else if (p.kind == PB_MID) a.blf[v * a.bl_stride + p.work + o] = x;
    else if (o < p.Mt) {                 // conj / Q, times c_k
      const double s = 1.0 / (double)p.T;
      a.X[v * a.stride + p.out + o] = zmul(make_double2(s * x.x, -s * x.y), a.chirp[p.chirp + o]);
    }
  };
  // every thread of a warp makes the same passes (the sums are shared by lanes)
  const int per = DFT_THREADS / sp, e0 = threadIdx.x / sp;
  if (p.La > 1) {                        // two steps: n = Lb na + nb, k = ka + La kb
    const int La = p.La, Lb = L / La, nout = nc * L;
    for (int b0 = 0; b0 < nout; b0 += per) {
      const int e = min(b0 + e0, nout - 1);
      const int c = e % nc, r = e / nc, ka = r / Lb, nb = r - ka * Lb;
      ZAcc s;
      s.zero();
      const int inc = ka * Lb;           // (na ka Lb) mod L
      int j = (inc * sub) % L;
      const int step = (inc * sp) % L;
#pragma unroll 4
      for (int na = sub; na < La; na += sp) {
        s.add(sx[(na * Lb + nb) * C + c], W(j));
        j += step;
        if (j >= L) j -= L;
      }
      const double2 x = lanes(s.value());
      if (sub == 0 && b0 + e0 < nout) sm[r * C + c] = zmul(x, W(nb * ka));
    }
    __syncthreads();
    for (int b0 = 0; b0 < nout; b0 += per) {
      const int e = min(b0 + e0, nout - 1);
      // pass A stores run along k, pass B stores along the columns
      const int c = p.kind <= PA_MID ? e / L : e % nc, k = p.kind <= PA_MID ? e % L : e / nc;
      const int kb = k / La, ka = k - kb * La;
      ZAcc s;
      s.zero();
      const int inc = kb * La;           // (nb kb La) mod L
      int j = (inc * sub) % L;
      const int step = (inc * sp) % L;
#pragma unroll 4
      for (int nb = sub; nb < Lb; nb += sp) {
        s.add(sm[(ka * Lb + nb) * C + c], W(j));
        j += step;
        if (j >= L) j -= L;
      }
      const double2 x = lanes(s.value());
      if (sub == 0 && b0 + e0 < nout) store(c, k, x);
    }
    return;
  }
  // direct: outputs k0 .. k0 + nk - 1 of the CTA's column, at most one per lane group
  const int k0 = chunk * p.KC, nk = min(p.KC, L - k0), nout = nc * nk;
  const int e = min(e0, nout - 1);
  const int c = p.kind <= PA_MID ? e / nk : e % nc, k = k0 + (p.kind <= PA_MID ? e % nk : e / nc);
  ZAcc s;
  s.zero();
  int j = (int)(((long long)k * sub) % L);
  const int step = (int)(((long long)k * sp) % L);
  for (int n0 = 0; n0 < L; n0 += chunk_len) {
    const int len = min(chunk_len, L - n0);
    if (n0 > 0) {   // the previous piece has been read
      __syncthreads();
      stage(n0, len);
      __syncthreads();
    }
#pragma unroll 4
    for (int n = sub; n < len; n += sp) {   // a piece's length is a multiple of sp but for the last
      s.add(sx[n * C + c], W(j));
      j += step;
      if (j >= L) j -= L;
    }
  }
  const double2 x = lanes(s.value());
  if (sub == 0 && e0 < nout) store(c, k, x);
}

// c_n = e^{-i pi n^2 / M}, the padded sequence conj(c) (in F) and the twiddles of length Q
__global__ void k_bl_tables(int M, int Q, double2* __restrict__ chirp, double2* __restrict__ F,
                            double2* __restrict__ twq) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= Q) return;
  double s, c;
  sincospi(2.0 * (double)i / (double)Q, &s, &c);
  twq[i] = make_double2(c, -s);
  const int n = i < M ? i : (Q - i < M ? Q - i : -1);
  double2 b = make_double2(0.0, 0.0);
  if (n >= 0) {
    const long long n2 = ((long long)n * n) % (2LL * M);
    sincospi((double)n2 / (double)M, &s, &c);
    b = make_double2(c, s);
    if (i < M) chirp[i] = make_double2(c, -s);
  }
  F[i] = b;
}

int largest_divisor(int M) {   // <= sqrt(M)
  int best = 1;
  for (int d = 1; (long long)d * d <= M; ++d)
    if (M % d == 0) best = d;
  return best;
}
int largest_prime(int M) {
  int best = 1;
  for (int d = 2; (long long)d * d <= M; ++d)
    while (M % d == 0) {
      best = std::max(best, d);
      M /= d;
    }
  return std::max(best, M);
}

// The split of one pass; returns its CTAs and raises *smem to what it needs.  terms:
// what direct sums would take over all jobs and vectors of the launch.  Below
// 300,000 (2 us of the chip's FP64 rate) latency counts, a term being 64 cycles:
// direct sums, 16 outputs a CTA, eight lanes each (1472 points in 32 x 46: 8.3 us a
// pass in two steps, 5.9 so).  Above it FP64 issue counts: two steps, and as many
// columns per CTA as give each thread an output once every SM has its share.
int plan_pass(DftP& p, int T, int L, long long terms, long long cols, size_t* smem) {
  p.T = T;
  p.L = L;
  p.cols = T / L;
  p.La = largest_divisor(L);
  p.C = 1;
  p.sp = 1;
  if (terms < 300000) {
    p.La = 1;
    p.KC = 16;
    p.sp = 8;
  } else if (L <= 64 || (p.La > 1 && L / p.La <= 64)) {
    p.KC = L;
    if (cols > 608) p.C = std::max(1, std::min(p.cols, DFT_THREADS / L));
  } else {               // a large prime factor: outputs shared by lanes and CTAs
    p.La = 1;
    p.KC = 32;
    while (p.KC > 4 && p.KC * L > 2048) p.KC /= 2;
    p.sp = DFT_THREADS / p.KC;
  }
  p.nch = (L + p.KC - 1) / p.KC;
  const int staged = p.La == 1 && L > DFT_TW_SMEM ? DFT_CHUNK : L;
  const size_t need = (size_t)p.C * staged * (p.La > 1 ? 2 : 1) + (L <= DFT_TW_SMEM ? L : 0);
  *smem = std::max(*smem, need * sizeof(double2));
  return (p.cols + p.C - 1) / p.C * p.nch;
}

cudaError_t launch_pass(cudaStream_t st, const DftArgs& a, int ctas, size_t smem, int nvec) {
  if (a.n == 0 || ctas == 0) return cudaSuccess;
  const cudaError_t e = raise_smem_limit((const void*)k_dft, smem);
  if (e != cudaSuccess) return e;
  k_dft<<<dim3(ctas, nvec), DFT_THREADS, smem, st>>>(a);
  return cudaGetLastError();
}

// jobs whose length takes Bluestein's form have q[i] > 0 (the padded length)
cudaError_t run_passes(cudaStream_t st, const DftJobs& J, DftArgs& a, const int* q, const int* bl_off,
                       int nvec, long long* launches) {
  int work[2 * BIE_MAXB + 2];
  bool any = false;
  int w = 0;
  for (int i = 0; i < J.n; ++i) {
    work[i] = w;
    w += q[i];
    any = any || q[i] > 0;
  }
  a.bl_stride = w;
  for (int pass = 0; pass < (any ? 4 : 2); ++pass) {
    const bool B = pass & 1, mid = pass >= 2;
    a.n = 0;
    int cta = 0;
    size_t smem = 0;
    long long cols = 0, terms = 0;   // columns, and terms of direct sums, over all jobs and vectors
    for (int i = 0; i < J.n; ++i) {
      if (mid && q[i] == 0) continue;
      const int T = q[i] > 0 ? q[i] : J.j[i].M, d1 = q[i] > 0 ? largest_divisor(T) : J.j[i].M1;
      cols += (long long)(B ? d1 : T / d1) * nvec;
      terms += (long long)T * (B ? T / d1 : d1) * nvec;
    }
    for (int i = 0; i < J.n; ++i) {
      const DftJob& jb = J.j[i];
      if (mid && q[i] == 0) continue;
      DftP& p = a.p[a.n++];
      const int T = q[i] > 0 ? q[i] : jb.M, d1 = q[i] > 0 ? largest_divisor(T) : jb.M1;
      p.cta0 = cta;
      cta += plan_pass(p, T, B ? T / d1 : d1, terms, cols, &smem);
      p.in = jb.off_in;
      p.out = jb.off_out;
      p.work = work[i];
      p.tw = q[i] > 0 ? bl_off[i] : jb.off_tw;
      p.mode = jb.mode;
      p.Mt = jb.M;
      p.chirp = jb.off_tw;
      p.bhat = bl_off[i];
      if (q[i] == 0) p.kind = B ? PB_OUT : PA_IN;
      else p.kind = mid ? (B ? PB_BL : PA_MID) : (B ? PB_MID : PA_BL);
    }
    const cudaError_t e = launch_pass(st, a, cta, smem, nvec);
    if (e != cudaSuccess) return e;
    if (launches) *launches += 1;
  }
  return cudaSuccess;
}

}  // namespace

bie_status dft_tables(bie_ctx* c) {
  int Q = 0;
  for (int k = 0; k < c->nb; ++k) {
    const int M = c->M[k];
    c->bl_q[k] = 0;
    c->bl_off[k] = Q;
    if ((long long)M * largest_prime(M) > (1LL << 20)) {
      int n = 1;
      while (n < 2 * M - 1) n *= 2;
      c->bl_q[k] = n;
      Q += n;
    }
  }
  if (Q == 0) return BIE_OK;
  double2 *chirp, *bhat, *twq, *F, *Y;
  BIE_GET(c, double2, "bl_chirp", c->N, chirp);
  BIE_GET(c, double2, "bl_bhat", Q, bhat);
  BIE_GET(c, double2, "bl_twq", Q, twq);
  BIE_GET(c, double2, "bl_tmp", Q, F);
  BIE_GET(c, double2, "bl_tmpY", Q, Y);
  DftJobs J;
  memset(&J, 0, sizeof(J));
  for (int k = 0; k < c->nb; ++k) {
    const int q = c->bl_q[k], o = c->bl_off[k];
    if (q == 0) continue;
    k_bl_tables<<<(q + 63) / 64, 64, 0, c->stream>>>(c->M[k], q, chirp + c->off[k], F + o, twq + o);
    BIE_LAUNCH_CHECK(c, "k_bl_tables");
    J.j[J.n++] = DftJob{q, largest_divisor(q), o, o, o, 3};
  }
  const cudaError_t e = dft_run_plain(c->stream, J, nullptr, F, twq, Y, bhat);
  if (e != cudaSuccess) return ctx_cuda(c, e, "k_dft (tables)");
  return BIE_OK;
}

bie_status dft_run(bie_ctx* c, const DftJobs& J, const double* xr, const double2* xc, double2* Y,
                   double2* X, int nvec, long long in_stride, long long stride, const double* xr2) {
  DftArgs a;
  memset(&a, 0, sizeof(a));
  bool oom = false;
  a.tw = (const double2*)ctx_buf(c, "dft_tw", sizeof(double2) * c->N, &oom);
  if (oom) return ctx_fail(c, BIE_ERR_OOM, "dft: twiddles");
  int q[2 * BIE_MAXB + 2], bo[2 * BIE_MAXB + 2];
  long long w = 0;
  for (int i = 0; i < J.n; ++i) {   // a job's boundary is the one its tables belong to
    q[i] = bo[i] = 0;
    for (int k = 0; k < c->nb; ++k)
      if (c->off[k] == J.j[i].off_tw && c->M[k] == J.j[i].M) {
        q[i] = c->bl_q[k];
        bo[i] = c->bl_off[k];
      }
    w += q[i];
  }
  if (w > 0) {
    int Q = 0;
    for (int k = 0; k < c->nb; ++k) Q += c->bl_q[k];
    a.chirp = (const double2*)ctx_buf(c, "bl_chirp", sizeof(double2) * c->N, &oom);
    a.bhat = (const double2*)ctx_buf(c, "bl_bhat", sizeof(double2) * Q, &oom);
    a.twq = (const double2*)ctx_buf(c, "bl_twq", sizeof(double2) * Q, &oom);
    if (oom) return ctx_fail(c, BIE_ERR_OOM, "dft: tables");
    BIE_GET(c, double2, "bl_Y", (size_t)w * nvec, a.bly);
    BIE_GET(c, double2, "bl_F", (size_t)w * nvec, a.blf);
  }
  a.xr = xr;
  a.xr2 = xr2;
  a.xc = xc;
  a.Y = Y;
  a.X = X;
  a.in_stride = in_stride;
  a.stride = stride;
  const cudaError_t e = run_passes(c->stream, J, a, q, bo, nvec, &c->launches);
  if (e != cudaSuccess) return ctx_cuda(c, e, "k_dft");
  return BIE_OK;
}

cudaError_t dft_run_plain(cudaStream_t st, const DftJobs& J, const double* xr, const double2* xc,
                          const double2* tw, double2* Y, double2* X) {
  DftArgs a;
  memset(&a, 0, sizeof(a));
  a.tw = tw;
  a.xr = xr;
  a.xc = xc;
  a.Y = Y;
  a.X = X;
  int zero[2 * BIE_MAXB + 2] = {0};
  return run_passes(st, J, a, zero, zero, 1, nullptr);
}
