// One solve in one cooperative kernel: the scheme of gmres.cu (delayed CGS2
// with one global reduction per Arnoldi step, FP64 Hessenberg, obstacle
// preconditioner, recycled subspace, refinement with the same residual rules)
// with every cycle, test and update on the device.
//
// What bounds a solve of up to a few thousand unknowns is not the matrix but
// the chain of small kernels around it: at 640 unknowns the 20 step pairs, 4
// updates and 5 residuals of the kernel-by-kernel solver took 640 us, of which
// the matrix products need 10.  Three things make up that chain, and each has
// its answer here:
//   * launches, drains and host round trips at the end of every cycle: one
//     launch, grid barriers (about a microsecond) between phases;
//   * L2 round trips for the basis: every CTA owns a chunk of rows for the
//     whole solve, so its slices of V and C (Z and U when they fit) live in
//     shared memory and only the new vector z_j and the partial sums are
//     exchanged; what shared memory is left holds the head of every row of the
//     inner storage (all of it up to ~3900 unknowns in 16 bits), read once;
//   * FP64 issue: an SM retires two FP64 lanes a cycle, and adding 50 rows of
//     152 partial sums in FP64 on every SM takes 5 us.  Partial sums are
//     exchanged and added on the FP32 pipes, in two or three floats (below).
// The Hessenberg work (a chain of ~200 dependent FP64 operations) runs on a
// warp of its own in every CTA, from identical data, so nothing is published;
// when a product is short (RsArgs::lag) it runs beside the next product, one
// step behind, and a cycle ends one discarded product late.
//
// Phases of a cycle, a grid barrier after each:
//   RESID  r = D (b - A x) of the own rows, partial |r|^2
//   START  |r|, tests; z_0 = r / |r|, its dots with C
//   G(j)   w = D A P z_j of the own rows; dots of w with [C, V_0..V_{j-1}, z_j, w]
//   D(j)   v_j, z_{j+1} of the own rows; dots of z_{j+1}
//   UPDATE x += |r| P (Z y + U (c_0 - B y)); C and U grow
//
// Measured (GB300, bie_solve_b back to back against the kernel-by-kernel solver): 640
// unknowns FP32 690 -> 340 us, 1001 FP64 665 -> 364, 2944 FP16 876 -> 487, 4099 BF16 796 -> 476,
// 8256 FP16 1344 -> 990, 16383 FP16 2697 -> 2530 (there HBM bounds it; what is saved is the
// chain between products).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "common.cuh"
#include "nvtx.cuh"
#include "gemv_dot.cuh"
#include "krylov.cuh"

#define RS_RQ 32          // recycled columns kept at most
#define RS_RK 16          // columns a cycle may add
#define RS_MINROWS 31     // rows per CTA on small problems: one per row warp
#define RS_MAXN 16384     // x / M staged as hi + lo in shared memory
#define RS_SMEM_MAX (224 * 1024)

int gemv_num_ctas();

struct RsOut {            // host-mapped result of a solve
  int iters, cycles, converged, nonfinite, stagnated;
  int timeout;            // set before the launch, cleared by the last CTA out if no wait ran out
  double rnorm, bnorm;
};
static_assert(sizeof(RsOut) <= sizeof(HostSlot) * BIE_NSLOTS, "result fits the slot ring");

// byte offsets of the shared-memory arrays
struct RsLayout {
  unsigned V, C, Z, U, w, r, ry, red, xo, s1, s3, cs, sn, g, hraw, braw, hfin, hnew, bnew, rinv, H, B, c0, y, tq, Ri, Mq, RiF, MqF,
      zmean, umean, f1, wt, A;
  unsigned total;
};

struct RsArgs {
  int N, m, R, G, nobs, obs0, rowflip, x0, max_cycles, lag, kv, zsm;
  int obs_off[BIE_MAXB + 1];
  float obs_invM[BIE_MAXB];
  float obs_coef;
  long long ld;
  double rtol, inner_tol, drift;
  double eps16;            // rounding of an inner-storage product (0: none cheaper than A_hi)
  const void* A;           // inner storage (the FP64 matrix in the plain scheme)
  const float* Ahi;
  const float* Alo;
  const float* wgt;
  const double* wgt64;
  const float* sgn;
  const int* blk;
  const double* b;
  double* x;
  void* zbuf;              // ld: z_j / M_l
  float* xh;               // ld: the vector of the next residual / M_l, hi (FP64 scheme: double)
  float* xl;               //     and lo
  void* Zg;                // (m + 1) x ld and RS_RQ x ld: Z and U when not in shared memory
  void* Ug;
  float4* part;            // 3 x [row][G] partial sums: of w, and two halves of z_j
  int prow;                // rows of one of them
  double* partn;           // [G]
  unsigned* bar;           // [0] arrivals, [1] leavers; zero between solves; [3] x is a solve's iterate
  int* err;
  unsigned spin_limit;
  RsOut* out;
  long long pf_bytes;      // head of the CTA's chunk of A fetched into L2 per step
  int stream;              // A is larger than L2 holds: evict-first loads
  RsLayout L;
};

// 1 / sqrt(d), d > 0: two Newton steps from the FP32 value (2^-22 -> 2^-43 ->
// rounding); the library's square root and division are a chain of ~40
// dependent FP64 operations on the critical path of every step
__device__ __forceinline__ double rs_rsqrt(double d) {
  if (!(d > 1e-30 && d < 1e30)) return 1.0 / sqrt(d);
  double x = (double)rsqrtf((float)d);
  const double h = 0.5 * d;
  x = x * fma(-h * x, x, 1.5);
  return x * fma(-h * x, x, 1.5);
}

// Givens rotation that zeroes b against a: (c, s, r) with c a + s b = r, and 1 / r
__device__ __forceinline__ void rs_givens(double a, double b, double& c, double& s, double& r, double& ir) {
  const double d = fma(a, a, b * b);   // entries of order one (Hessenberg columns of unit vectors)
  c = 1.0;
  s = r = ir = 0.0;
  if (d > 0.0) {
    ir = rs_rsqrt(d);
    c = a * ir;
    s = b * ir;
    r = d * ir;
  }
}

// The rotations 0..n-1 (cs, sn) applied to two Hessenberg columns at once by one
// warp (see givens_apply_warp: the recurrence is a scan of affine maps, whose
// slopes the columns share).  hA[0..n-1] is rewritten rotated; uA, uB are the
// entries at n after the rotations.
__device__ __forceinline__ void rs_rotate2(double* hA, const double* hB, const double* cs, const double* sn,
                                           int n, double& uA, double& uB) {
  const int lane = threadIdx.x & 31;
  double a = hA[0], b = hB[0];
  for (int base = 0; base < n; base += 64) {
    const int e0 = base + 2 * lane, e1 = e0 + 1;
    const bool v0 = e0 < n, v1 = e1 < n;
    const double c0 = v0 ? cs[e0] : 1.0, s0 = v0 ? sn[e0] : 0.0;
    const double c1 = v1 ? cs[e1] : 1.0, s1 = v1 ? sn[e1] : 0.0;
    const double p0 = v0 ? hA[e0 + 1] : 0.0, p1 = v1 ? hA[e1 + 1] : 0.0;
    const double q0 = v0 ? hB[e0 + 1] : 0.0, q1 = v1 ? hB[e1 + 1] : 0.0;
    const double A0 = v0 ? -s0 : 1.0, A1 = v1 ? -s1 : 1.0;
    const double P0 = c0 * p0, P1 = c1 * p1, Q0 = c0 * q0, Q1 = c1 * q1;   // 0 past n
    double A = A1 * A0, P = fma(A1, P0, P1), Q = fma(A1, Q0, Q1);
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const double Ap = __shfl_up_sync(0xffffffffu, A, d);
      const double Pp = __shfl_up_sync(0xffffffffu, P, d);
      const double Qp = __shfl_up_sync(0xffffffffu, Q, d);
      if (lane >= d) {
        P = fma(A, Pp, P);
        Q = fma(A, Qp, Q);
        A = A * Ap;
      }
    }
    double Ae = __shfl_up_sync(0xffffffffu, A, 1), Pe = __shfl_up_sync(0xffffffffu, P, 1);
    if (lane == 0) {
      Ae = 1.0;
      Pe = 0.0;
    }
    const double u0 = fma(Ae, a, Pe);
    const double u1 = fma(A0, u0, P0);
    const double la = fma(A1, u1, P1), lb = fma(A, b, Q);   // after this lane's two rotations
    __syncwarp();
    if (v0) hA[e0] = fma(c0, u0, s0 * p0);
    if (v1) hA[e1] = fma(c1, u1, s1 * p1);
    a = __shfl_sync(0xffffffffu, la, 31);
    b = __shfl_sync(0xffffffffu, lb, 31);
    __syncwarp();
  }
  uA = a;
  uB = b;
}

// ---------------------------------------------------------------------------
// Partial sums, no less accurate than the kernel-by-kernel solver's.  The dots of
// w = A z_j and of a cycle's z_0 and the sums over obstacles, FP64 there, are three floats
// (tfl.h, 72 bits) from the lanes' products, exact in two floats, to the sum over the
// CTAs.  The dots of the later z_j, FP32 runs of eight added in FP64 there, are
// double-float (48 bits).  FP64 vectors are added in FP64 within a CTA and exchanged as
// three floats.  (FP64 throughout takes 1.5 us on every SM for 10 additions a row over
// 20 rows, twice a step.  Double-float throughout, 5 bits short of FP64, took 342 us at
// 640 unknowns and 461 at 4099, this 340 and 476.)
// Three floats have FP32's exponents: |z| = 1, and |A z|^2 would have to leave 2^-96 ..
// 2^127 for a word to be lost, where the diagonal of +-1/2 makes the system singular to
// FP64 anyway (condition above 10^14 at the one end, 10^19 at the other).
// ---------------------------------------------------------------------------
template <class VT, bool F> struct RsAcc;   // F: three words exchanged, else two
template <> struct RsAcc<float, true> {
  typedef tfl T;           // a lane's sum
  typedef tfl X;           // as exchanged and added over the CTAs
  typedef float4 S;        // a sum over the CTAs: its nearest float first, unused last
  static constexpr int LD = 5;   // exchanged values in flight per lane
  static __device__ __forceinline__ T zero() { return {0.f, 0.f, 0.f}; }
  static __device__ __forceinline__ T mad(T s, float a, float b) {
    const dfl p = df_two_prod(a, b);
    tf_add(s, p.hi, p.lo);
    return s;
  }
  static __device__ __forceinline__ T addv(T s, float a) {
    tf_add(s, a, 0.f);
    return s;
  }
  static __device__ __forceinline__ T warp(T a) { return tf_warp_sum(a); }
  static __device__ __forceinline__ X split(T a) { return a; }
  static __device__ __forceinline__ S pack(X a) {
    a = tf_norm(a);
    return make_float4(a.s, a.e, a.f, 0.f);
  }
};
template <> struct RsAcc<float, false> {
  typedef dfl T;
  typedef dfl X;
  typedef float4 S;
  static constexpr int LD = 10;
  static __device__ __forceinline__ T zero() { return {0.f, 0.f}; }
  static __device__ __forceinline__ T mad(T s, float a, float b) {
    const dfl p = df_two_prod(a, b);
    const dfl t = df_two_sum(s.hi, p.hi);
    return df_fast_two_sum(t.hi, t.lo + (s.lo + p.lo));
  }
  static __device__ __forceinline__ T warp(T a) { return warp_sum(a); }
  static __device__ __forceinline__ X split(T a) { return a; }
  static __device__ __forceinline__ S pack(X a) { return make_float4(a.hi, a.lo, 0.f, 0.f); }
};
template <> struct RsAcc<double, true> {
  typedef double T;
  typedef tfl X;
  typedef double S;
  static constexpr int LD = 5;
  static __device__ __forceinline__ T zero() { return 0.0; }
  static __device__ __forceinline__ T mad(T s, double a, double b) { return fma(a, b, s); }
  static __device__ __forceinline__ T addv(T s, double a) { return s + a; }
  static __device__ __forceinline__ T warp(T a) { return warp_sum(a); }
  static __device__ __forceinline__ X split(T a) {
    const float h = (float)a;
    const double r = a - (double)h;
    const float l = (float)r;
    return {h, l, (float)(r - (double)l)};
  }
  static __device__ __forceinline__ S pack(X a) { return tf_to_double(a); }
};

// Exchange: value i (row r of CTA c at i = r G + c) of a region, 16 bytes as three words or 8
// as two.  The rows of one region in two words come before those in three.
__device__ __forceinline__ void rs_put(float4* p, size_t i, tfl v) { p[i] = make_float4(v.s, v.e, v.f, 0.f); }
__device__ __forceinline__ void rs_put(float4* p, size_t i, dfl v) {
  reinterpret_cast<float2*>(p)[i] = make_float2(v.hi, v.lo);
}
__device__ __forceinline__ void rs_get(const float4* p, size_t i, tfl& v) {
  const float4 a = __ldcg(p + i);
  v = {a.x, a.y, a.z};
}
__device__ __forceinline__ void rs_get(const float4* p, size_t i, dfl& v) {
  const float2 a = __ldcg(reinterpret_cast<const float2*>(p) + i);
  v = {a.x, a.y};
}
__device__ __forceinline__ void rs_zero(tfl& v) { v = {0.f, 0.f, 0.f}; }
__device__ __forceinline__ void rs_zero(dfl& v) { v = {0.f, 0.f}; }
__device__ __forceinline__ void rs_zero(double& v) { v = 0.0; }
__device__ __forceinline__ tfl rs_lane(tfl s, int o) { return tf_lane(s, o); }
__device__ __forceinline__ dfl rs_lane(dfl s, int o) {
  return {__shfl_xor_sync(0xffffffffu, s.hi, o), __shfl_xor_sync(0xffffffffu, s.lo, o)};
}
__device__ __forceinline__ double rs_lane(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
// a sum over the CTAs: its value, and its head in the vectors' type
__device__ __forceinline__ double rs_value(const float4& a) { return tf_to_double({a.x, a.y, a.z}); }
__device__ __forceinline__ double rs_value(double a) { return a; }
__device__ __forceinline__ float rs_head(const float4& a) { return a.x; }
__device__ __forceinline__ float rs_head(dfl a) { return a.hi; }
__device__ __forceinline__ double rs_head(double a) { return a; }

// What follows from the sums (nu, h_j, beta) is ~35 dependent operations: 2400 cycles in
// double-float, 4100 in three floats, 6600 in FP64 beside other FP64 work.  The Hessenberg
// matrix takes the three-float values, formed by three warps beside the row work; the rows
// take the double-float ones (43 bits and more), rounded to their own FP32.
__device__ __forceinline__ void rs_sc(const float4& a, dfl& v) { v = {a.x, a.y}; }
__device__ __forceinline__ void rs_sc(const float4& a, tfl& v) { v = {a.x, a.y, a.z}; }
__device__ __forceinline__ void rs_sc(double a, double& v) { v = a; }
// 1 / sqrt(a), 0 for a <= 0
__device__ __forceinline__ dfl rs_rsqrt_pos(dfl a) {   // one Newton step from the FP32 value
  if (!(a.hi > 0.f)) return {0.f, 0.f};
  const float x = rsqrtf(a.hi);
  const dfl e = dfl{1.f, 0.f} - a * df_two_prod(x, x);
  return df_fast_two_sum(x, 0.5f * x * e.hi);
}
__device__ __forceinline__ double rs_rsqrt_pos(double a) { return a > 0.0 ? rs_rsqrt(a) : 0.0; }
__device__ __forceinline__ tfl rs_rsqrt_pos(tfl a) { return tf_rsqrt_from(a, rsqrtf(a.s)); }

template <class VT> struct RsHead { typedef dfl T; };   // what the rows' scalars are formed in
template <> struct RsHead<double> { typedef double T; };
// sum_i a_i b_i, i < n, by one warp (every lane gets it)
template <class T, class S>
__device__ __forceinline__ T rs_sum(const S* a, const S* b, int n) {
  T t;
  rs_zero(t);
  for (int i = threadIdx.x & 31; i < n; i += 32) {
    T u, v;
    rs_sc(a[i], u);
    rs_sc(b[i], v);
    t = t + u * v;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t = t + rs_lane(t, o);
  return t;
}
template <class T> struct RsScal {
  T nu, inu, hj, beta, ibe;
};
// nu, h_j, beta of a step (see k_dcgs) by one warp; s3, s1: the sums of z_j and of w
template <class T, class S>
__device__ __forceinline__ RsScal<T> rs_scalars(const S* s3, const S* s1, int nb) {
  T ta, tas, tss;
  rs_zero(ta);
  rs_zero(tas);
  rs_zero(tss);
  for (int i = threadIdx.x & 31; i < nb; i += 32) {
    T v3, v1;
    rs_sc(s3[i], v3);
    rs_sc(s1[i], v1);
    ta = ta + v3 * v3;
    tas = tas + v3 * v1;
    tss = tss + v1 * v1;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    ta = ta + rs_lane(ta, o);
    tas = tas + rs_lane(tas, o);
    tss = tss + rs_lane(tss, o);
  }
  T a, sg, om;
  rs_sc(s3[nb], a);
  rs_sc(s1[nb], sg);
  rs_sc(s1[nb + 1], om);
  RsScal<T> r;
  const T nu2 = a - ta;
  r.inu = rs_rsqrt_pos(nu2);
  r.nu = nu2 * r.inu;
  r.hj = (sg - tas) * r.inu;
  const T be2 = om - tss - r.hj * r.hj;
  r.ibe = rs_rsqrt_pos(be2);
  r.beta = be2 * r.ibe;
  return r;
}

// coef a im rounded to FP32 (a few 2^-48 more): an obstacle's share of the preconditioner
// from its sum a
__device__ __forceinline__ float rs_share(const float4& a, float im, float coef) {
  const dfl p = df_two_prod(a.x, im);
  return fmaf(coef, p.hi, coef * fmaf(a.y, im, p.lo));
}
__device__ __forceinline__ double rs_share(double a, double im, double coef) { return coef * (a * im); }

// ---------------------------------------------------------------------------
// grid barrier: arrivals counted upward through the solve (epoch e waits for
// e G of them), a bounded wait
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool rs_barrier(const RsArgs& a, unsigned& epoch, int* s_ok) {
  __syncthreads();
  if (threadIdx.x == 0) {
    epoch += (unsigned)a.G;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.bar) : "memory");
    unsigned v, it = 0;
    int ok = 1;
    while (true) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a.bar) : "memory");
      if (v >= epoch) break;
      if ((++it & 1023u) == 0 && *(volatile int*)a.err) {
        ok = 0;
        break;
      }
      if (it > a.spin_limit) {
        atomicExch(a.err, 1);
        ok = 0;
        break;
      }
    }
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok != 0;
}

__device__ __forceinline__ void rs_bar_rows(int n) {   // the row warps only
  asm volatile("bar.sync 1, %0;" ::"r"(n) : "memory");
}

// the scalars of a step: ready (not waiting), and waited for by the Hessenberg warp
__device__ __forceinline__ void rs_arrive_scal(int n) {
  __syncwarp();
  asm volatile("bar.arrive 3, %0;" ::"r"(n) : "memory");
}
__device__ __forceinline__ void rs_bar_scal(int n) {
  asm volatile("bar.sync 3, %0;" ::"r"(n) : "memory");
}

// Sums over the G CTAs of the rows of `part`, fixed order, LN lanes per row: 16, or 32 where
// the loads in flight of 16 lanes would not cover the CTAs (a second round of loads costs
// as much as the first: 4099 unknowns 510 -> 487 us).  The first rows' loads are issued by
// rs_load so that other work can hide them; rs_reduce adds them and takes the remaining
// rows (nthr threads take part).
template <class AC, int LN>
__device__ __forceinline__ void rs_load(const float4* part, int cnt, int G, typename AC::X* v, int base = 0) {
  const int i = base + (int)threadIdx.x / LN, q = threadIdx.x % LN;
#pragma unroll
  for (int u = 0; u < AC::LD; ++u) {
    const int c = q + LN * u;
    rs_zero(v[u]);
    if (i < cnt && c < G) rs_get(part, (size_t)i * G + c, v[u]);
  }
}
template <class AC, int LN>
__device__ __forceinline__ void rs_reduce(const float4* part, int cnt, int G, typename AC::X* v,
                                          typename AC::S* out, int nthr) {
  const int q = threadIdx.x % LN;
  for (int base = 0; base < cnt; base += nthr / LN) {
    const int i = base + (int)threadIdx.x / LN;
    if (base > 0) rs_load<AC, LN>(part, cnt, G, v, base);
    typename AC::X s = v[0];
#pragma unroll
    for (int u = 1; u < AC::LD; ++u)
      if (LN * u < G) s = s + v[u];
    if (i < cnt) {
      for (int c = q + LN * AC::LD; c < G; c += LN) {
        typename AC::X t;
        rs_get(part, (size_t)i * G + c, t);
        s = s + t;
      }
    }
    __syncwarp();
#pragma unroll
    for (int o = LN / 2; o > 0; o >>= 1) s = s + rs_lane(s, o);
    if (i < cnt && q == 0) out[i] = AC::pack(s);
  }
}

// sum of the G FP64 partials by one warp (every lane gets it)
__device__ __forceinline__ double rs_sum_partn(const double* p, int G) {
  double s = 0.0;
  for (int c = threadIdx.x & 31; c < G; c += 32) s += __ldcg(p + c);
  return warp_sum(s);
}

__device__ __forceinline__ uint4 rs_ld(const uint4* p, unsigned long long pol) {
  uint4 v;
  asm("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
      : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
      : "l"(p), "l"(pol));
  return v;
}

// ---------------------------------------------------------------------------
// row products
// ---------------------------------------------------------------------------
// Inner storage, FP32 accumulation: one warp, four rows, the 16-byte vectors
// [v0, v1) of each.  Four rows share every read of x: with one row per warp
// the 32 bytes of x per 16 bytes of matrix were two thirds of the shared-memory
// traffic that bounds a product whose rows sit in shared memory (4099 unknowns
// in 16 bits, 74% of them there: 7.1 -> 4.5 us).  Vectors below kv are in
// shared memory; a missing row repeats the last one.
template <class TA>
__device__ __forceinline__ void rs_quad(const uint4* A, const uint4* sA, int t0, int nr, int kv, int nvec,
                                        int v0, int v1, const float* xs, unsigned long long pol,
                                        float* acc) {
  constexpr int E = Dot16<TA>::E;
  const int lane = threadIdx.x & 31;
  const uint4 *p[4], *h[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int t = min(t0 + i, nr - 1);
    p[i] = A + (size_t)t * nvec;
    h[i] = sA + (size_t)t * kv;
    acc[i] = 0.f;
  }
  int v = max(v0, kv) + lane;
  for (; v + 32 < v1; v += 64) {
    uint4 q[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      q[i] = rs_ld(p[i] + v, pol);
      q[4 + i] = rs_ld(p[i] + v + 32, pol);
    }
#pragma unroll
    for (int u = 0; u < 2; ++u)
      Dot16<TA>::run4(acc, q + 4 * u, xs + (size_t)(v + 32 * u) * E);
  }
  if (v < v1) {
    uint4 q[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) q[i] = rs_ld(p[i] + v, pol);
    Dot16<TA>::run4(acc, q, xs + (size_t)v * E);
  }
  for (v = v0 + lane; v < min(v1, kv); v += 32) {
    uint4 q[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) q[i] = h[i][v];
    Dot16<TA>::run4(acc, q, xs + (size_t)v * E);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) acc[i] = warp_sum(acc[i]);
}

// The same with one warp per row, for a matrix larger than L2 (RsArgs::stream; no
// heads in shared memory): HBM bounds it, and four loads in flight per lane along
// one row beat eight over four rows (16383 unknowns in FP16: 81 against 84 us)
template <class TA>
__device__ __forceinline__ float rs_row_lowp(const uint4* row, int nvec, const float* xs, unsigned long long pol) {
  constexpr int E = Dot16<TA>::E;
  constexpr int U = 4;
  const int lane = threadIdx.x & 31;
  float acc = 0.f;
  int v = lane;
  for (; v + 32 * (U - 1) < nvec; v += 32 * U) {
    uint4 q[U];
#pragma unroll
    for (int u = 0; u < U; ++u) q[u] = rs_ld(row + v + 32 * u, pol);
#pragma unroll
    for (int u = 0; u < U; ++u) acc = Dot16<TA>::run(acc, q[u], xs + (size_t)(v + 32 * u) * E);
  }
  for (; v < nvec; v += 32) acc = Dot16<TA>::run(acc, rs_ld(row + v, pol), xs + (size_t)v * E);
  return warp_sum(acc);
}

// FP64 storage
__device__ __forceinline__ double rs_row_f64(const uint4* row, const uint4* head, int kv, int nvec,
                                             const double* xs, unsigned long long pol) {
  const int lane = threadIdx.x & 31;
  const double2* x2 = reinterpret_cast<const double2*>(xs);
  double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
  int v = kv + lane;
  for (; v + 32 < nvec; v += 64) {
    const uint4 q0 = rs_ld(row + v, pol), q1 = rs_ld(row + v + 32, pol);
    const double2 b0 = x2[v], b1 = x2[v + 32];
    a0 = fma(__hiloint2double(q0.y, q0.x), b0.x, a0);
    a1 = fma(__hiloint2double(q0.w, q0.z), b0.y, a1);
    a2 = fma(__hiloint2double(q1.y, q1.x), b1.x, a2);
    a3 = fma(__hiloint2double(q1.w, q1.z), b1.y, a3);
  }
  for (; v < nvec; v += 32) {
    const uint4 q0 = rs_ld(row + v, pol);
    const double2 b0 = x2[v];
    a0 = fma(__hiloint2double(q0.y, q0.x), b0.x, a0);
    a1 = fma(__hiloint2double(q0.w, q0.z), b0.y, a1);
  }
  for (v = lane; v < kv; v += 32) {
    const uint4 q0 = head[v];
    const double2 b0 = x2[v];
    a2 = fma(__hiloint2double(q0.y, q0.x), b0.x, a2);
    a3 = fma(__hiloint2double(q0.w, q0.z), b0.y, a3);
  }
  return warp_sum((a0 + a1) + (a2 + a3));
}

// hi + lo (or hi alone) storage with double-float x: short runs in double-float,
// flushed into a three-float sum (see tfl)
template <bool LO, int U>
__device__ __forceinline__ tfl rs_row_hilo(const float4* rh, const float4* rl, int nvec,
                                           const float4* xh, const float4* xl) {
  const int lane = threadIdx.x & 31;
  tfl acc = {0.f, 0.f, 0.f};
  int v = lane;
  for (; v + 32 * (U - 1) < nvec; v += 32 * U) {
    float4 h[U], l[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      h[u] = __ldcs(rh + v + 32 * u);
      l[u] = LO ? __ldcs(rl + v + 32 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    dfl run = {0.f, 0.f};
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const float4 p = xh[v + 32 * u], q = xl[v + 32 * u];
      run = df_acc_prod(run, h[u].x, l[u].x, p.x, q.x);
      run = df_acc_prod(run, h[u].y, l[u].y, p.y, q.y);
      run = df_acc_prod(run, h[u].z, l[u].z, p.z, q.z);
      run = df_acc_prod(run, h[u].w, l[u].w, p.w, q.w);
    }
    tf_add(acc, run.hi, run.lo);
  }
  for (; v < nvec; v += 32) {
    const float4 h = __ldcs(rh + v);
    const float4 l = LO ? __ldcs(rl + v) : make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 p = xh[v], q = xl[v];
    dfl run = {0.f, 0.f};
    run = df_acc_prod(run, h.x, l.x, p.x, q.x);
    run = df_acc_prod(run, h.y, l.y, p.y, q.y);
    run = df_acc_prod(run, h.z, l.z, p.z, q.z);
    run = df_acc_prod(run, h.w, l.w, p.w, q.w);
    tf_add(acc, run.hi, run.lo);
  }
  return tf_warp_sum(acc);
}

// 16-byte copies of n elements of T (n a multiple of 64) from global memory
// written by other CTAs into shared memory, by the row warps
template <class T>
__device__ __forceinline__ void rs_stage(T* dst, const void* src, long long n, int nthr) {
  const uint4* s = reinterpret_cast<const uint4*>(src);
  uint4* d = reinterpret_cast<uint4*>(dst);
  const int nv = (int)(n * sizeof(T) / 16);
#pragma unroll 4
  for (int c = threadIdx.x; c < nv; c += nthr) d[c] = __ldcg(s + c);
}

// ---------------------------------------------------------------------------
// the kernel: blockDim = 32 (row warps + 1), grid = RsArgs::G, one CTA per SM
// ---------------------------------------------------------------------------
template <class TA, class VT>
__global__ void __launch_bounds__(1024, 1) k_resident(const __grid_constant__ RsArgs a) {
  constexpr bool RC = sizeof(VT) == 4;      // refined scheme: recycled space, hi + lo residuals
  typedef RsAcc<VT, true> AC;        // dots of w and of z_0
  typedef RsAcc<VT, !RC> AZ;         // dots of the later z_j
  extern __shared__ __align__(16) unsigned char sm[];
  VT* xs = reinterpret_cast<VT*>(sm);       // 8 ld bytes: x (FP64), or hi and lo
  const RsLayout& L = a.L;
  VT* V = reinterpret_cast<VT*>(sm + L.V);  // (m + 1) x R
  VT* C = reinterpret_cast<VT*>(sm + L.C);  // RS_RQ x R
  VT* sw = reinterpret_cast<VT*>(sm + L.w);
  double* sr = reinterpret_cast<double*>(sm + L.r);
  double* sx = reinterpret_cast<double*>(sm + L.xo);   // x, then the last increment (2 x R)
  typedef typename AC::S PS;
  typedef typename AC::T PT;
  PS* s1 = reinterpret_cast<PS*>(sm + L.s1);           // reduced dots of w
  PS* s3 = reinterpret_cast<PS*>(sm + L.s3);           // reduced dots of z_j, 2 halves
  const int s3n = a.prow;
  double* ry = reinterpret_cast<double*>(sm + L.ry);   // row products of a residual (16 bytes a row)
  double* h_cs = reinterpret_cast<double*>(sm + L.cs);
  double* h_sn = reinterpret_cast<double*>(sm + L.sn);
  double* h_g = reinterpret_cast<double*>(sm + L.g);
  double* h_raw = reinterpret_cast<double*>(sm + L.hraw);
  double* h_braw = reinterpret_cast<double*>(sm + L.braw);
  double* h_fin = reinterpret_cast<double*>(sm + L.hfin);   // a Hessenberg column being finished
  double* h_new = reinterpret_cast<double*>(sm + L.hnew);    // the provisional column, not yet accepted
  double* h_bnew = reinterpret_cast<double*>(sm + L.bnew);
  double* h_rinv = reinterpret_cast<double*>(sm + L.rinv);  // 1 / R_ii
  double* Hm = reinterpret_cast<double*>(sm + L.H);    // column c at c (c + 1) / 2
  double* Bm = reinterpret_cast<double*>(sm + L.B);    // column c at c RS_RQ
  double* c0 = reinterpret_cast<double*>(sm + L.c0);
  double* y = reinterpret_cast<double*>(sm + L.y);
  double* tq = reinterpret_cast<double*>(sm + L.tq);
  double* Ri = reinterpret_cast<double*>(sm + L.Ri);
  double* Mq = reinterpret_cast<double*>(sm + L.Mq);
  float* RiF = reinterpret_cast<float*>(sm + L.RiF);
  float* MqF = reinterpret_cast<float*>(sm + L.MqF);
  double* zmean = reinterpret_cast<double*>(sm + L.zmean);   // (m + 1) x nobs
  double* umean = reinterpret_cast<double*>(sm + L.umean);   // RS_RQ x nobs
  VT* f1 = reinterpret_cast<VT*>(sm + L.f1);                  // y, and c_0 - B y from m + 2 on
  VT* swt = reinterpret_cast<VT*>(sm + L.wt);                // 1 / M, diagonal and row flip of the own rows (3 x R)
  uint4* sA = reinterpret_cast<uint4*>(sm + L.A);            // kv vectors of every own row
  __shared__ int s_ok, s_done, s_iters, s_nonf, s_state, s_kd, s_kn, s_lost;
  __shared__ double s_bprev, s_ua, s_ub;   // the Hessenberg warp's, between its two parts
  __shared__ double s_gpre, s_rn, s_inv, s_tol, s_red[4];
  __shared__ double s_nu, s_hj, s_beta;
  __shared__ tfl s_less[2];                // z_j^T w and |w|^2 less their parts in [C, V]
  __shared__ VT s_c, s_s;
  __shared__ VT s_xc[BIE_MAXB];
  __shared__ double s_dm[BIE_MAXB];
  __shared__ VT s_inu, s_ib, s_vh;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nw = blockDim.x >> 5, nrw = nw - 1, nrt = 32 * nrw;
  const bool hwarp = warp == nrw;           // the Hessenberg warp; the others take rows
  const int R = a.R, G = a.G, N = a.N, m = a.m, nobs = a.nobs;
  const long long ld = a.ld;
  const int c0r = blockIdx.x * R;           // own rows c0r .. c0r + nr - 1
  const int nr = max(0, min(R, N - c0r));
  VT* Z = a.zsm ? reinterpret_cast<VT*>(sm + L.Z) : reinterpret_cast<VT*>(a.Zg) + c0r;
  VT* Uc = a.zsm ? reinterpret_cast<VT*>(sm + L.U) : reinterpret_cast<VT*>(a.Ug) + c0r;
  const size_t zst = a.zsm ? (size_t)R : (size_t)ld;         // stride of Z and U columns
  VT* zb = reinterpret_cast<VT*>(a.zbuf);
  const size_t phalf = (size_t)a.prow * G;
  float4* const part1 = a.part;             // partial sums of w; then two halves of those of z_j
  auto part3 = [&](int h) -> float4* { return a.part + (h + 1) * phalf; };
  constexpr int E = 16 / (int)sizeof(TA);
  const int nvec = (int)(ld / E), kv = a.kv;
  const uint4* A = reinterpret_cast<const uint4*>(a.A) + (size_t)c0r * nvec;
  unsigned epoch = 0;
  unsigned long long pol;
  if (a.stream) asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  else asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));

  // the heads of the own rows, once; weights and signs of the own rows
  for (int t = warp; t < nr; t += nw)
    for (int v = lane; v < kv; v += 32) sA[(size_t)t * kv + v] = rs_ld(A + (size_t)t * nvec + v, pol);
  for (int t = threadIdx.x; t < nr; t += blockDim.x) {
    swt[t] = sizeof(VT) == 4 ? (VT)a.wgt[c0r + t] : (VT)a.wgt64[c0r + t];
    swt[R + t] = (VT)a.sgn[c0r + t];
    swt[2 * R + t] = (a.rowflip && a.blk[c0r + t] == 0) ? (VT)-1 : (VT)1;
  }
  auto flip = [&](int t) -> bool { return swt[2 * R + t] < (VT)0; };
  auto qv = [&](int q, int i) -> const VT* { return i < q ? C + (size_t)i * R : V + (size_t)(i - q) * R; };
  // The last CTA out zeroes the barrier for the next solve and reports: a CTA may have given
  // up at a barrier that the others passed, its rows of x then not being the result's.
  auto leave = [&]() {
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      if (atomicAdd(a.bar + 1, 1u) == (unsigned)G - 1) {
        __threadfence();
        const int err = *(volatile int*)a.err;
        a.out->timeout = err;
        a.bar[3] = !err && s_state != 2 && !s_nonf;
        a.bar[0] = 0;
        a.bar[1] = 0;
        __threadfence();
      }
    }
  };
  // partn[cta] = sum of v[t]^2 over the own rows (warps 0..3 at most take rows;
  // FP64 instructions of the other warps would cost as much as these)
  const int rwarps = min(4, (nr + 31) >> 5);
  auto norm_part = [&](const double* v) {
    if (warp < rwarps) {
      double acc = 0.0;
      for (int t = threadIdx.x; t < nr; t += 32 * rwarps) acc = fma(v[t], v[t], acc);
      acc = warp_sum(acc);
      if (lane == 0) s_red[warp] = acc;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int w2 = 0; w2 < rwarps; ++w2) t += s_red[w2];
      a.partn[blockIdx.x] = t;
    }
  };
  // the vector of the next residual over the own rows, divided by M_l, as the
  // product wants it (kind 4: FP32 in the inner storage's weights)
  auto publish = [&](int t, double v, int kind) {
    const int mrow = c0r + t;
    if constexpr (!RC) {
      reinterpret_cast<double*>(a.xh)[mrow] = v * a.wgt64[mrow];
    } else if (kind == 4) {
      a.xh[mrow] = (float)v * (float)swt[t];
    } else {
      const dfl d = df_from_double(v * a.wgt64[mrow]);
      a.xh[mrow] = d.hi;
      a.xl[mrow] = d.lo;
    }
  };

  __syncthreads();   // swt, sA
  // red[s R4 + t] = the column segment s's part of row t of the inner storage
  // times x (in xf): (row quad, segment) tasks over the row warps
  const int nquad = (nr + 3) >> 2, R4 = (R + 3) & ~3;
  const int nseg = a.stream ? 1 : max(1, 4 * nrw / R4);   // nseg R4 <= max(R4, 4 nrw)
  float* red = reinterpret_cast<float*>(sm + L.red);
  auto quads = [&](const float* xf) {
    if constexpr (RC) {
      if (a.stream) {
        for (int t = warp; t < nr; t += nrw) {
          const float y = rs_row_lowp<TA>(A + (size_t)t * nvec, nvec, xf, pol);
          if (lane == 0) red[t] = y;
        }
        return;
      }
      const int nch = (nvec + 31) >> 5;
      for (int task = warp; task < nquad * nseg; task += nrw) {
        const int sg = task / nquad, qd = task - sg * nquad;
        const int v0 = 32 * (nch * sg / nseg), v1 = min(nvec, 32 * (nch * (sg + 1) / nseg));
        float acc[4];
        rs_quad<TA>(A, sA, 4 * qd, nr, kv, nvec, v0, v1, xf, pol, acc);
        if (lane == 0) *reinterpret_cast<float4*>(red + sg * R4 + 4 * qd) = make_float4(acc[0], acc[1], acc[2], acc[3]);
      }
    }
  };
  auto row_sum = [&](int t) -> float {
    float y = 0.f;
    for (int sg = 0; sg < nseg; ++sg) y += red[sg * R4 + t];
    return y;
  };
  int q = 0, cycles = 0, total = 0;
  int kind = 0;                    // how the next residual is formed (0: D b)
  // state of the refinement, kept by thread 0 (every CTA from the same data)
  int stall = 0, r_exact = 1;
  double bnorm = 0.0, prev_rn = 0.0;

  // x = 0 (or the caller's guess, whose ||D b|| comes first)
  for (int t = threadIdx.x; t < nr; t += blockDim.x) sx[t] = a.x0 ? a.x[c0r + t] : 0.0;
  if (a.x0) {
    for (int t = threadIdx.x; t < nr; t += blockDim.x) {
      sr[t] = a.b[c0r + t];
      publish(t, sx[t], 1);
    }
    __syncthreads();
    norm_part(sr);
    kind = 1;
    if (!rs_barrier(a, epoch, &s_ok)) { leave(); return; }
    if (warp == 0) {
      const double s2 = rs_sum_partn(a.partn, G);
      bnorm = sqrt(s2);
      if (lane == 0) s_state = bnorm == 0.0;
    }
    __syncthreads();
    if (s_state) {   // b = 0 has the solution 0
      for (int t = threadIdx.x; t < nr; t += blockDim.x) {
        sx[t] = 0.0;
        publish(t, 0.0, 1);
      }
    }
    // the norms are read before the next phase's partials overwrite them
    if (!rs_barrier(a, epoch, &s_ok)) { leave(); return; }
  }

  for (int cycle = 0;; ++cycle) {
    // ---- RESID: r = D (b - A x), or r - D A_s d from the last increment ----
    // One warp per row forms the stored part's product; the diagonal term and
    // the difference follow with one thread per row (FP64 issue).
    if (kind == 0) {
      __syncthreads();
    } else if constexpr (!RC) {
      rs_stage<double>(reinterpret_cast<double*>(sm), a.xh, ld, blockDim.x);
      __syncthreads();
      for (int t = warp; t < nr; t += nw) {
        const double yv = rs_row_f64(A + (size_t)t * nvec, sA + (size_t)t * kv, kv, nvec,
                                     reinterpret_cast<const double*>(sm), pol);
        if (lane == 0) ry[2 * t] = yv;
      }
    } else if (kind == 4) {
      rs_stage<float>(reinterpret_cast<float*>(sm), a.xh, ld, blockDim.x);
      __syncthreads();
      if (!hwarp) quads(reinterpret_cast<const float*>(sm));
    } else {
      float* fh = reinterpret_cast<float*>(sm);
      float* fl = fh + ld;
      rs_stage<float>(fh, a.xh, ld, blockDim.x);
      rs_stage<float>(fl, a.xl, ld, blockDim.x);
      __syncthreads();
      const int nv4 = (int)(ld >> 2);
      const float4* xh4 = reinterpret_cast<const float4*>(fh);
      const float4* xl4 = reinterpret_cast<const float4*>(fl);
      for (int t = warp; t < nr; t += nw) {
        const float4* rh = reinterpret_cast<const float4*>(a.Ahi + (size_t)(c0r + t) * ld);
        const float4* rl = reinterpret_cast<const float4*>(a.Alo + (size_t)(c0r + t) * ld);
        const tfl yv = kind == 1 ? rs_row_hilo<true, 4>(rh, rl, nv4, xh4, xl4)
                                 : rs_row_hilo<false, 8>(rh, rl, nv4, xh4, xl4);
        if (lane == 0) *reinterpret_cast<float4*>(ry + 2 * t) = make_float4(yv.s, yv.e, yv.f, 0.f);
      }
    }
    __syncthreads();
    for (int t = threadIdx.x; t < nr; t += blockDim.x) {
      const double bv = kind >= 3 ? sr[t] : a.b[c0r + t];
      double o = bv;
      if (kind > 0) {
        double yv;
        if constexpr (RC) {
          if (kind == 4) {
            yv = (double)row_sum(t);
          } else {
            const float4 f = *reinterpret_cast<const float4*>(ry + 2 * t);
            yv = tf_to_double(tfl{f.x, f.y, f.z});
          }
        } else {
          yv = ry[2 * t];
        }
        yv = fma((double)swt[R + t], kind >= 3 ? sx[R + t] : sx[t], yv);
        // kinds 3, 4 update the flipped residual: D (D r - y) = r - D y
        o = kind >= 3 ? (flip(t) ? -bv : bv) - yv : bv - yv;
      }
      sr[t] = flip(t) ? -o : o;
    }
    __syncthreads();
    norm_part(sr);
    if (!rs_barrier(a, epoch, &s_ok)) { leave(); return; }
    // ---- START: |r|, tests (thread 0), z_0 ----
    if (warp == 0) {
      const double s2 = rs_sum_partn(a.partn, G);
      if (lane == 0) {
        const double rn = sqrt(s2);
        if (cycle == 0 && !a.x0) bnorm = rn;
        int state = 0;   // 1 converged, 2 non-finite, 3 stagnated, 4 out of cycles
        if (!isfinite(rn)) state = 2;
        else if (rn <= a.rtol * bnorm || rn == 0.0) state = 1;
        if (cycle > 0 && state == 0) {   // stagnation, as in run_solver
          stall = rn > 0.9 * prev_rn ? stall + 1 : 0;
          if (stall >= 3) state = 3;
        }
        prev_rn = cycle == 0 ? rn : fmin(prev_rn, rn);
        if (state == 0 && cycle >= a.max_cycles) state = 4;
        // the next residual (the rules of run_solver), if this cycle makes an increment and if not
        if (kind == 2) r_exact = 0;
        else if (kind <= 1) r_exact = 1;
        const int kn = RC && rn > 1e-4 * bnorm ? 2 : 1;
        int kd = kn;
        if (RC && r_exact && a.rtol >= 1e-14) {
          if (a.eps16 > 0.0 && a.eps16 * rn <= a.drift * bnorm) kd = 4;
          else if (0x1p-24 * rn <= a.drift * bnorm) kd = 3;
        }
        s_kd = kd;
        s_kn = kn;
        s_state = state;
        s_rn = rn;
        s_inv = 1.0 / rn;
        s_tol = fmax(a.inner_tol, 0.5 * a.rtol * bnorm / fmax(rn, 1e-300));
        s_done = 0;
        s_iters = 0;
        s_nonf = 0;
      }
    }
    __syncthreads();
    if (s_state != 0) break;
    for (int t = threadIdx.x; t < nr; t += blockDim.x) {
      const VT z = (VT)(sr[t] * s_inv);
      V[t] = z;
      Z[t] = z;
      zb[c0r + t] = z * swt[t];
    }
    __syncthreads();
    // C_i^T z_0, z_0^2, obstacle sums
    for (int i = warp; i <= q + nobs; i += nw) {
      PT s = AC::zero();
      if (i <= q) {
        const VT* ci = i < q ? C + (size_t)i * R : V;
        for (int t = lane; t < nr; t += 32) s = AC::mad(s, ci[t], V[t]);
      } else {
        const int k = i - q - 1;
        const int a0 = max(0, a.obs_off[k] - c0r), a1 = min(nr, a.obs_off[k + 1] - c0r);
        for (int t = a0 + lane; t < a1; t += 32) s = AC::addv(s, V[t]);
      }
      s = AC::warp(s);
      if (lane == 0) rs_put(part3(0), (size_t)i * G + blockIdx.x, AC::split(s));
    }
    if (!rs_barrier(a, epoch, &s_ok)) { leave(); return; }

    // Hessenberg columns j - 1 (final) and j (provisional), rotations, test; by the
    // Hessenberg warp (see k_dcgs for the derivation).  First what the sums alone give ...
    auto hcolumns = [&](int j) {
      const PS* S3 = s3 + (size_t)(j & 1) * s3n;
      auto v1 = [&](int i) -> double { return rs_value(s1[i]); };
      auto v3 = [&](int i) -> double { return rs_value(S3[i]); };
      for (int o = lane; o < nobs; o += 32)   // means of z_j over the obstacles
        zmean[(size_t)j * nobs + o] = v3(q + j + 1 + o) * (double)a.obs_invM[o];
      // column j - 1 is final: h + bprev a', subdiagonal bprev nu
      const double bprev = j > 0 ? h_raw[j] : 0.0;
      for (int i = lane; i < j; i += 32) {
        h_fin[i] = fma(bprev, v3(q + i), h_raw[i]);
        h_new[i] = v1(q + i);
      }
      for (int i = lane; i < q; i += 32) {
        if (j > 0) Bm[(size_t)(j - 1) * RS_RQ + i] = fma(bprev, v3(i), h_braw[i]);
        else c0[i] = v3(i);
        h_bnew[i] = v1(i);
      }
      __syncwarp();
      if (j > 0) {
        double ua, ub;
        rs_rotate2(h_fin, h_new, h_cs, h_sn, j - 1, ua, ub);
        if (lane == 0) {
          s_bprev = bprev;
          s_ua = ua;
          s_ub = ub;
        }
      }
      __syncwarp();
    };
    // ... then what takes nu, h_j and beta
    auto hfinish = [&](int j, bool lost, bool brk) {
      const double nu = s_nu, hj = s_hj, beta = s_beta;
      if (!lost) {   // the provisional column j replaces column j - 1 as the last raw one
        for (int i = lane; i < j; i += 32) h_raw[i] = h_new[i];
        for (int i = lane; i < q; i += 32) h_braw[i] = h_bnew[i];
        if (lane == 0) {
          h_raw[j] = hj;
          h_raw[j + 1] = beta;
        }
      }
      double gj = nu, uj = hj;   // z_0 = C c_0 + nu v_0: the right-hand side in H is nu e_1
      if (j > 0) {
        double c, s, rr, ir;
        rs_givens(s_ua, s_bprev * nu, c, s, rr, ir);
        const double gpre = s_gpre;
        gj = -s * gpre;
        uj = fma(-s, s_ub, c * hj);
        __syncwarp();
        if (lane == 0) {
          h_cs[j - 1] = c;
          h_sn[j - 1] = s;
          h_rinv[j - 1] = ir;
          h_g[j - 1] = c * gpre;
          h_fin[j - 1] = rr;
        }
        __syncwarp();
        double* Hc = Hm + (size_t)(j - 1) * j / 2;
        for (int i = lane; i < j; i += 32) Hc[i] = h_fin[i];
        __syncwarp();
      }
      if (lane == 0) {
        if (lost) {
          s_iters = j;
          if (!isfinite(gj)) s_nonf = 1;
          s_done = 1;
        } else {
          // |g_{j+1}| after the provisional rotation: |g_j| beta / sqrt(u_j^2 + beta^2)
          const double d = fma(uj, uj, beta * beta), e = gj * beta;
          const bool nf = !isfinite(d) || !isfinite(e);
          s_gpre = gj;
          s_iters = j + 1;
          if (nf) s_nonf = 1;
          if (nf || brk || e * e <= s_tol * s_tol * d || j + 1 >= m) s_done = 1;
        }
      }
      __syncwarp();
    };

    // ---- Arnoldi steps ----
    int k = 0;
    for (int j = 0;; ++j) {
      const int nb = q + j;   // basis vectors before z_j
      const bool lagged = a.lag && j > 0;
      // G(j)
      if (!hwarp) {
        const int n3 = nb + 1 + nobs;
        PS* S3 = s3 + (size_t)(j & 1) * s3n;
        auto take = [&](auto acc) {   // the dots of z_j reduce while it is staged
          typedef decltype(acc) A3;
          constexpr bool all = std::is_same<A3, AC>::value;   // the sums over obstacles too
          constexpr int LN = RC ? 16 : 32;
          const int nd = all ? n3 : nb + 1;
          typename A3::X ld3[A3::LD];
          // an obstacle's sum (three words) goes to a warp that has none of the first rows; with
          // more obstacles than warps they are all taken in rounds below
          const int ob = nrw - 1 - warp;
          const bool mine = !all && ob < nobs && nobs <= nrw && 2 * warp >= nd && nd <= nrt / LN &&
                            G <= 32 * A3::LD / 2;
          if constexpr (!all) {
            if (mine) {
#pragma unroll
              for (int u = 0; u < A3::LD / 2; ++u) {
                tfl v = {0.f, 0.f, 0.f};
                if (lane + 32 * u < G) rs_get(part3(j & 1), (size_t)(nb + 1 + ob) * G + lane + 32 * u, v);
                ld3[2 * u] = {v.s, v.e};
                ld3[2 * u + 1] = {v.f, 0.f};
              }
            } else {
              rs_load<A3, LN>(part3(j & 1), nd, G, ld3);
            }
          } else {
            rs_load<A3, LN>(part3(j & 1), nd, G, ld3);
          }
          rs_stage<VT>(xs, zb, ld, nrt);
          if constexpr (!all) {
            if (mine) {
              tfl s = {ld3[0].hi, ld3[0].lo, ld3[1].hi};
#pragma unroll
              for (int u = 1; u < A3::LD / 2; ++u) s = s + tfl{ld3[2 * u].hi, ld3[2 * u].lo, ld3[2 * u + 1].hi};
              s = tf_warp_sum(s);
              if (lane == 0) S3[nb + 1 + ob] = AC::pack(s);
            } else {
              rs_reduce<A3, LN>(part3(j & 1), nd, G, ld3, S3, nrt);
              for (int o = ob; o < nobs; o += nrw) {
                tfl s = {0.f, 0.f, 0.f};
                for (int c = lane; c < G; c += 32) {
                  tfl v;
                  rs_get(part3(j & 1), (size_t)(nb + 1 + o) * G + c, v);
                  s = s + v;
                }
                s = tf_warp_sum(s);
                if (lane == 0) S3[nb + 1 + o] = AC::pack(s);
              }
            }
          } else {
            rs_reduce<A3, LN>(part3(j & 1), nd, G, ld3, S3, nrt);
          }
        };
        if (j == 0) take(AC());
        else take(AZ());
        rs_bar_rows(nrt);
        if (nobs > 0) {   // P z_j: each obstacle's entries lower by coef mean / M
          if ((int)threadIdx.x < nobs)
            s_xc[threadIdx.x] = rs_share(S3[nb + 1 + threadIdx.x], a.obs_invM[threadIdx.x], a.obs_coef);
          for (int o = 0; o < nobs; ++o) {
            const VT im = (VT)a.obs_invM[o];
            const VT cw = rs_share(S3[nb + 1 + o], im, a.obs_coef) * im;
            for (int c = a.obs_off[o] + (int)threadIdx.x; c < a.obs_off[o + 1]; c += nrt) xs[c] -= cw;
          }
          rs_bar_rows(nrt);
        }
        const VT* zj = V + (size_t)j * R;
        if constexpr (RC) {
          quads(reinterpret_cast<const float*>(xs));
        } else {
          for (int t = warp; t < nr; t += nrw) {
            const double yv = rs_row_f64(A + (size_t)t * nvec, sA + (size_t)t * kv, kv, nvec,
                                         reinterpret_cast<const double*>(xs), pol);
            if (lane == 0) ry[2 * t] = yv;
          }
        }
        rs_bar_rows(nrt);
        for (int t = threadIdx.x; t < nr; t += nrt) {
          VT yv;
          if constexpr (RC) yv = row_sum(t);
          else yv = ry[2 * t];
          VT xm = zj[t];
          if (nobs > 0 && c0r + t >= a.obs0) {
            int o = 0;
            while (o + 1 < nobs && c0r + t >= a.obs_off[o + 1]) ++o;
            xm -= s_xc[o];
          }
          sw[t] = fma(swt[R + t], xm, yv) * swt[2 * R + t];
        }
        rs_bar_rows(nrt);
        for (int i = warp; i <= nb + 1; i += nrw) {
          const VT* qi = i <= nb ? qv(q, i) : sw;
          PT s = AC::zero();
          for (int t = lane; t < nr; t += 32) s = AC::mad(s, qi[t], sw[t]);
          s = AC::warp(s);
          if (lane == 0) rs_put(part1, (size_t)i * G + blockIdx.x, AC::split(s));
        }
      } else if (lagged) {
        hcolumns(j - 1);
        hfinish(j - 1, false, false);
      }
      if (!rs_barrier(a, epoch, &s_ok)) { leave(); return; }
      if (lagged && s_done) {   // the previous step ended the cycle; this product is dropped
        k = s_iters;
        break;
      }
      // D(j)
      if (a.pf_bytes > 0 && threadIdx.x == 0) {   // head of the own rows into L2 for the next product
        const unsigned char* p = reinterpret_cast<const unsigned char*>(A);
        const long long pfb = min(a.pf_bytes, (long long)nr * nvec * 16);
        for (long long o = 0; o < pfb; o += 65536) {
          const unsigned n = (unsigned)min(65536LL, pfb - o);
          asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p + o), "r"(n) : "memory");
        }
      }
      {
        typename AC::X ld1[AC::LD];
        if (G > 16 * AC::LD) {
          rs_load<AC, 32>(part1, nb + 2, G, ld1);
          rs_reduce<AC, 32>(part1, nb + 2, G, ld1, s1, blockDim.x);
        } else {
          rs_load<AC, 16>(part1, nb + 2, G, ld1);
          rs_reduce<AC, 16>(part1, nb + 2, G, ld1, s1, blockDim.x);
        }
      }
      __syncthreads();
      const PS* S3 = s3 + (size_t)(j & 1) * s3n;
      // The row warps subtract the basis from z_j (into vn, free until z_{j+1} goes there) and
      // from w, while one warp forms the scalars the rows take, three the Hessenberg
      // column's (FP64 vectors: the same ones) and the Hessenberg warp the columns
      VT* vj = V + (size_t)j * R;
      VT* vn = V + (size_t)(j + 1) * R;
      const int nrow_w = RC ? nrw - 3 : nrw;          // row warps here, the last of them for the scalars
      if (hwarp) {
        if (!a.lag) hcolumns(j);
        rs_bar_scal(RC ? 96 : 64);
        const bool lost = s_lost == 2, brk = s_lost != 0;
        if (!a.lag || brk || j + 1 >= m) {            // the test is made in this phase
          if (a.lag) hcolumns(j);
          hfinish(j, lost, brk);
        }
      } else if (warp >= nrow_w) {                    // RC: the Hessenberg column's scalars, a sum each
        if constexpr (RC) {
          tfl v;
          if (warp == nrow_w) {
            rs_sc(S3[nb], v);
            const tfl nu2 = v - rs_sum<tfl>(S3, S3, nb);
            const tfl inu = rs_rsqrt_pos(nu2);
            const double nu = tf_to_double(nu2 * inu);
            asm volatile("bar.sync 4, 96;" ::: "memory");
            const tfl hj = s_less[0] * inu;
            const tfl be2 = s_less[1] - hj * hj;
            const double beta = tf_to_double(be2 * rs_rsqrt_pos(be2));
            if (lane == 0) {
              s_nu = nu;
              s_hj = tf_to_double(hj);
              s_beta = beta;
            }
            rs_arrive_scal(96);
          } else {
            const bool sg = warp == nrow_w + 1;
            rs_sc(s1[sg ? nb : nb + 1], v);
            v = v - rs_sum<tfl>(sg ? S3 : s1, s1, nb);
            if (lane == 0) s_less[sg ? 0 : 1] = v;
            __syncwarp();
            asm volatile("bar.arrive 4, 96;" ::: "memory");
          }
        }
      } else {
        if (warp == nrow_w - 1) {
          typedef typename RsHead<VT>::T T;
          const RsScal<T> r = rs_scalars<T>(S3, s1, nb);
          if (lane == 0) {
            const VT nuh = rs_head(r.nu), bh = rs_head(r.beta), vh = rs_head(r.hj);
            // z_j lies in span [C, V] (to rounding): column j - 1 is the cycle's last one
            const bool lost = !(nuh > (VT)0) || !isfinite(nuh) || !isfinite(vh);
            const bool brk = lost || !(bh > (VT)0) || !isfinite(bh);
            if constexpr (!RC) {
              s_nu = r.nu;
              s_hj = r.hj;
              s_beta = r.beta;
            }
            s_vh = vh;
            s_inu = rs_head(r.inu);
            s_ib = brk ? (VT)0 : rs_head(r.ibe);
            s_lost = lost ? 2 : brk ? 1 : 0;
          }
          rs_arrive_scal(RC ? 96 : 64);
        } else {
          for (int t = threadIdx.x; t < nr; t += 32 * (nrow_w - 1)) {
            VT tv = vj[t], u = sw[t];
#pragma unroll 4
            for (int i = 0; i < nb; ++i) {
              const VT v = qv(q, i)[t];
              tv -= rs_head(S3[i]) * v;
              u -= rs_head(s1[i]) * v;
            }
            vn[t] = tv;
            sw[t] = u;
          }
        }
        rs_bar_rows(32 * nrow_w);
        const bool lost = s_lost == 2, brk = s_lost != 0;
        if (!lost) {
          const VT inu = s_inu, ib = s_ib, vh = s_vh;
          for (int t = threadIdx.x; t < nr; t += 32 * nrow_w) {
            const VT tv = vn[t], u = sw[t];
            const VT vt = tv * inu;
            vj[t] = vt;
            const VT zz = brk ? (VT)0 : (u - vh * vt) * ib;
            vn[t] = zz;
            Z[(size_t)(j + 1) * zst + t] = zz;
            zb[c0r + t] = zz * swt[t];
          }
          rs_bar_rows(32 * nrow_w);
          // a' = Q_i^T z_{j+1} (i <= nb, v_j included), |z_{j+1}|^2, obstacle sums
          float4* p3 = part3((j + 1) & 1);
          const int nrow = nb + 2 + nobs;
          for (int i = warp; i < nrow; i += nrow_w) {
            if (i <= nb + 1) {
              const VT* qi = qv(q, i);
              typename AZ::T s = AZ::zero();
              for (int t = lane; t < nr; t += 32) s = AZ::mad(s, qi[t], vn[t]);
              s = AZ::warp(s);
              if (lane == 0) rs_put(p3, (size_t)i * G + blockIdx.x, AZ::split(s));
            } else {
              const int o = i - (nb + 2);
              const int a0 = max(0, a.obs_off[o] - c0r), a1 = min(nr, a.obs_off[o + 1] - c0r);
              typename AC::T s = AC::zero();
              for (int t = a0 + lane; t < a1; t += 32) s = AC::addv(s, vn[t]);
              s = AC::warp(s);
              if (lane == 0) rs_put(p3, (size_t)i * G + blockIdx.x, AC::split(s));
            }
          }
        }
      }
      if (!rs_barrier(a, epoch, &s_ok)) { leave(); return; }
      if ((!a.lag || s_lost != 0 || j + 1 >= m) && s_done) {   // the test was made in this phase
        k = s_iters;
        break;
      }
    }
    if (s_nonf) break;

    // ---- UPDATE with k columns ----
    const int ext = (RC && k >= 1 && k <= RS_RK && q + k <= RS_RQ) ? 1 : 0;
    kind = k > 0 ? s_kd : s_kn;
    if (k > 0) {
      PS* pa = s3 + (size_t)(k & 1) * s3n;                    // dots of z_k, q + k + 1
      {
        typename AZ::X ld3[AZ::LD];
        rs_load<AZ, 16>(part3(k & 1), q + k + 1, G, ld3);
        rs_reduce<AZ, 16>(part3(k & 1), q + k + 1, G, ld3, pa, blockDim.x);
      }
      __syncthreads();
      auto pv = [&](int i) -> double { return rs_value(pa[i]); };
      double* hl = h_fin;                                     // column k - 1
      double* bl = h_braw;                                    // becomes its C-part
      auto Rent = [&](int i, int c) -> double { return c == k - 1 ? hl[i] : Hm[(size_t)c * (c + 1) / 2 + i]; };
      auto Bent = [&](int l, int i) -> double { return i == k - 1 ? bl[l] : Bm[(size_t)i * RS_RQ + l]; };
      if (warp == 0) {
        const double bk = h_raw[k];
        for (int i = lane; i < k; i += 32) hl[i] = fma(bk, pv(q + i), h_raw[i]);
        for (int l = lane; l < q; l += 32) bl[l] = fma(bk, pv(l), bl[l]);
        __syncwarp();
        const double u = givens_apply_warp(hl, h_cs, h_sn, k - 1);
        rs_bar_scal(64);
        const double nu = s_nu;
        double c, s, rr, ir;
        rs_givens(u, bk * nu, c, s, rr, ir);
        if (lane == 0) {
          hl[k - 1] = rr;
          h_rinv[k - 1] = ir;
          s_c = (VT)c;
          s_s = (VT)s;
        }
        __syncwarp();
        // warp 1 forms R^-1 and -B R^-1 beside this warp's solve for y
        if (ext) asm volatile("bar.sync 2, 64;" ::: "memory");
        const double gl = c * s_gpre;
        if (k <= 32) {   // by columns with y_i in lane i
          double yv = 0.0, rv = 0.0;
          if (lane < k) {
            yv = lane == k - 1 ? gl : h_g[lane];
            rv = h_rinv[lane];
          }
          for (int l = k - 1; l >= 0; --l) {
            const double Rc = lane < l ? Rent(lane, l) : 0.0;
            if (lane == l) yv *= rv;
            const double yl = __shfl_sync(0xffffffffu, yv, l);
            if (lane < l) yv = fma(-Rc, yl, yv);
          }
          if (lane < k) {
            y[lane] = yv;
            f1[lane] = (VT)yv;
          }
          __syncwarp();
        } else {
          for (int i = k - 1; i >= 0; --i) {
            double t = 0.0;
            for (int l = i + 1 + lane; l < k; l += 32) t += Rent(i, l) * y[l];
            t = warp_sum(t);
            if (lane == 0) y[i] = ((i == k - 1 ? gl : h_g[i]) - t) * h_rinv[i];
            __syncwarp();
          }
          for (int i = lane; i < k; i += 32) f1[i] = (VT)y[i];
        }
        for (int l = lane; l < q; l += 32) {   // c_0 - B y
          double t = c0[l];
          for (int i = 0; i < k; ++i) t = fma(-Bent(l, i), y[i], t);
          tq[l] = t;
          f1[m + 2 + l] = (VT)t;
        }
      } else if (warp == 2) {   // the norm of z_k less its parts, beside warp 0's rotations
        double ta = 0.0;
        for (int i = lane; i < q + k; i += 32) ta = fma(pv(i), pv(i), ta);
        ta = warp_sum(ta);
        const double nu2 = pv(q + k) - ta, inu = rs_rsqrt_pos(nu2);
        if (lane == 0) {
          s_nu = nu2 * inu;
          s_inu = (VT)inu;
        }
        rs_arrive_scal(64);
      } else if (warp == 1 && ext) {
        asm volatile("bar.sync 2, 64;" ::: "memory");
        if (lane < k) {
          const int cc = lane;
          for (int i = k - 1; i > cc; --i) Ri[i * RS_RK + cc] = 0.0;
          for (int i = cc; i >= 0; --i) {
            double t = i == cc ? 1.0 : 0.0;
            for (int l = i + 1; l <= cc; ++l) t -= Rent(i, l) * Ri[l * RS_RK + cc];
            Ri[i * RS_RK + cc] = t * h_rinv[i];
          }
          for (int i = 0; i < k; ++i) RiF[i * RS_RK + cc] = (float)Ri[i * RS_RK + cc];
        }
        __syncwarp();
        for (int e = lane; e < q * k; e += 32) {
          const int l = e / k, cc = e - l * k;
          double t = 0.0;
          for (int i = 0; i <= cc; ++i) t = fma(-Bent(l, i), Ri[i * RS_RK + cc], t);
          Mq[l * RS_RK + cc] = t;
          MqF[l * RS_RK + cc] = (float)t;
        }
      }
      __syncthreads();
      // coef x the correction's mean over each obstacle: a warp per obstacle
      for (int o = warp; o < nobs; o += nw) {
        double t = 0.0;
        for (int i = lane; i < k + q; i += 32)
          t = i < k ? fma(y[i], zmean[(size_t)i * nobs + o], t)
                    : fma(tq[i - k], umean[(size_t)(i - k) * nobs + o], t);
        t = warp_sum(t);
        if (lane == 0) s_dm[o] = (double)a.obs_coef * t;
      }
      __syncthreads();
    }
    // the own rows: x on the first warps, the new U columns on the others, their
    // means on the Hessenberg warp
    if (warp < rwarps) {
      for (int t = threadIdx.x; t < nr; t += 32 * rwarps) {
        if (k > 0) {
          const VT* yv = f1;
          const VT* tqv = f1 + m + 2;
          // runs of eight terms in the basis type, the runs summed in FP64
          double acc = 0.0;
          for (int i0 = 0; i0 < k; i0 += 8) {
            VT v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = i0 + u < k ? Z[(size_t)(i0 + u) * zst + t] : (VT)0;
            VT run = 0;
#pragma unroll
            for (int u = 0; u < 8; ++u)
              if (i0 + u < k) run = fma(yv[i0 + u], v[u], run);
            acc += (double)run;
          }
          for (int l0 = 0; l0 < q; l0 += 8) {
            VT v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = l0 + u < q ? Uc[(size_t)(l0 + u) * zst + t] : (VT)0;
            VT run = 0;
#pragma unroll
            for (int u = 0; u < 8; ++u)
              if (l0 + u < q) run = fma(tqv[l0 + u], v[u], run);
            acc += (double)run;
          }
          if (nobs > 0 && c0r + t >= a.obs0) {
            int o = 0;
            while (o + 1 < nobs && c0r + t >= a.obs_off[o + 1]) ++o;
            acc -= s_dm[o];
          }
          const double dlt = s_rn * acc;
          sx[t] += dlt;
          sx[R + t] = dlt;
          if (ext) {   // C gains the cycle's rotated V (see k_update)
            const PS* pa = s3 + (size_t)(k & 1) * s3n;
            VT vk = V[(size_t)k * R + t];
#pragma unroll 4
            for (int l = 0; l < q + k; ++l) vk -= rs_head(pa[l]) * qv(q, l)[t];
            vk *= s_inu;
            VT cur = V[t];
            for (int i = 0; i < k; ++i) {
              const VT nxt = i + 1 < k ? V[(size_t)(i + 1) * R + t] : vk;
              const VT ci = i + 1 < k ? (VT)h_cs[i] : s_c, si = i + 1 < k ? (VT)h_sn[i] : s_s;
              C[(size_t)(q + i) * R + t] = ci * cur + si * nxt;
              cur = -si * cur + ci * nxt;
            }
          }
        }
        publish(t, kind >= 3 ? sx[R + t] : sx[t], kind);
      }
    } else if (ext && !hwarp) {   // U gains (Z - U B) R^-1
      for (int e = threadIdx.x - 32 * rwarps; e < nr * k; e += nrt - 32 * rwarps) {
        const int cc = e / nr, t = e - cc * nr;
        VT s = 0;
        for (int i = 0; i <= cc; ++i) s += (VT)RiF[i * RS_RK + cc] * Z[(size_t)i * zst + t];
#pragma unroll 4
        for (int l = 0; l < q; ++l) s += (VT)MqF[l * RS_RK + cc] * Uc[(size_t)l * zst + t];
        Uc[(size_t)(q + cc) * zst + t] = s;
      }
    } else if (ext && hwarp) {   // means of the new U columns
      for (int e = lane; e < nobs * k; e += 32) {
        const int o = e / k, cc = e - o * k;
        double t = 0.0;
        for (int i = 0; i <= cc; ++i) t = fma(zmean[(size_t)i * nobs + o], Ri[i * RS_RK + cc], t);
        for (int l = 0; l < q; ++l) t = fma(umean[(size_t)l * nobs + o], Mq[l * RS_RK + cc], t);
        umean[(size_t)(q + cc) * nobs + o] = t;
      }
    }
    if (ext) q += k;
    total += k;
    ++cycles;
    if (!rs_barrier(a, epoch, &s_ok)) { leave(); return; }
  }
  for (int t = threadIdx.x; t < nr; t += blockDim.x) a.x[c0r + t] = sx[t];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    RsOut* o = a.out;
    o->iters = total;
    o->cycles = cycles;
    o->converged = s_state == 1;
    o->nonfinite = s_state == 2 || s_nonf;
    o->stagnated = s_state == 3;
    o->rnorm = s_rn;
    o->bnorm = bnorm;
  }
  leave();
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
struct RsPlan {
  RsLayout L;
  int R, G, threads, kv, zsm, lag, stream;
};

// Rows per CTA, warps and the shared-memory layout; false when the solve does
// not fit (the kernel-by-kernel solver takes it).
static bool rs_plan(const bie_ctx* c, const bie_solve_opts* o, int nobs, RsPlan& P) {
  const int N = c->N, m = o->restart;
  const bool f64 = c->precision == BIE_FP64;
  const size_t vt = f64 ? 8 : 4, ta = f64 ? 8 : c->precision == BIE_FP32_IR ? 4 : 2;
  if (N > RS_MAXN || m < 1 || m > 256) return false;
  const int nsm = gemv_num_ctas();
  // one row per row warp on small problems (few CTAs: fewer partial sums; 640
  // unknowns take 21 CTAs), beyond that every SM
  // (the FP64 products are bound by FP64 issue: every SM from the start)
  P.G = f64 ? nsm : std::min(nsm, (N + RS_MINROWS - 1) / RS_MINROWS);
  P.R = (N + P.G - 1) / P.G;
  P.G = (N + P.R - 1) / P.R;
  int nrw = 31;
  long long best = -1;
  for (int w = 31; w >= 20; --w) {   // rounds x warps, ties to more warps
    const long long cost = (long long)((P.R + w - 1) / w) * w;
    if (best < 0 || cost < best) {
      best = cost;
      nrw = w;
    }
  }
  P.threads = 32 * (nrw + 1);
  const size_t R = P.R, rq = f64 ? 0 : RS_RQ, no = std::max(1, nobs);
  size_t at = 8 * (size_t)c->ld;
  auto take = [&](size_t bytes) {
    const size_t p = at;
    at += (bytes + 15) / 16 * 16;
    return (unsigned)p;
  };
  RsLayout& L = P.L;
  L.V = take(vt * (m + 1) * R);
  L.C = take(vt * rq * R);
  L.w = take(vt * R);
  L.r = take(8 * R);
  L.ry = take(16 * R);
  L.red = take(4 * (4 * 32 + R + 4));
  L.xo = take(8 * 2 * R);
  L.wt = take(vt * 3 * R);
  const size_t ps = f64 ? sizeof(RsAcc<double, true>::S) : sizeof(RsAcc<float, true>::S);
  L.s1 = take(ps * (m + 2 + RS_RQ));
  L.s3 = take(ps * 2 * (m + 2 + RS_RQ + (size_t)nobs));
  L.cs = take(8 * m);
  L.sn = take(8 * m);
  L.g = take(8 * (m + 1));
  L.hraw = take(8 * (m + 2));
  L.braw = take(8 * RS_RQ);
  L.hfin = take(8 * (m + 2));
  L.hnew = take(8 * (m + 2));
  L.bnew = take(8 * RS_RQ);
  L.rinv = take(8 * (m + 1));
  L.H = take(8 * (size_t)m * (m + 1) / 2);
  L.B = take(8 * rq * m);
  L.c0 = take(8 * RS_RQ);
  L.y = take(8 * m);
  L.tq = take(8 * RS_RQ);
  L.Ri = take(8 * RS_RK * RS_RK);
  L.Mq = take(8 * RS_RQ * RS_RK);
  L.RiF = take(4 * RS_RK * RS_RK);
  L.MqF = take(4 * RS_RQ * RS_RK);
  L.zmean = take(8 * (m + 1) * no);
  L.umean = take(8 * RS_RQ * no);
  L.f1 = take(vt * (m + 2 + 2 * RS_RQ));
  if (at > RS_SMEM_MAX) return false;
  // Z and U, then the heads of the own rows, while there is room
  const size_t zu = (vt * (m + 1) * R + 15) / 16 * 16 + (vt * rq * R + 15) / 16 * 16;
  P.zsm = at + zu <= RS_SMEM_MAX ? 1 : 0;
  L.Z = L.U = 0;
  if (P.zsm) {
    L.Z = take(vt * (m + 1) * R);
    L.U = take(vt * rq * R);
  }
  const long long nvec = c->ld * (long long)ta / 16;
  long long kv = (long long)(RS_SMEM_MAX - at) / (16 * (long long)R);
  kv = kv >= nvec ? nvec : kv / 32 * 32;
  const double abytes = (double)N * (double)c->ld * (double)ta;
  P.stream = abytes > 90e6 ? 1 : 0;
  if (P.stream) kv = 0;
  P.kv = (int)kv;
  L.A = take(16 * (size_t)kv * R);
  L.total = (unsigned)at;
  // a product beside the Hessenberg work is worth the one that is dropped per
  // cycle only while it is short (640 unknowns: 6 us; at 4099, 12 us, it cost 60 us a solve)
  P.lag = abytes <= 10e6 ? 1 : 0;
  return true;
}

template <class TA, class VT>
static cudaError_t rs_launch(const RsPlan& P, RsArgs& a, cudaStream_t st) {
  auto kern = k_resident<TA, VT>;
  cudaError_t e = raise_smem_limit((const void*)kern, P.L.total);
  if (e != cudaSuccess) return e;
  void* args[] = {&a};
  return cudaLaunchCooperativeKernel((const void*)kern, dim3(P.G), dim3(P.threads), args, P.L.total, st);
}

// Enqueue a solve of the assembled system (b, x as in solve_system) as one
// kernel; *taken = false (and nothing enqueued) when it does not qualify: a
// row-partitioned context (its products pass through the caller's exchange),
// profiling (events around every product), more than RS_MAXN unknowns or a
// restart length whose basis does not fit.  resident_result waits for it; *usable (may
// be NULL) points to a device word that is zero after a solve whose x is no iterate
// (non-finite, or a wait that ran out), for kernels enqueued behind it.
bie_status resident_launch(bie_ctx* c, const bie_solve_opts* o, double* x, const double* b, bool* taken,
                           const unsigned** usable) {
  *taken = false;
  if (partitioned(c) || c->profiling) return BIE_OK;
  const bool ir = c->precision != BIE_FP64;
  RsArgs a;
  memset(&a, 0, sizeof(a));
  int ob = 0;   // obstacles of the right preconditioner (see run_solver)
  if (ir && c->variant == 0 && !c->asm_noE) {
    if (!c->asm_vs && c->nb > 2) {
      ob = 2;
      a.obs_coef = 1.5f;
    } else if (c->asm_vs && c->nb > 1) {
      ob = 1;
      a.obs_coef = 0.5f;
    }
  }
  a.nobs = ob > 0 ? c->nb - ob : 0;
  a.obs0 = a.nobs > 0 ? c->off[ob] : c->N;
  for (int k = 0; k < a.nobs; ++k) {
    a.obs_off[k] = c->off[ob + k];
    a.obs_invM[k] = (float)(1.0 / (double)c->M[ob + k]);
  }
  a.obs_off[a.nobs] = a.nobs > 0 ? c->off[c->nb] : c->N;
  RsPlan P;
  if (!rs_plan(c, o, a.nobs, P)) return BIE_OK;
  BIE_NVTX("gmres_resident");
  const size_t NN = (size_t)c->N * (size_t)c->ld;
  const size_t vt = ir ? 4 : 8;
  a.N = c->N;
  a.m = o->restart;
  a.R = P.R;
  a.G = P.G;
  a.rowflip = o->row_flip ? 1 : 0;
  a.x0 = o->x0 != 0;
  a.max_cycles = o->max_cycles;
  a.lag = P.lag;
  a.kv = P.kv;
  a.zsm = P.zsm;
  a.stream = P.stream;
  a.ld = c->ld;
  a.rtol = o->rtol;
  a.inner_tol = o->inner_tol > 0.0 ? o->inner_tol
                : !ir ? 0.0 : c->precision == BIE_FP32_IR ? 1e-4 : 5e-4;
  a.eps16 = c->precision == BIE_FP16_IR ? 0x1p-11 : c->precision == BIE_BF16_IR ? 0x1p-8 : 0.0;
  if (a.eps16 > 0.0) a.eps16 += (double)(c->ld / 32) * 0x1p-24;   // FP32 sums of ld / 32 terms per lane
  a.drift = 6e-15;   // kResidDrift of gmres.cu
  bool oom = false;
  const void* A16 = nullptr;
  if (!ir) {
    a.A = ctx_buf(c, "A_f64", sizeof(double) * NN, &oom);
  } else {
    a.Ahi = (const float*)ctx_buf(c, "A_hi", sizeof(float) * NN, &oom);
    a.Alo = oom ? nullptr : (const float*)ctx_buf(c, "A_lo", sizeof(float) * NN, &oom);
    if (c->precision != BIE_FP32_IR && !oom) A16 = ctx_buf(c, "A_16", 2 * NN, &oom);
    a.A = c->precision == BIE_FP32_IR ? (const void*)a.Ahi : A16;
  }
  if (oom) return ctx_fail(c, BIE_ERR_OOM, "solve: stored matrix");
  a.wgt = (const float*)ctx_buf(c, "wgt", sizeof(float) * c->ld, &oom);
  a.wgt64 = (const double*)ctx_buf(c, "wgt64", sizeof(double) * c->ld, &oom);
  a.sgn = (const float*)ctx_buf(c, "sgn", sizeof(float) * c->ld, &oom);
  a.blk = (const int*)ctx_buf(c, "blk", sizeof(int) * c->ld, &oom);
  if (oom) return ctx_fail(c, BIE_ERR_OOM, "solve: node buffers");
  a.b = b;
  a.x = x;
  // one exchange buffer: z_j, xh, xl (zero past N), partial sums, barrier
  const size_t ldb = 8 * (size_t)c->ld;
  a.prow = a.m + 2 + RS_RQ + a.nobs;
  const size_t pbytes = 3 * sizeof(float4) * (size_t)a.prow * P.G;
  unsigned char* xb;
  unsigned* bar;
  BIE_GET(c, unsigned char, "rs_x", 3 * ldb, xb);
  unsigned char* pb;
  BIE_GET(c, unsigned char, "rs_part", pbytes + 8 * (size_t)P.G, pb);
  a.part = (float4*)pb;
  a.partn = (double*)(pb + pbytes);
  BIE_GET(c, unsigned, "rs_bar", 4, bar);
  if (c->rs_bar != bar) {
    BIE_CUDA_TRY(c, cudaMemsetAsync(bar, 0, 4 * sizeof(unsigned), c->stream));
    c->rs_bar = bar;
  }
  // The padding past N stays zero: N, ld and the element width say where it lies (the
  // FP64 scheme's doubles cover what are padding floats of a refined solve)
  if (c->rs_ld != c->ld || c->rs_n != c->N || c->rs_vt != (int)vt || c->rs_x != xb) {
    BIE_CUDA_TRY(c, cudaMemsetAsync(xb, 0, 3 * ldb, c->stream));
    c->rs_ld = c->ld;
    c->rs_n = c->N;
    c->rs_vt = (int)vt;
    c->rs_x = xb;
  }
  a.zbuf = xb;
  a.xh = (float*)(xb + ldb);
  a.xl = (float*)(xb + 2 * ldb);
  if (!P.zsm) {
    BIE_GET(c, unsigned char, "rs_Z", vt * (size_t)(a.m + 1) * c->ld, a.Zg);
    if (ir) BIE_GET(c, unsigned char, "rs_U", vt * (size_t)RS_RQ * c->ld, a.Ug);
  }
  a.bar = bar;
  if (usable) *usable = bar + 3;
  a.err = (int*)(bar + 2);
  a.spin_limit = 1u << 22;
  a.out = reinterpret_cast<RsOut*>(c->slots_dev);
  // as the kernel-by-kernel solver: a quarter of L2 is filled during the vector work
  if (P.stream) {
    int l2 = 0;
    cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, c->device);
    a.pf_bytes = ((long long)(0.25 * (double)l2) / P.G) & ~15LL;
  }
  a.L = P.L;
  reinterpret_cast<RsOut*>(c->slots_host)->timeout = 1;
  cudaError_t e;
  switch (c->precision) {
    case BIE_FP64: e = rs_launch<double, double>(P, a, c->stream); break;
    case BIE_FP32_IR: e = rs_launch<float, float>(P, a, c->stream); break;
    case BIE_FP16_IR: e = rs_launch<__half, float>(P, a, c->stream); break;
    default: e = rs_launch<__nv_bfloat16, float>(P, a, c->stream); break;
  }
  if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {
    cudaGetLastError();   // a device (or a share of one) that cannot hold the grid
    return BIE_OK;
  }
  if (e != cudaSuccess) return ctx_cuda(c, e, "k_resident");
  c->launches += 1;
  *taken = true;
  return BIE_OK;
}

// Wait for the stream and read the result of the last resident_launch.
bie_status resident_result(bie_ctx* c, bie_solve_info* info) {
  BIE_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  RsOut o;
  memcpy(&o, c->slots_host, sizeof(o));
  if (o.timeout) {
    c->rs_bar = nullptr;   // cleared again before the next solve
    return ctx_fail(c, BIE_ERR_TIMEOUT, "solve: a grid barrier gave up waiting");
  }
  if (info) {
    info->iters = o.iters;
    info->cycles = o.cycles;
    info->converged = o.converged;
    info->rel_resid = o.bnorm > 0 ? o.rnorm / o.bnorm : o.rnorm;
  }
  if (o.nonfinite) return ctx_fail(c, BIE_ERR_NAN, "solve: non-finite residual");
  if (!o.converged)
    return ctx_fail(c, BIE_ERR_NOCONV, o.stagnated ? "solve: residual stagnated above rtol"
                                                   : "solve: rtol not reached within max_cycles");
  return BIE_OK;
}
