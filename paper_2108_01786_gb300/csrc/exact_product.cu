// The full-accuracy (hi + lo, ~48-bit) operator times a block of columns on the
// tensor cores, by exact integer slices (an Ozaki-type splitting of both operands).
//
// Row m of the stored matrix is scaled by 2^-e_m (|A_ml| < 2^e_m) and cut into
// OZ_S slices of OZ_BITS bits: A_ml = 2^e_m sum_s a_s,ml 2^-5(s+1) + (below
// 2^-50 of the row scale), every a_s an integer with |a_0| <= 32, |a_s| <= 16,
// stored exactly in FP16.  Each column x_c (already divided by M_l) is cut the
// same way with its own scale 2^f_c.  With the integer sums of a level,
//   I_L = sum_{s+t=L} sum_l a_s,ml x_t,cl,
// y = 2^(e_m + f_c) sum_{L<S} 2^-5(L+2) I_L carries only the truncation of the
// pairs s + t >= S (2^-5S of the row scale) and the FP64 rounding of S terms.
//
// One kernel forms every level at once: the accumulators of level L are tensor-
// memory columns [L P, L P + P) (P: the columns padded to 16), so slice a_s
// times ALL the x slices t < S - s is one product whose result starts at column
// s P.  Each tile of A is read once and each tile of x once per K step for all S
// slices of A.  (One GEMM per slice with its own output per pair (s, t) read the
// x tiles again for every s, wrote 55 partial results per column and summed them
// in FP64; 8191 unknowns, 24 columns: 341 us of products and 79 us of sums, now
// 220 us = 6.1 TB/s of slices, 0.90 of the measured copy rate, and 9.6 us.)
// A piece of at most OZ_PIECE K tiles adds |I_L| <= 64 OZ_PIECE (2 x 512 + 8 x 256)
// < 2^24, so the FP32 accumulation is exact; pieces are added as 32-bit integers.
#include <algorithm>

#include "exact_product.cuh"
#include "nvtx.cuh"
#include "tc_common.cuh"

#define OZ_PIECE 84          // K tiles per exact FP32 accumulation (84 x 64 x 3072 < 2^24)
#define OZ_TILE 16384        // bytes of a 128 x 64 FP16 tile
#define OZ_STAGES 12         // most A tiles in flight
#define OZ_XSTAGES 2
#define OZ_RING (225 * 1024) // shared memory of the two rings

// e_m: max_l |A_ml| (1 + 2^-20) < 2^e_m, one warp per row
__global__ void k_oz_rowexp(int N, long long ld, const float* __restrict__ Ahi, int* __restrict__ e) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (warp >= N) return;
  const float4* row = reinterpret_cast<const float4*>(Ahi + (size_t)warp * ld);
  float mx = 0.f;
  for (long long v = lane; v < ld / 4; v += 32) {
    const float4 q = row[v];
    mx = fmaxf(mx, fmaxf(fmaxf(fabsf(q.x), fabsf(q.y)), fmaxf(fabsf(q.z), fabsf(q.w))));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) {
    int k = 0;
    if (mx > 0.f) frexp((double)mx * (1.0 + 0x1p-20), &k);   // mx (1 + 2^-20) < 2^k
    e[warp] = k;
  }
}

// Byte of element (row, col) in a 64-column tile as the tensor cores' 128-byte
// swizzle wants it: 16-byte chunk c of row r sits at chunk c ^ (r mod 8).
__device__ __forceinline__ int oz_swz(int row, int chunk) {
  return row * 128 + ((chunk ^ (row & 7)) << 4);
}

// Slices of the hi + lo storage (exact integers in FP16), laid out as the product
// reads them: unit (row block, K tile), then the slice, then a swizzled 128 x 64
// tile, so that one bulk copy of contiguous bytes fetches a tile and the S tiles
// of a unit follow one another.  Rows past N are zero.  One thread: eight columns.
__global__ void __launch_bounds__(256) k_oz_slice_A(int N, int nrb, long long ld,
                                                    const float* __restrict__ Ahi,
                                                    const float* __restrict__ Alo,
                                                    const int* __restrict__ e,
                                                    unsigned char* __restrict__ S) {
  const int nkt = (int)(ld / MM_KT);
  const size_t total = (size_t)nrb * nkt * 1024;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (size_t)gridDim.x * blockDim.x) {
    const size_t unit = i >> 10;
    const int r = (int)(i >> 3) & 127, ch = (int)i & 7;
    const int rb = (int)(unit / nkt), kt = (int)(unit - (size_t)rb * nkt);
    const int m = rb * 128 + r;
    unsigned char* dst = S + unit * ((size_t)OZ_S * OZ_TILE) + oz_swz(r, ch);
    if (m >= N) {
#pragma unroll
      for (int s = 0; s < OZ_S; ++s)
        *reinterpret_cast<uint4*>(dst + (size_t)s * OZ_TILE) = make_uint4(0, 0, 0, 0);
      continue;
    }
    const size_t src = (size_t)m * ld + (size_t)kt * MM_KT + ch * 8;
    float x[8], y[8];   // the entries scaled by 2^-e_m: x + y, |x + y| < 1
    *reinterpret_cast<float4*>(x) = *reinterpret_cast<const float4*>(Ahi + src);
    *reinterpret_cast<float4*>(x + 4) = *reinterpret_cast<const float4*>(Ahi + src + 4);
    *reinterpret_cast<float4*>(y) = *reinterpret_cast<const float4*>(Alo + src);
    *reinterpret_cast<float4*>(y + 4) = *reinterpret_cast<const float4*>(Alo + src + 4);
    const int em = e[m];
    if (em > -126 && em < 126) {
      const float sc = __int_as_float((127 - em) << 23);   // 2^-e_m exactly
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        x[u] *= sc;
        y[u] *= sc;
      }
    } else {
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        x[u] = ldexpf(x[u], -em);
        y[u] = ldexpf(y[u], -em);
      }
    }
#pragma unroll
    for (int s = 0; s < OZ_S; ++s) {
      __half h[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        x[u] *= (float)(1 << OZ_BITS);
        y[u] *= (float)(1 << OZ_BITS);
        const float a = rintf(x[u]);
        x[u] -= a;                                           // exact
        const float t = x[u] + y[u], bb = t - x[u];          // (x, y) <- two-sum (exact pair)
        y[u] = (x[u] - (t - bb)) + (y[u] - bb);
        x[u] = t;
        h[u] = __float2half_rn(a);                           // |a| <= 32: exact
      }
      *reinterpret_cast<uint4*>(dst + (size_t)s * OZ_TILE) = *reinterpret_cast<uint4*>(h);
    }
  }
}

// Scale and slices of one column by a cluster of eight CTAs, the column's values
// in registers between the two: f_c with max_l |x_cl w_l| < 2^f_c, then the fixed-
// point number round(|v| 2^5S) <= 2^5S, v = x_cl w_l 2^-f_c, cut into S digits
// -16 .. 15 (the first 0 .. 32) from the low end in integers, signs applied after.
// (The digits by FP64 scale, round and subtract were bound by FP64 issue, and one
// CTA per column for the maximum left the chip idle: 20.6 + 16.5 us for 24 columns of
// 8191, this kernel 10.4.)  Columns past nrhs are zero; a value that is not finite
// makes its column NaN.
// Layout: group g of columns, K tile, then a swizzled tile of S P rows, row t P + c.
#define OZ_CL 8
__global__ void __cluster_dims__(OZ_CL, 1, 1) __launch_bounds__(256)
    k_oz_slice_x(int N, long long ld, int nrhs, int S, int P, const double* __restrict__ X,
                 long long xs, const double* __restrict__ wgt64, int* __restrict__ f,
                 unsigned char* __restrict__ XS) {
  constexpr int PAIRS = OZ_KMAX / (2 * 256 * OZ_CL);   // column pairs per thread
  __shared__ unsigned red[8], cmax;
  const int rank = blockIdx.x, tid = threadIdx.x;
  const int col = blockIdx.y, g = col / P, cc = col - g * P;
  const int nkt = (int)(ld / MM_KT);
  const bool real = col < nrhs;
  double v[PAIRS][2];
  unsigned mx = 0;   // largest high word of a finite |v|: 2^-20 of the value, like the rows' scale
#pragma unroll
  for (int p = 0; p < PAIRS; ++p)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int l = ((p * OZ_CL + rank) * 256 + tid) * 2 + h;
      v[p][h] = (real && l < N) ? X[(size_t)col * xs + l] * (wgt64 ? wgt64[l] : 1.0) : 0.0;
      const unsigned hw = (unsigned)__double2hiint(v[p][h]) & 0x7fffffffu;
      if (hw < 0x7ff00000u) mx = max(mx, hw);
    }
  mx = __reduce_max_sync(0xffffffffu, mx);
  if ((tid & 31) == 0) red[tid >> 5] = mx;
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < 8; ++w) mx = max(mx, red[w]);
    cmax = mx;
  }
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
  mx = 0;
#pragma unroll
  for (int q = 0; q < OZ_CL; ++q) {
    unsigned a, t;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(mm_sa(&cmax)), "r"(q));
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(t) : "r"(a) : "memory");
    mx = max(mx, t);
  }
  // every CTA has read the maxima before any leaves
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
  int fe = 0;   // every |v| < the double with the next high word <= 2^fe
  if (mx > 0) frexp(__hiloint2double((int)mx, -1), &fe);
  if (real && rank == 0 && tid == 0) f[col] = fe;
  const int sh = OZ_BITS * S - fe;
  const bool plain = sh > -1000 && sh < 1000;
  const double sc = plain ? ldexp(1.0, sh) : 0.0;
#pragma unroll
  for (int p = 0; p < PAIRS; ++p) {
    const int l = ((p * OZ_CL + rank) * 256 + tid) * 2;
    if (l >= ld) break;
    unsigned lo[2], hi[2];
    bool neg[2], bad[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const double s = plain ? v[p][h] * sc : ldexp(v[p][h], sh);
      const int hw = __double2hiint(v[p][h]);
      bad[h] = (hw & 0x7fffffff) >= 0x7ff00000;
      neg[h] = hw < 0;
      const unsigned long long V = bad[h] ? 0ull : (unsigned long long)__double2ll_rn(fabs(s));
      lo[h] = (unsigned)V & ((1u << 25) - 1u);   // the last five digits
      hi[h] = (unsigned)(V >> 25);               // and the others
    }
    unsigned char* dst = XS + ((size_t)g * nkt + l / MM_KT) * ((size_t)S * P * 128);
    const int ch = (l & 63) >> 3, at = (l & 7) * 2;
    for (int t = S - 1; t >= 0; --t) {
      __half d2[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        int d;
        if (t == 0) {                            // what is left, up to 32
          d = S > 5 ? (int)hi[h] : (int)(lo[h] + (hi[h] << OZ_BITS));
        } else if (S - 1 - t < 5) {
          d = (int)((lo[h] + 16u) & 31u) - 16;
          lo[h] = (lo[h] - (unsigned)d) >> OZ_BITS;
          if (S - 1 - t == 4) hi[h] += lo[h];    // the carry out of the fifth digit
        } else {
          d = (int)((hi[h] + 16u) & 31u) - 16;
          hi[h] = (hi[h] - (unsigned)d) >> OZ_BITS;
        }
        d2[h] = bad[h] ? __ushort_as_half(0x7fffu) : __int2half_rn(neg[h] ? -d : d);
      }
      *reinterpret_cast<__half2*>(dst + oz_swz(t * P + cc, ch) + at) = __halves2half2(d2[0], d2[1]);
    }
  }
}

// pieces of K tiles, cut evenly over all (row block, K tile) units: range q holds
// units [U q / NP, U (q + 1) / NP), U = nrb nkt; a range that crosses a row block
// is one piece in each.  oz_range_of(u) is the range that holds unit u.
__host__ __device__ __forceinline__ int oz_range_of(long long u, long long U, int NP) {
  return (int)(((u + 1) * NP - 1) / U);
}

struct OzTc {
  const unsigned char* A;   // unit, slice, tile
  const unsigned char* X;   // group, K tile, tile of S P rows
  float* Yp;                // [slot][S][nrhs][ld]
  long long ld;
  int nrb, nkt, S, P, R, nrhs, ng, NP, w, NA;
  int* err;
};

__device__ __forceinline__ bool oz_wait(unsigned long long* b, unsigned parity,
                                        volatile int* fail) {
  for (unsigned it = 0; it < MM_SPIN; ++it) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(mm_sa(b)), "r"(parity)
        : "memory");
    if (ok) return true;
    if (*fail) return false;
  }
  return false;
}
__device__ __forceinline__ void oz_bulk(void* dst, const void* src, int bytes,
                                        unsigned long long* bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mm_sa(bar)),
               "r"(bytes)
               : "memory");
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          mm_sa(dst)),
      "l"(src), "r"(bytes), "r"(mm_sa(bar))
      : "memory");
}
__device__ __forceinline__ void oz_commit(unsigned long long* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          mm_sa(bar))
      : "memory");
}

// The four K = 16 products of one 64-column tile pair; acc = 0: the first one starts
// the accumulators anew.
__device__ __forceinline__ void oz_mma4(unsigned td, uint64_t ad, uint64_t bd, uint32_t idesc,
                                        unsigned acc) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t.reg .b64 a, b;\n\t"
      "setp.ne.b32 p, %4, 0;\n\tsetp.eq.b32 q, %3, %3;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t"
      "add.s64 a, %1, 2;\n\tadd.s64 b, %2, 2;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, q;\n\t"
      "add.s64 a, %1, 4;\n\tadd.s64 b, %2, 4;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, q;\n\t"
      "add.s64 a, %1, 6;\n\tadd.s64 b, %2, 6;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, q;\n\t}" ::"r"(td),
      "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
      : "memory");
}

// Persistent: CTA b works on ranges [w i, w i + w), i = b / ng, of column group
// b % ng (the CTAs of one range read the same tiles of A together, from L2 after
// the first).  Warp 4 copies (a ring of NA tiles of A and two of x), warp 5
// issues the products, warps 0-3 take finished pieces out of tensor memory while
// the copies for the next piece run.  Bound by reading the slices of A from HBM.
// Every wait is bounded; after one runs out, *err is set, the copies and products
// in flight are waited for, the tensor memory is freed and the CTA returns.
__global__ void __launch_bounds__(192, 1) k_oz_mma(const OzTc a) {
  extern __shared__ __align__(1024) unsigned char oz_raw[];
  unsigned char* sm = (unsigned char*)(((uintptr_t)oz_raw + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) unsigned long long afull[OZ_STAGES], aempty[OZ_STAGES],
      xfull[OZ_XSTAGES], xempty[OZ_XSTAGES], done, tfree, drain;
  __shared__ unsigned tslot;
  __shared__ volatile int fail;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int cols = a.S * a.P;               // <= 512
  const int xbytes = cols * 128;
  const int tcols = cols <= 32 ? 32 : cols <= 64 ? 64 : cols <= 128 ? 128 : cols <= 256 ? 256 : 512;
  unsigned char* const ring_a = sm + (size_t)OZ_XSTAGES * xbytes;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     mm_sa(&tslot)),
                 "r"(tcols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 32) {
    auto init = [](unsigned long long* b, unsigned n) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mm_sa(b)), "r"(n) : "memory");
    };
    for (int s = 0; s < OZ_STAGES; ++s) {
      init(&afull[s], 1);
      init(&aempty[s], 1);
    }
    for (int s = 0; s < OZ_XSTAGES; ++s) {
      init(&xfull[s], 1);
      init(&xempty[s], 1);
    }
    init(&done, 1);
    init(&tfree, 128);
    init(&drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fail = 0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned tmem = tslot;
  const int g = (int)blockIdx.x % a.ng, i0 = (int)blockIdx.x / a.ng;
  const long long U = (long long)a.nrb * a.nkt;
  const int q0 = i0 * a.w, q1 = min(a.NP, q0 + a.w);
  const long long ub = U * q0 / a.NP, ue = U * q1 / a.NP;   // this CTA's units
  auto give_up = [&]() {
    fail = 1;
    atomicExch(a.err, 1);
  };
  if (warp == 4 && lane == 0) {   // copies: unit by unit, no matter where pieces end
    int na = 0, nx = 0;           // tiles issued
    int as = 0;                   // next A stage and the parity of its last release
    unsigned aph = 1u;
    int kt = (int)(ub % a.nkt);
    bool ok = true;
    for (long long u = ub; u < ue && ok; ++u, kt = kt + 1 == a.nkt ? 0 : kt + 1) {
      const int xs = nx % OZ_XSTAGES;
      if (nx >= OZ_XSTAGES && !oz_wait(&xempty[xs], (unsigned)(nx / OZ_XSTAGES - 1) & 1u, &fail)) {
        ok = false;
        break;
      }
      oz_bulk(sm + (size_t)xs * xbytes, a.X + ((size_t)g * a.nkt + kt) * xbytes, xbytes,
              &xfull[xs]);
      ++nx;
      const unsigned char* src = a.A + (size_t)u * ((size_t)OZ_S * OZ_TILE);
      for (int s = 0; s < a.S; ++s) {
        if (na >= a.NA && !oz_wait(&aempty[as], aph, &fail)) {
          ok = false;
          break;
        }
        oz_bulk(ring_a + (size_t)as * OZ_TILE, src + (size_t)s * OZ_TILE, OZ_TILE, &afull[as]);
        ++na;
        if (++as == a.NA) {
          as = 0;
          aph ^= 1u;   // 0 for the second round
        }
      }
    }
    if (!ok) give_up();
    // no copy is in flight when the CTA returns
    for (int k = max(0, na - a.NA); k < na; ++k) mm_wait(&afull[k % a.NA], (unsigned)(k / a.NA) & 1u);
    for (int k = max(0, nx - OZ_XSTAGES); k < nx; ++k)
      mm_wait(&xfull[k % OZ_XSTAGES], (unsigned)(k / OZ_XSTAGES) & 1u);
  } else if (warp == 5 && lane == 0) {   // products
    // The loop over tiles carries no division and forms its descriptors by adding
    // to their low words: with both computed anew per tile the issuing thread, not
    // the tensor cores or HBM, set the pace (8191 unknowns, 24 columns: 315 us, now 220).
    int nx = 0, np = 0, as = 0;
    unsigned aph = 0u;   // parity of the current round of the ring
    bool ok = true;
    // FP32 accumulators, FP16 operands, both K-major, M = 128; N goes in below
    const uint32_t idesc0 = (1u << 4) | ((uint32_t)(128 >> 4) << 24);
    const uint64_t dbase = mm_desc_sw128(mm_sa(ring_a)), xbase = mm_desc_sw128(mm_sa(sm));
    uint64_t ad = dbase;
    for (int q = q0; q < q1 && ok; ++q) {
      const long long e1 = U * (q + 1) / a.NP;
      for (long long u = U * q / a.NP; u < e1 && ok;) {
        const long long rb = u / a.nkt, pe = min(e1, (rb + 1) * a.nkt);   // one piece
        if (np > 0 && !oz_wait(&tfree, (unsigned)(np - 1) & 1u, &fail)) ok = false;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        for (bool first = true; u < pe && ok; ++u) {
          const int xs = nx % OZ_XSTAGES;
          if (!oz_wait(&xfull[xs], (unsigned)(nx / OZ_XSTAGES) & 1u, &fail)) {
            ok = false;
            break;
          }
          const uint64_t xd = xbase + (uint64_t)((unsigned)(xs * xbytes) >> 4);
          unsigned td = tmem, fresh = first ? 0u : 1u;
          for (int nc = cols; nc > 0; nc -= a.P, td += a.P) {   // slice s: levels s .. S-1
            if (!oz_wait(&afull[as], aph, &fail)) {
              ok = false;
              break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            oz_mma4(td, ad, xd, idesc0 | ((uint32_t)(min(nc, 256) >> 3) << 17), fresh);
            if (nc > 256)
              oz_mma4(td + 256u, ad, xd + (256u * 128u >> 4),
                      idesc0 | ((uint32_t)((nc - 256) >> 3) << 17), fresh);
            fresh = 1u;
            oz_commit(&aempty[as]);
            ad += OZ_TILE >> 4;
            if (++as == a.NA) {
              as = 0;
              aph ^= 1u;
              ad = dbase;
            }
          }
          if (!ok) break;
          oz_commit(&xempty[xs]);
          ++nx;
          first = false;
        }
        if (ok) oz_commit(&done);
        ++np;
      }
    }
    if (!ok) give_up();
    oz_commit(&drain);   // every product has finished before the tensor memory goes
    mm_wait(&drain, 0u);
  } else if (warp < 4) {   // finished pieces
    int np = 0;
    bool ok = true;
    for (int q = q0; q < q1 && ok; ++q) {
      const long long e1 = U * (q + 1) / a.NP;
      for (long long u = U * q / a.NP; u < e1 && ok;) {
        const long long rb = u / a.nkt;
        u = min(e1, (rb + 1) * a.nkt);
        ok = __all_sync(0xffffffffu, oz_wait(&done, (unsigned)np & 1u, &fail)) != 0;
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int slot = q - oz_range_of(rb * a.nkt, U, a.NP);
        const int row = (int)rb * 128 + warp * 32 + lane;
        const unsigned ta = tmem + ((unsigned)(warp * 32) << 16);
        for (int L = 0; L < a.S; ++L) {
          const size_t at = ((size_t)slot * a.S + L) * a.nrhs;
          for (int c = 0; c < a.P && g * a.P + c < a.nrhs; c += 16) {
            uint32_t v[16];
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,"
                "%12,%13,%14,%15}, [%16];"
                : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]),
                  "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]),
                  "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
                : "r"(ta + (unsigned)(L * a.P + c))
                : "memory");
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (row < a.R) {
#pragma unroll
              for (int j = 0; j < 16; ++j)
                if (g * a.P + c + j < a.nrhs)
                  a.Yp[(at + g * a.P + c + j) * a.ld + row] = __uint_as_float(v[j]);
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mm_sa(&tfree)) : "memory");
        ++np;
      }
    }
    if (!ok) give_up();
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tcols)
                 : "memory");
}

// Y[c ys + m] = 2^(e_m + f_c) sum_L 2^-5(L+2) I_L (+ sgn_m x_cm), the pieces of a
// level added as integers (|I_L| <= 16384 x 3072 < 2^31) and the levels smallest
// first; a partial result that is no exact integer (NaN) makes the value NaN.
// One CTA per row block and column, two rows per thread (8-byte loads): bound by the
// loads' latency, 9.6 us for 24 columns of 8191 (one row per thread with the piece
// range found by every thread: 20.5).
__global__ void __launch_bounds__(64)
    k_oz_combine(OzTc a, const int* __restrict__ e, const int* __restrict__ f,
                 const double* __restrict__ X, long long xs, const float* __restrict__ sgn,
                 double* __restrict__ Y, long long ys) {
  const int m0 = blockIdx.x * 128 + threadIdx.x * 2, c = blockIdx.y;
  if (m0 >= a.R) return;
  const long long U = (long long)a.nrb * a.nkt, u0 = (long long)blockIdx.x * a.nkt;
  const int ns = oz_range_of(u0 + a.nkt - 1, U, a.NP) - oz_range_of(u0, U, a.NP) + 1;
  int I[2][OZ_S];
  bool bad[2] = {false, false};
#pragma unroll
  for (int L = 0; L < OZ_S; ++L) I[0][L] = I[1][L] = 0;
  for (int k = 0; k < ns; ++k) {
    const float* p = a.Yp + ((size_t)k * a.S * a.nrhs + c) * a.ld + m0;   // m0 < ld: both rows exist
#pragma unroll
    for (int L = 0; L < OZ_S; ++L)
      if (L < a.S) {
        const float2 t = *reinterpret_cast<const float2*>(p + (size_t)L * a.nrhs * a.ld);
        bad[0] = bad[0] || !(fabsf(t.x) <= 16777216.f);
        bad[1] = bad[1] || !(fabsf(t.y) <= 16777216.f);
        I[0][L] += (int)t.x;
        I[1][L] += (int)t.y;
      }
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int m = m0 + h;
    if (m >= a.R) break;
    // five levels at a time as one exact integer (< 2^47): FP64 issue bounded a
    // conversion and a product per level
    long long hi = 0, lo = 0;
#pragma unroll
    for (int L = 0; L < 5; ++L) {
      hi = (hi << OZ_BITS) + I[h][L];
      lo = (lo << OZ_BITS) + I[h][L + 5];
    }
    double y = fma((double)lo, 0x1p-25, (double)hi);
    y = bad[h] ? __longlong_as_double(0x7ff8000000000000ll) : ldexp(y, e[m] + f[c] - 6 * OZ_BITS);
    if (sgn) y += (double)sgn[m] * X[(size_t)c * xs + m];
    Y[(size_t)c * ys + m] = y;
  }
}

// which = 0: the matrix A (N rows, "A_hi"/"A_lo"); which = 1: the surface
// U-matrix (M_0 rows, "V_hi"/"V_lo").  Slices are built once per assembly.
struct OzMat {
  const char *hi, *lo, *slices, *exps;
  int rows;
};
static OzMat oz_mat(const bie_ctx* c, int which) {
  return which == 0 ? OzMat{"A_hi", "A_lo", "oz_A", "oz_e", c->N}
                    : OzMat{"V_hi", "V_lo", "oz_V", "oz_ev", c->M[0]};
}

static bie_status oz_prepare(bie_ctx* c, const OzMat& mt, int& held, int nsm, unsigned char** S,
                             int** e) {
  const long long ld = c->ld;
  const int nrb = (mt.rows + 127) / 128;
  BIE_GET(c, int, mt.exps, mt.rows, *e);
  BIE_GET(c, unsigned char, mt.slices, (size_t)OZ_S * 256 * nrb * ld, *S);
  if (held == c->asm_count) return BIE_OK;
  bool oom = false;
  const float* Ahi = (const float*)ctx_buf(c, mt.hi, sizeof(float) * (size_t)mt.rows * ld, &oom);
  const float* Alo = (const float*)ctx_buf(c, mt.lo, sizeof(float) * (size_t)mt.rows * ld, &oom);
  if (oom) return ctx_fail(c, BIE_ERR_OOM, "exact product: storage");
  k_oz_rowexp<<<(unsigned)((32LL * mt.rows + 255) / 256), 256, 0, c->stream>>>(mt.rows, ld, Ahi, *e);
  BIE_LAUNCH_CHECK(c, "k_oz_rowexp");
  k_oz_slice_A<<<8 * nsm, 256, 0, c->stream>>>(mt.rows, nrb, ld, Ahi, Alo, *e, *S);
  BIE_LAUNCH_CHECK(c, "k_oz_slice_A");
  held = c->asm_count;
  return BIE_OK;
}

bie_status oz_product(bie_ctx* c, int which, int nrhs, const double* X, long long xs, int apply_w,
                      int S, double* Y, long long ys, const float* sgn, int* err) {
  const long long ld = c->ld;
  if (ld > OZ_KMAX)
    return ctx_fail(c, BIE_ERR_ARG, "exact product: more than 16384 unknowns per row");
  const OzMat mt = oz_mat(c, which);
  int nsm = 0;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, c->device);
  unsigned char *SA, *XS;
  int *e, *f;
  bie_status st = oz_prepare(c, mt, which == 0 ? c->oz_count : c->ozv_count, nsm, &SA, &e);
  if (st != BIE_OK) return st;
  OzTc a;
  a.A = SA;
  a.ld = ld;
  a.R = mt.rows;
  a.nrb = (mt.rows + 127) / 128;
  a.nkt = (int)(ld / MM_KT);
  a.S = S;
  a.nrhs = nrhs;
  // one group of columns where its levels fit the 512 columns of tensor memory
  // (48 right-hand sides at S = 10), else two (at most 64 are accepted): 8191
  // unknowns, 48 columns 311 us, 64 columns 500
  a.P = (nrhs + 15) / 16 * 16;
  a.ng = 1;
  if (S * a.P > 512) {
    a.ng = 2;
    a.P = ((nrhs + 1) / 2 + 15) / 16 * 16;
  }
  // one CTA per SM, each as many ranges as keep a piece within OZ_PIECE tiles
  const long long U = (long long)a.nrb * a.nkt;
  const int G = (int)std::min<long long>(U, nsm / a.ng);
  a.w = (int)((U + (long long)G * (OZ_PIECE - 1) - 1) / ((long long)G * (OZ_PIECE - 1)));
  a.NP = G * a.w;
  int slots = 1;
  for (int rb = 0; rb < a.nrb; ++rb)
    slots = std::max(slots, oz_range_of((long long)(rb + 1) * a.nkt - 1, U, a.NP) -
                                oz_range_of((long long)rb * a.nkt, U, a.NP) + 1);
  const int xbytes = S * a.P * 128;
  a.NA = std::min(OZ_STAGES, (OZ_RING - OZ_XSTAGES * xbytes) / OZ_TILE);
  a.err = err;
  BIE_GET(c, int, "oz_f", nrhs, f);
  BIE_GET(c, unsigned char, "oz_X", (size_t)a.ng * a.nkt * xbytes, XS);
  BIE_GET(c, float, "oz_P", (size_t)slots * S * nrhs * ld, a.Yp);
  a.X = XS;
  const double* w = nullptr;
  if (apply_w) {
    bool oom = false;
    w = (const double*)ctx_buf(c, "wgt64", sizeof(double) * ld, &oom);
    if (oom) return ctx_fail(c, BIE_ERR_OOM, "exact product: weights");
  }
  k_oz_slice_x<<<dim3(OZ_CL, a.ng * a.P), 256, 0, c->stream>>>(c->N, ld, nrhs, S, a.P, X, xs, w, f,
                                                               XS);
  BIE_LAUNCH_CHECK(c, "k_oz_slice_x");
  const size_t smem = (size_t)a.NA * OZ_TILE + (size_t)OZ_XSTAGES * xbytes + 1024;
  BIE_CUDA_TRY(c, raise_smem_limit((const void*)k_oz_mma, smem));
  k_oz_mma<<<G * a.ng, 192, smem, c->stream>>>(a);
  BIE_LAUNCH_CHECK(c, "k_oz_mma");
  k_oz_combine<<<dim3(a.nrb, nrhs), 64, 0, c->stream>>>(a, e, f, X, xs, sgn, Y, ys);
  BIE_LAUNCH_CHECK(c, "k_oz_combine");
  return BIE_OK;
}

// Y[r][m] = sum_l A_ml X_rl / M_l + s_m X_rm with the full-accuracy storage
extern "C" bie_status bie_matmat_full(bie_ctx* c, int nrhs, const double* X_dev, double* Y_dev) {
  if (!c) return BIE_ERR_ARG;
  if (c && c->part_n > 1)
    return ctx_fail(c, BIE_ERR_STATE, "bie_matmat_full: not available on a row-partitioned context");
  BIE_NVTX("bie_matmat_full");
  if (!c->assembled) return ctx_fail(c, BIE_ERR_STATE, "bie_matmat_full: not assembled");
  if (c->transposed)
    return ctx_fail(c, BIE_ERR_STATE, "bie_matmat_full: storage holds the adjoint operator; assemble again");
  if (c->precision == BIE_FP64)
    return ctx_fail(c, BIE_ERR_STATE, "bie_matmat_full: needs the hi + lo storage of a refined scheme");
  if (c->ld > OZ_KMAX)
    return ctx_fail(c, BIE_ERR_ARG, "bie_matmat_full: at most 16384 unknowns");
  if (nrhs < 1 || nrhs > 64) return ctx_fail(c, BIE_ERR_ARG, "bie_matmat_full: 1 <= nrhs <= 64");
  if (!X_dev || !Y_dev) return ctx_fail(c, BIE_ERR_ARG, "bie_matmat_full: null pointer");
  cudaSetDevice(c->device);
  int* err;
  BIE_GET(c, int, "oz_err", 1, err);
  bool oom = false;
  const float* sgn = (const float*)ctx_buf(c, "sgn", sizeof(float) * c->ld, &oom);
  if (oom) return ctx_fail(c, BIE_ERR_OOM, "bie_matmat_full: node buffers");
  BIE_CUDA_TRY(c, cudaMemsetAsync(err, 0, sizeof(int), c->stream));
  bie_status s = oz_product(c, 0, nrhs, X_dev, c->N, 1, OZ_S, Y_dev, c->N, sgn, err);
  if (s != BIE_OK) return s;
  int herr = 0;
  BIE_CUDA_TRY(c, cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  BIE_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  if (herr) return ctx_fail(c, BIE_ERR_TIMEOUT, "exact product: a pipeline wait timed out");
  return BIE_OK;
}
