// Krylov drivers on pJDS matrices in the permuted basis (include/pjds_krylov.h):
// mixed-precision CG with fp64 residual refinement, Lanczos, fp64 Ritz refine.
//
// Small systems of pjds_cg_solve run in one launch (cg.cu). Everything else runs
// in the kernels below; the host only sequences launches, reads one residual norm
// per outer CG step and solves the small tridiagonal eigenproblem. Scalars (alpha,
// beta, norms) live in device memory and are read by the kernels that need them,
// so a run of inner iterations has no host round trip. Its launches follow one
// another by programmatic dependent launch; no graph is recorded (a step takes
// longer than its five launches, and a graph of 24 Lanczos steps took 0.3 ms to
// record). Inner products accumulate in fp64 or, for vectors of floats, in three
// floats that are as good: per-CTA partial sums into the workspace, which a launch of
// one CTA adds before it applies the scalar update. The sums depend on the number of
// CTAs alone, so results are bitwise reproducible.
#include <float.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "cg.h"
#include "common.h"
#include "gridsum.cuh"
#include "pjds_krylov.h"
#include "spmv_kernels.cuh"

namespace pjds {
namespace kry {

constexpr int KT = 256;  // threads per CTA of the vector and product kernels

// slots of the device scalar block
// (S_LALPHA, S_LBETA + (j & 1): the Lanczos coefficients of step j; beside
// them and 1 / beta their upper and lower halves as floats, SF_*)
enum { S_RR = 0, S_ALPHA, S_BETA, S_NRM, S_INVNRM, S_AUX0, S_AUX1, S_AUX2, S_LALPHA, S_LBETA, SF_ALPHA = 11, SF_BETA,
       SF_INV = 14, S_COUNT = 16 };
// finalisation operations
enum { F_ALPHA = 0, F_BETA, F_RR, F_NORM, F_LALPHA, F_LBETA, F_STORE };

// Whether fp32 holds a product p and its rounding error, and sums of some of them.
__device__ __forceinline__ bool in_range(float p) { return fabsf(p) >= 0x1p-96f && fabsf(p) <= 0x1p100f; }

// a + b as its rounded sum, and what the rounding left out added to err (Knuth, "The Art of Computer
// Programming", vol. 2, 4.2.2; exact whatever the operands' sizes).
__device__ __forceinline__ float two_sum(float a, float b, float &err) {
  const float t = __fadd_rn(a, b), z = __fsub_rn(t, a);
  err = __fadd_rn(__fsub_rn(a, __fsub_rn(t, z)), __fsub_rn(b, z));
  return t;
}

// Running inner product of one thread. Vectors of floats: products and sums in
// three times the working precision (Ogita, Rump, Oishi, "Accurate sum and dot
// product", 2005, DotK with K = 3: error-free products and sums in fp32, their
// errors added up the same way, and the errors of that beside), as an fp64
// multiply-add and its conversions take 16 cycles of the SM's fp64 pipe a warp:
// with them the two inner products of a CG step on 2M rows alone take 20 us. A
// thread adds at most KEEP products (launch_dot). What is lost is the rounding of
// the last part: of the sum P of KEEP products' magnitudes, the second part's 2 KEEP
// terms are at most 2^-24 P each, their errors 2 KEEP 2^-48 P each, and the 4 KEEP
// roundings in the sum of those below 16 KEEP^3 2^-72 P = 2^-53 P, against KEEP 2^-53
// P for multiply-adds in fp64. A thread with a product outside that range takes all
// of its products again, in fp64, after its loop (again(); with fp64 products inside
// the loop the product kernel took 3 us longer).
constexpr int KEEP = 32;
template <typename TX>
struct Dot;
template <>
struct Dot<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double a, double b) { s = __fma_rn(a, b, s); }
  template <typename F>
  __device__ __forceinline__ Fixed warp(F) const {
    const Fixed a[1] = {fixed_of(s)};
    return warp_sum<1>(a);
  }
};
template <>
struct Dot<float> {
  float s = 0.0f, c = 0.0f, l = 0.0f;
  bool far = false;  // a product too small or too large (or a NaN, as 0 times an infinity)
  __device__ __forceinline__ void add(float a, float b) {
    const float p = __fmul_rn(a, b);
    far = far || !(in_range(p) || (p == 0.0f && (a == 0.0f || b == 0.0f)));
    float q, r, t;
    s = two_sum(s, p, q);
    c = two_sum(c, q, r);
    c = two_sum(c, __fmaf_rn(a, b, -p), t);
    l = __fadd_rn(l, __fadd_rn(r, t));
  }
  template <typename F>
  __device__ __forceinline__ Fixed warp(F again) const {
    Fixed a[3] = {fixed_of(s), fixed_of(c), fixed_of(l)};
    if (far) a[0] = fixed_of(again()), a[1] = a[2] = Fixed{0, 1};
    return warp_sum<3>(a);
  }
};

// sum of a_i b_i in fp64 over the elements i0 + q stride + r below n, q from 0 to most - 1, r from 0 to width - 1
__device__ __forceinline__ double products(const float *a, const float *b, int64_t i0, int64_t stride, int width, int most,
                                           int64_t n) {
  double d = 0.0;
#pragma unroll 1
  for (; i0 < n && most > 0; i0 += stride, --most)
#pragma unroll 1
    for (int64_t i = i0; i < min(i0 + width, n); ++i) d = __fma_rn((double)a[i], (double)b[i], d);
  return d;
}
__device__ __forceinline__ double products(const double *, const double *, int64_t, int64_t, int, int, int64_t) {
  return 0.0;  // (Dot<double> does not ask)
}

// Where a reduction's result goes: the scalar block and the update.
struct Fin {
  double *scal;
  double *out;
  int32_t op, j;
};

// Programmatic dependent launch: every kernel lets the next one on the stream
// start (so that its launch is over when this one ends), and that one waits for
// this one, completed and visible, before it touches memory. A load through the
// read-only path may be moved ahead of that wait, so no pointer in those kernels
// is __restrict__. The products, which gather through it, are launched after the
// kernel before them has ended.
__device__ __forceinline__ void begin() {
  dev::let_next_start();
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// v as the sum of two floats (in the place of a double).
__device__ __forceinline__ void halves(double *out, double v) {
  const float h = (float)v;
  *reinterpret_cast<float2 *>(out) = make_float2(h, (float)(v - (double)h));
}

// The scalar update `op` with the complete sum v.
__device__ __forceinline__ void apply_op(double v, const Fin &f) {
  double *scal = f.scal;
  switch (f.op) {
    case F_ALPHA:  // alpha = (r, r) / (p, A p)
      scal[S_ALPHA] = v != 0.0 ? scal[S_RR] / v : 0.0;
      break;
    case F_BETA:  // beta = (r', r') / (r, r)
      scal[S_BETA] = scal[S_RR] != 0.0 ? v / scal[S_RR] : 0.0;
      scal[S_RR] = v;
      break;
    case F_RR:
      scal[S_RR] = v;
      break;
    case F_NORM: {
      const double nrm = sqrt(v);
      scal[S_NRM] = nrm;
      scal[S_INVNRM] = nrm > 0.0 ? 1.0 / nrm : 0.0;
      break;
    }
    case F_LALPHA:
      f.out[f.j] = v;
      scal[S_LALPHA] = v;
      halves(scal + SF_ALPHA, v);
      break;
    case F_LBETA: {
      const double nrm = sqrt(v), inv = nrm > 0.0 ? 1.0 / nrm : 0.0;
      f.out[f.j] = nrm;
      scal[S_LBETA + (f.j & 1)] = nrm;
      halves(scal + SF_BETA + (f.j & 1), nrm);
      scal[S_INVNRM] = inv;
      halves(scal + SF_INV, inv);
      break;
    }
    default:  // F_STORE
      scal[f.j] = v;
      break;
  }
}

// End of a kernel with a reduction: the CTA's sum goes to its slot, and
// reduce_kernel, the next launch, adds the slots. With an arrival counter, and so
// a gpu-scope fence, in every CTA the product on 2M rows took 123 us in place of
// 112 (a fence holds up the SM's other CTAs).
template <typename TX, typename F>
__device__ __forceinline__ void store_partial(const Dot<TX> &dot, double *partial, F again) {
  __shared__ Fixed sh[KT / 32];
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  const Fixed s = dot.warp(again);
  if (l == 0) sh[w] = s;
  __syncthreads();
  if (w != 0) return;
  const Fixed b[1] = {l < KT / 32 ? sh[l] : Fixed{0, 1}};
  const double t = double_of(warp_sum<1>(b));
  if (l == 0) partial[blockIdx.x] = t;
}

constexpr int RT = 1024;  // threads of reduce_kernel

// Adds n partial sums (one or two a thread after a product) and applies the
// scalar update. One CTA.
__global__ void __launch_bounds__(RT) reduce_kernel(const double *partial, int32_t n, Fin f) {
  __shared__ Fixed sh[RT / 32];
  begin();
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  double v = 0.0;
  for (int32_t k = threadIdx.x; k < n; k += RT) v += __ldcg(partial + k);
  const Fixed one[1] = {fixed_of(v)};
  const Fixed t = warp_sum<1>(one);
  if (l == 0) sh[w] = t;
  __syncthreads();
  if (w != 0) return;
  const Fixed a[1] = {l < RT / 32 ? sh[l] : Fixed{0, 1}};
  v = double_of(warp_sum<1>(a));
  if (l == 0) apply_op(v, f);
}

// One sorted row's product in the permuted basis (Listing 2 with the loop
// bound of the row's block; pads carry column -1 and are skipped).
template <typename TV, typename TX, typename IDX>
__device__ __forceinline__ typename dev::Acc<TV>::T row_product(const TV *__restrict__ val,
                                                                 const int32_t *__restrict__ col,
                                                                 const int64_t *__restrict__ col_start, int32_t L,
                                                                 int64_t i, const TX *__restrict__ x) {
  using TA = typename dev::Acc<TV>::T;
  constexpr int U = 4;
  TA acc = TA(0);
  for (int32_t j = 0; j < L; j += U) {
    int32_t c[U];
    TV v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (j + u < L) {
        const IDX o = (IDX)__ldg(col_start + j + u) + (IDX)i;
        c[u] = __ldcs(col + o);
        v[u] = dev::ld_stream1(val + o);
      } else {
        c[u] = -1;
        v[u] = TV{};
      }
    }
    TX xv[U];
#pragma unroll
    for (int u = 0; u < U; ++u) xv[u] = dev::gather(x, c[u]);
#pragma unroll
    for (int u = 0; u < U; ++u) acc = c[u] >= 0 ? dev::fma_acc(dev::to_acc(v[u]), (TA)xv[u], acc) : acc;
  }
  return acc;
}

// Two adjacent sorted rows i, i+1 (i even, so both lie in one block): one
// paired load of col and of val per jagged diagonal, then each row's product
// exactly as row_product computes it.
template <typename TV, typename TX, typename IDX>
__device__ __forceinline__ void row_product2(const TV *__restrict__ val, const int32_t *__restrict__ col,
                                             const int64_t *__restrict__ col_start, int32_t L, int64_t i,
                                             const TX *__restrict__ x, typename dev::Acc<TV>::T (&acc)[2]) {
  using TA = typename dev::Acc<TV>::T;
  constexpr int U = 4;
  acc[0] = acc[1] = TA(0);
  for (int32_t j = 0; j < L; j += U) {
    int32_t c[U][2];
    TV v[U][2];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (j + u < L) {
        const IDX o = (IDX)__ldg(col_start + j + u) + (IDX)i;
        dev::ld_stream<2>(col + o, c[u]);
        dev::ld_stream<2>(val + o, v[u]);
      } else {
        c[u][0] = c[u][1] = -1;
        v[u][0] = v[u][1] = TV{};
      }
    }
    TX xv[U][2];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int r = 0; r < 2; ++r) xv[u][r] = dev::gather(x, c[u][r]);
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int r = 0; r < 2; ++r)
        acc[r] = c[u][r] >= 0 ? dev::fma_acc(dev::to_acc(v[u][r]), (TA)xv[u][r], acc[r]) : acc[r];
  }
}

// The product kernels run a grid of as many CTAs as fit on the GPU at once and
// stride over the rows: a CTA ends with a barrier and the sum, and with one row
// per thread those ends cost a tenth (200 steps of CG on 2M rows, CTAs per SM
// fp64 all / 32 / 16 / 8 29.9 / 28.4 / 27.6 / 27.4 ms, two rows per thread fp32
// all / 16 / 8 / 6 20.8 / 18.3 / 20.7 / 18.4; eight fit in fp64, six of two rows
// per thread).

// MODE 0: y = A x and the reduction of sum x_i y_i.  MODE 1: y = bv - A x and
// the reduction of sum y_i^2 (the fp64 residual of the refinement loop). The
// value array arrives untyped so that every instance for one vector type has
// the same signature.
template <typename TV, typename TX, typename IDX, int MODE>
__global__ void __launch_bounds__(KT)
    spmv_dot_kernel(const void *__restrict__ val_, const int32_t *__restrict__ col,
                    const int64_t *__restrict__ col_start, const int32_t *__restrict__ block_len,
                    const TX *__restrict__ x, TX *__restrict__ y, const TX *__restrict__ bv,
                    double *__restrict__ partial, int32_t n_rows, int32_t b) {
  dev::let_next_start();
  const TV *__restrict__ val = static_cast<const TV *>(val_);
  Dot<TX> dot;
  // rows in sorted order: the tile traversal table measured 1.7% slower here
  // (fp64 CG on the 27-point stencil, 4.5M rows)
  for (int64_t i = (int64_t)blockIdx.x * KT + threadIdx.x; i < n_rows; i += (int64_t)gridDim.x * KT) {
    const int32_t L = __ldg(block_len + (uint32_t)i / (uint32_t)b);
    const auto acc = row_product<TV, TX, IDX>(val, col, col_start, L, i, x);
    TX yi;
    if constexpr (MODE == 0) {
      yi = (TX)acc;
      dot.add(x[i], yi);
    } else {
      yi = (TX)((double)bv[i] - (double)acc);
      dot.add(yi, yi);
    }
    y[i] = yi;
  }
  store_partial(dot, partial, [&] {
    return products(MODE == 0 ? x : y, y, (int64_t)blockIdx.x * KT + threadIdx.x, (int64_t)gridDim.x * KT, 1, KEEP, n_rows);
  });
}

// y = A x and the reduction of sum x_i y_i with two adjacent rows per thread
// (row pair p: rows 2p, 2p+1; the second is a padding row when n_rows is odd).
// Six CTAs on an SM, 40 registers: five, 48, are up to 4% faster on half a million
// to a million rows and up to 4% slower from 1.3M on.
template <typename TV, typename TX, typename IDX>
__global__ void __launch_bounds__(KT, 6)
    spmv_dot2_kernel(const void *__restrict__ val_, const int32_t *__restrict__ col,
                     const int64_t *__restrict__ col_start, const int32_t *__restrict__ block_len,
                     const TX *__restrict__ x, TX *__restrict__ y, const TX *__restrict__ bv,
                     double *__restrict__ partial, int32_t n_rows, int32_t b) {
  dev::let_next_start();
  const TV *__restrict__ val = static_cast<const TV *>(val_);
  Dot<TX> dot;
  for (int64_t i = 2 * ((int64_t)blockIdx.x * KT + threadIdx.x); i < n_rows; i += 2 * (int64_t)gridDim.x * KT) {
    const int32_t L = __ldg(block_len + (uint32_t)i / (uint32_t)b);
    typename dev::Acc<TV>::T acc[2];
    row_product2<TV, TX, IDX>(val, col, col_start, L, i, x, acc);
#pragma unroll
    for (int r = 0; r < 2; ++r)
      if (i + r < n_rows) {
        const TX yi = (TX)acc[r];
        dot.add(x[i + r], yi);
        y[i + r] = yi;
      }
  }
  store_partial(dot, partial, [&] {
    return products(x, y, 2 * ((int64_t)blockIdx.x * KT + threadIdx.x), 2 * (int64_t)gridDim.x * KT, 2, KEEP, n_rows);
  });
}

// 16-byte groups of workspace vectors (the workspace is 256-byte aligned):
// W elements per load and store.
template <typename TX>
struct G16 {
  static constexpr int W = 16 / (int)sizeof(TX);
  __device__ static void load(const TX *p, TX (&v)[W]) {
    const uint4 u = *reinterpret_cast<const uint4 *>(p);
    memcpy(v, &u, 16);
  }
  __device__ static void store(TX *p, const TX (&v)[W]) {
    uint4 u;
    memcpy(&u, v, 16);
    *reinterpret_cast<uint4 *>(p) = u;
  }
};

// VG consecutive blocks of KT 16-byte groups of n elements per CTA, one group of
// each per thread; the elements past the last group go one per thread of CTA 0.
// load(q, first element) for all of a thread's groups, then use(q, first
// element); tail(element).
constexpr int VG = 2;
template <typename TX, typename FL, typename FU, typename FT>
__device__ __forceinline__ void groups(int32_t n, FL load, FU use, FT tail) {
  constexpr int W = G16<TX>::W;
  const int64_t ng = n / W, k = (int64_t)blockIdx.x * (VG * KT) + threadIdx.x;
#pragma unroll
  for (int q = 0; q < VG; ++q)
    if (k + q * KT < ng) load(q, (k + q * KT) * W);
#pragma unroll
  for (int q = 0; q < VG; ++q)
    if (k + q * KT < ng) use(q, (k + q * KT) * W);
  if (blockIdx.x == 0 && threadIdx.x < n - ng * W) tail(ng * W + threadIdx.x);
}

// sum of v_e^2 over this thread's elements of groups()
template <typename TX>
__device__ __forceinline__ double squares(const TX *v, int32_t n) {
  constexpr int W = G16<TX>::W;
  const int64_t whole = n / W * W;
  double d = products(v, v, ((int64_t)blockIdx.x * (VG * KT) + threadIdx.x) * W, (int64_t)KT * W, W, VG, whole);
  if (blockIdx.x == 0) d += products(v, v, whole + threadIdx.x, 1, 1, 1, n);
  return d;
}

template <typename TX>
static int32_t group_grid(int32_t n) {
  const int64_t per = (int64_t)VG * KT * G16<TX>::W;
  return (int32_t)std::max<int64_t>(1, (n + per - 1) / per);
}

// r -= alpha q; reduces sum r_i^2.
template <typename TX>
__global__ void __launch_bounds__(KT)
    cg_update_kernel(TX *r, const TX *q, const double *scal,
                     double *partial, int32_t n) {
  begin();
  constexpr int W = G16<TX>::W;
  const TX a = (TX)scal[S_ALPHA];
  Dot<TX> dot;
  TX rv[VG][W], qv[VG][W];
  groups<TX>(
      n,
      [&](int g, int64_t e) {
        G16<TX>::load(r + e, rv[g]);
        G16<TX>::load(q + e, qv[g]);
      },
      [&](int g, int64_t e) {
#pragma unroll
        for (int w = 0; w < W; ++w) {
          rv[g][w] = rv[g][w] - a * qv[g][w];
          dot.add(rv[g][w], rv[g][w]);
        }
        G16<TX>::store(r + e, rv[g]);
      },
      [&](int64_t i) {
        const TX ri = r[i] - a * q[i];
        r[i] = ri;
        dot.add(ri, ri);
      });
  store_partial(dot, partial, [&] { return squares(r, n); });
}

// d += alpha p (here, where p is read anyway), p = r + beta p.
template <typename TX>
__global__ void __launch_bounds__(KT)
    cg_dir_kernel(TX *d, TX *p, const TX *r, const double *scal,
                  int32_t n) {
  begin();
  constexpr int W = G16<TX>::W;
  const TX a = (TX)scal[S_ALPHA], be = (TX)scal[S_BETA];
  TX dv[VG][W], pv[VG][W], rv[VG][W];
  groups<TX>(
      n,
      [&](int g, int64_t e) {
        G16<TX>::load(d + e, dv[g]);
        G16<TX>::load(p + e, pv[g]);
        G16<TX>::load(r + e, rv[g]);
      },
      [&](int g, int64_t e) {
#pragma unroll
        for (int w = 0; w < W; ++w) {
          dv[g][w] = dv[g][w] + a * pv[g][w];
          pv[g][w] = rv[g][w] + be * pv[g][w];
        }
        G16<TX>::store(d + e, dv[g]);
        G16<TX>::store(p + e, pv[g]);
      },
      [&](int64_t i) {
        d[i] = d[i] + a * p[i];
        p[i] = r[i] + be * p[i];
      });
}

// Start of an inner solve: r = p = (r64 / ||r64||) in the inner type, d = 0,
// reduces sum r_i^2.
template <typename TL>
__global__ void __launch_bounds__(KT)
    ir_start_kernel(const double *r64, TL *r, TL *p, TL *d,
                    const double *scal, double *partial, int32_t n) {
  begin();
  const double inv = scal[S_INVNRM];
  Dot<TL> dot;
  const int64_t i = (int64_t)blockIdx.x * KT + threadIdx.x;
  if (i < n) {
    const TL ri = (TL)(r64[i] * inv);
    r[i] = ri;
    p[i] = ri;
    d[i] = TL(0);
    dot.add(ri, ri);
  }
  store_partial(dot, partial, [&] { return products(r, r, i, 1, 1, 1, n); });
}

// x += ||r64|| d (fp64)
template <typename TL>
__global__ void __launch_bounds__(KT)
    ir_correct_kernel(double *x, const TL *d, const double *scal, int32_t n) {
  begin();
  const int64_t i = (int64_t)blockIdx.x * KT + threadIdx.x;
  if (i < n) x[i] = fma(scal[S_NRM], (double)d[i], x[i]);
}

template <typename TX>
__global__ void __launch_bounds__(KT) sumsq_kernel(const TX *v, double *partial, int32_t n) {
  begin();
  Dot<TX> dot;
  const int64_t i = (int64_t)blockIdx.x * KT + threadIdx.x;
  if (i < n) dot.add(v[i], v[i]);
  store_partial(dot, partial, [&] { return products(v, v, i, 1, 1, 1, n); });
}

// v = v0 / ||v0||
template <typename TX>
__global__ void __launch_bounds__(KT)
    lanczos_start_kernel(const TX *v0, TX *v, const double *scal, int32_t n) {
  begin();
  const int64_t i = (int64_t)blockIdx.x * KT + threadIdx.x;
  if (i < n) v[i] = (TX)((double)v0[i] * scal[S_INVNRM]);
}

// The fp64 arithmetic of the Lanczos vectors, for floats without the fp64 pipe
// (six conversions and multiply-adds an element took 20 us a step on 1M rows):
// error-free products and sums in fp32 give r, the result rounded once, and d, what
// that rounding left out, within a bound E that covers their own errors and those of
// the fp64 expression. Where r + d - E and r + d + E both round to r, so does the
// fp64 expression; else (a few elements in 2^16 and those outside the range where
// fp32 holds the products' errors) it is evaluated. So the vectors are those of the
// fp64 arithmetic, bit for bit.
// (not inlined, so that the fp64 operations are not speculated on every element)
__device__ __noinline__ float far_times(float w, double a) { return (float)((double)w * a); }
__device__ __noinline__ float far_orth(float w, double a, float v, double b, float p) {
  return (float)((double)w - a * (double)v - b * (double)p);
}
// whether every value within E of r + d rounds to r
__device__ __forceinline__ bool certain(float r, float d, float E) {
  return __fadd_rn(r, __fadd_rn(d, E)) == r && __fadd_rn(r, __fsub_rn(d, E)) == r;
}
template <typename TX>
struct Coef;
template <>
struct Coef<double> {
  double d;
  __device__ __forceinline__ Coef(const double *wide, const double *) : d(*wide) {}
  __device__ __forceinline__ double times(double w) const { return w * d; }
  // w - a v - b p
  __device__ __forceinline__ static double orth(double w, const Coef &a, double v, const Coef &b, double p) {
    return w - a.d * v - b.d * p;
  }
};
template <>
struct Coef<float> {
  const double *wide;
  float2 h;
  __device__ __forceinline__ Coef(const double *w, const double *two)
      : wide(w), h(*reinterpret_cast<const float2 *>(two)) {
    // a lower half that fp32 does not hold to 2^-48 of the whole: no product is then in range
    if (h.x != 0.0f && fabsf(h.x) < 0x1p-100f) h.x = __int_as_float(0x7fffffff);
  }
  // errors: fma(w, h.y, e) 2^-47 of p, the halves of the factor 2^-48, the sum in certain() 2^-48, the fp64
  // product 2^-53
  __device__ __forceinline__ float times(float w) const {
    const float p = __fmul_rn(w, h.x), c = __fmaf_rn(w, h.y, __fmaf_rn(w, h.x, -p)), r = __fadd_rn(p, c);
    if ((p == 0.0f && w == 0.0f) ||
        (in_range(p) && certain(r, __fadd_rn(__fsub_rn(p, r), c), 0x1p-45f * fabsf(p))))
      return r;
    return far_times(w, *wide);
  }
  // errors: ex 1.5 2^-47 of x, ey of y, et + eu 2^-47 of the sum M of the magnitudes, ex + ey 2^-47, their difference
  // 2^-46, the sum in certain() 2^-48, the fp64 expression 2^-52: below 2^-44.4 M
  __device__ __forceinline__ static float orth(float w, const Coef &a, float v, const Coef &b, float p) {
    const float x = __fmul_rn(a.h.x, v), y = __fmul_rn(b.h.x, p);
    const float ex = __fmaf_rn(a.h.y, v, __fmaf_rn(a.h.x, v, -x)), ey = __fmaf_rn(b.h.y, p, __fmaf_rn(b.h.x, p, -y));
    float et, eu, d;
    const float t = two_sum(w, -x, et), u = two_sum(t, -y, eu);
    const float r = two_sum(u, __fsub_rn(__fadd_rn(et, eu), __fadd_rn(ex, ey)), d);
    if (((x == 0.0f && v == 0.0f) || in_range(x)) && ((y == 0.0f && p == 0.0f) || in_range(y)) &&
        (w == 0.0f || in_range(w)) && certain(r, d, 0x1p-44f * (fabsf(w) + fabsf(x) + fabsf(y))))
      return r;
    return far_orth(w, *a.wide, v, *b.wide, p);
  }
};

// W elements at p, by one load if p allows it (a basis row is caller memory).
template <typename TX>
__device__ __forceinline__ void load_any(const TX *p, TX (&v)[G16<TX>::W]) {
  if (((uintptr_t)p & 15) == 0) {
    G16<TX>::load(p, v);
  } else {
#pragma unroll
    for (int e = 0; e < G16<TX>::W; ++e) v[e] = p[e];
  }
}

// w = w - alpha_j v - beta_j vprev (in fp64, stored in TX); reduces sum w_i^2.
// vprev: NULL for the first step.
template <typename TX>
__global__ void __launch_bounds__(KT)
    lanczos_orth_kernel(TX *w, const TX *v, const TX *vprev,
                        const double *scal, double *partial, int32_t j, int32_t n) {
  constexpr int W = G16<TX>::W;
  begin();
  const Coef<TX> a(scal + S_LALPHA, scal + SF_ALPHA), b(scal + S_LBETA + (j & 1), scal + SF_BETA + (j & 1));
  Dot<TX> dot;
  TX wv[VG][W], vv[VG][W], pv[VG][W];
  groups<TX>(
      n,
      [&](int g, int64_t e) {
        G16<TX>::load(w + e, wv[g]);
        load_any(v + e, vv[g]);
        if (vprev) {
          load_any(vprev + e, pv[g]);
        } else {
#pragma unroll
          for (int k = 0; k < W; ++k) pv[g][k] = TX(0);
        }
      },
      [&](int g, int64_t e) {
#pragma unroll
        for (int k = 0; k < W; ++k) {
          wv[g][k] = Coef<TX>::orth(wv[g][k], a, vv[g][k], b, pv[g][k]);
          dot.add(wv[g][k], wv[g][k]);
        }
        G16<TX>::store(w + e, wv[g]);
      },
      [&](int64_t i) {
        const TX x = Coef<TX>::orth(w[i], a, v[i], b, vprev ? vprev[i] : TX(0));
        w[i] = x;
        dot.add(x, x);
      });
  store_partial(dot, partial, [&] { return squares(w, n); });
}

// v = w / beta_{j+1}: the next vector, in its row of the basis if there is one.
template <typename TX>
__global__ void __launch_bounds__(KT)
    lanczos_next_kernel(TX *v, const TX *w, const double *scal, int32_t n) {
  constexpr int W = G16<TX>::W;
  begin();
  const Coef<TX> inv(scal + S_INVNRM, scal + SF_INV);
  const bool v16 = ((uintptr_t)v & 15) == 0;
  TX wv[VG][W];
  groups<TX>(
      n, [&](int g, int64_t e) { G16<TX>::load(w + e, wv[g]); },
      [&](int g, int64_t e) {
#pragma unroll
        for (int k = 0; k < W; ++k) wv[g][k] = inv.times(wv[g][k]);
        if (v16) {
          G16<TX>::store(v + e, wv[g]);
        } else {
#pragma unroll
          for (int k = 0; k < W; ++k) v[e + k] = wv[g][k];
        }
      },
      [&](int64_t i) { v[i] = inv.times(w[i]); });
}

// y = sum_j s_j basis[j] (fp64); reduces sum y_i^2
template <typename TB>
__global__ void __launch_bounds__(KT)
    ritz_combine_kernel(const TB *basis, const double *s, int32_t k, int32_t n,
                        double *y, double *partial) {
  begin();
  Dot<double> dot;
  const int64_t i = (int64_t)blockIdx.x * KT + threadIdx.x;
  if (i < n) {
    double acc = 0.0;
    for (int32_t j = 0; j < k; ++j) acc = fma(s[j], (double)__ldcs(basis + (int64_t)j * n + i), acc);
    y[i] = acc;
    dot.add(acc, acc);
  }
  store_partial(dot, partial, [] { return 0.0; });
}

// reduces sum (w_i - theta y_i)^2 with theta = scal[S_AUX1] / scal[S_AUX0]
__global__ void __launch_bounds__(KT)
    ritz_residual_kernel(const double *w, const double *y, const double *scal,
                         double *partial, int32_t n) {
  begin();
  const double theta = scal[S_AUX1] / scal[S_AUX0];
  Dot<double> dot;
  const int64_t i = (int64_t)blockIdx.x * KT + threadIdx.x;
  if (i < n) {
    const double e = w[i] - theta * y[i];
    dot.add(e, e);
  }
  store_partial(dot, partial, [] { return 0.0; });
}

// ----------------------------------------------------------------------------- host helpers

static inline size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }
static inline int32_t n_blocks_of(int32_t n) { return (int32_t)(((int64_t)n + KT - 1) / KT); }

struct Carve {
  char *base;
  size_t off, cap;
  template <typename T>
  T *take(size_t count) {
    T *p = reinterpret_cast<T *>(base + off);
    off += align256(count * sizeof(T));
    return p;
  }
};

static int launch_check(const char *what) {
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? PJDS_OK : set_error(PJDS_ECUDA, "%s: %s", what, cudaGetErrorString(e));
}

static int check_square_permuted(const pjds_dev *A, const char *name) {
  if (!A) return set_error(PJDS_EINVAL, "%s is NULL", name);
  if (value_bytes(A->dtype) == 0) return set_error(PJDS_EINVAL, "%s: unknown dtype", name);
  if (!A->permute_cols || A->n_rows != A->n_cols)
    return set_error(PJDS_EINVAL, "%s must be square and created with permute_cols = 1", name);
  if (A->b <= 0 || A->b % 32 || (int64_t)A->n_pad != ((int64_t)A->n_rows + A->b - 1) / A->b * A->b)
    return set_error(PJDS_EINVAL, "%s: inconsistent n_pad / b", name);
  if (A->n_stored > 0 && (!A->val || !A->col || !A->col_start || !A->block_len))
    return set_error(PJDS_EINVAL, "%s: a matrix array is NULL", name);
  return PJDS_OK;
}

// A product-and-reduce kernel chosen by value type and index width, the rows of
// a CTA and the CTAs resident on all SMs at once.
template <typename TX, int MODE>
struct DotKernel {
  void (*fn)(const void *, const int32_t *, const int64_t *, const int32_t *, const TX *, TX *, const TX *, double *,
             int32_t, int32_t);
  int32_t rows, resident;
};

template <typename TV, typename TX, int MODE>
static void dot_typed(const pjds_dev *A, DotKernel<TX, MODE> *d) {
  const bool wide = A->n_stored + A->n_pad >= 0x7fffffffLL;
  d->fn = wide ? spmv_dot_kernel<TV, TX, int64_t, MODE> : spmv_dot_kernel<TV, TX, int32_t, MODE>;
  d->rows = KT;
}

// fp32 / bf16 values: two rows per thread when val and col allow the paired
// loads (one 8- or 4-byte value load and one 8-byte column load per diagonal)
template <typename TV>
static void dot_float(const pjds_dev *A, DotKernel<float, 0> *d) {
  const bool pair = ((uintptr_t)A->val % (2 * value_bytes(A->dtype))) == 0 && ((uintptr_t)A->col % 8) == 0;
  if (!pair) return dot_typed<TV, float, 0>(A, d);
  const bool wide = A->n_stored + A->n_pad >= 0x7fffffffLL;
  d->fn = wide ? spmv_dot2_kernel<TV, float, int64_t> : spmv_dot2_kernel<TV, float, int32_t>;
  d->rows = 2 * KT;
}

template <typename TX, int MODE>
static int make_dot(const pjds_dev *A, DotKernel<TX, MODE> *d) {
  if constexpr (sizeof(TX) == 8)
    dot_typed<double, double, MODE>(A, d);
  else if (A->dtype == PJDS_BF16)
    dot_float<dev::bf16_t>(A, d);
  else
    dot_float<float>(A, d);
  int dev = 0, sms = 0, per_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, d->fn, KT, 0);
  if (e != cudaSuccess) return set_error(PJDS_ECUDA, "occupancy query: %s", cudaGetErrorString(e));
  if (sms < 1 || per_sm < 1) return set_error(PJDS_ECUDA, "kernel does not fit on an SM");
  d->resident = sms * per_sm;
  return PJDS_OK;
}

template <typename T>
struct Same {
  using type = T;
};

// What the reductions need in a workspace, before its vectors: partial sums and
// the scalar block.
struct Reduce {
  double *partial, *scal;
  static size_t bytes(int32_t n) { return align256((size_t)n_blocks_of(n) * 8) + align256(S_COUNT * 8); }
  static Reduce take(Carve &cv, int32_t n) {
    Reduce r;
    r.partial = cv.take<double>((size_t)n_blocks_of(n));
    r.scal = cv.take<double>(S_COUNT);
    return r;
  }
  int clear(cudaStream_t s) const {
    const cudaError_t e = cudaMemsetAsync(scal, 0, S_COUNT * 8, s);
    return e == cudaSuccess ? PJDS_OK : set_error(PJDS_ECUDA, "workspace: %s", cudaGetErrorString(e));
  }
  // add the n partial sums of the kernel before
  void sum(int64_t n, cudaStream_t s, int32_t op, int32_t j = 0, double *out = nullptr) const {
    dev::launch_early(reduce_kernel, 1, RT, s, partial, (int32_t)n, Fin{scal, out, op, j});
  }
};

// y = A x and the inner product into red (the vector type is taken from the
// kernel alone).
template <typename TX, int MODE>
static void launch_dot(const DotKernel<TX, MODE> &d, const pjds_dev *A, const typename Same<TX>::type *x,
                       typename Same<TX>::type *y, const typename Same<TX>::type *bv, const Reduce &red, cudaStream_t s,
                       int32_t op, int32_t j = 0, double *out = nullptr) {
  // no more CTAs than fit at once, but with floats no more rows of a thread than KEEP (from 7.5M rows on)
  const int64_t all = ((int64_t)A->n_rows + d.rows - 1) / d.rows;
  const int64_t least = sizeof(TX) == 4 ? (all * (d.rows / KT) + KEEP - 1) / KEEP : 1;
  const int64_t grid = std::min<int64_t>(all, std::max<int64_t>(d.resident, least));
  d.fn<<<(unsigned)grid, KT, 0, s>>>(A->val, A->col, A->col_start, A->block_len, x, y, bv, red.partial, A->n_rows, A->b);
  red.sum(grid, s, op, j, out);
}

// ----------------------------------------------------------------------------- CG

static size_t cg_bytes(int32_t n, int vec_bytes) {
  return Reduce::bytes(n) + 4 * align256((size_t)n * vec_bytes) + align256((size_t)n * 8) +
         align256(sizeof(CgOut)) + align256(cg_slots_bytes());
}

template <typename TL>
static int cg_run(const pjds_dev *Ah, const pjds_dev *Al, const double *b, double *x, const pjds_cg_opts &o,
                  pjds_cg_result *res, void *work, cudaStream_t s) {
  const int32_t n = Ah->n_rows, nb = n_blocks_of(n);
  Carve cv{static_cast<char *>(work), 0, 0};
  const Reduce red = Reduce::take(cv, n);
  double *const scal = red.scal;
  TL *r = cv.take<TL>((size_t)n), *p = cv.take<TL>((size_t)n), *q = cv.take<TL>((size_t)n);
  TL *d = cv.take<TL>((size_t)n);
  double *r64 = cv.take<double>((size_t)n);
  CgOut *small_out = cv.take<CgOut>(1);
  char *slots = cv.take<char>(cg_slots_bytes());
  pjds_cg_result small_res;
  bool small = false;
  const int rc_small = cg_small(
      Ah, Al, CgSystem{b, x, r64, r, p, q, slots, small_out, &small_res, o.max_outer, o.inner_iters, o.tol}, &small, s);
  if (rc_small) return rc_small;
  if (small) {
    if (res) *res = small_res;
    return PJDS_OK;
  }
  DotKernel<TL, 0> dot_lo;
  DotKernel<double, 1> dot_res;
  const int32_t g_vec = group_grid<TL>(n);
  int rc;
  if ((rc = make_dot(Al, &dot_lo)) || (rc = make_dot(Ah, &dot_res)) || (rc = red.clear(s))) return rc;
  // ||b||
  dev::launch_early(sumsq_kernel<double>, nb, KT, s, b, red.partial, n);
  red.sum(nb, s, F_STORE, S_AUX2);
  double bn2 = 0.0;
  if ((rc = launch_check("cg ||b||"))) return rc;
  cudaError_t e = cudaMemcpyAsync(&bn2, scal + S_AUX2, sizeof(double), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return set_error(PJDS_ECUDA, "cg: %s", cudaGetErrorString(e));
  const double bnorm = sqrt(bn2);

  pjds_cg_result out;
  memset(&out, 0, sizeof(out));
  double rel = 0.0;
  rc = PJDS_OK;
  for (int outer = 0;; ++outer) {
    launch_dot(dot_res, Ah, x, r64, b, red, s, F_NORM);  // r64 = b - A x, ||r64||
    if ((rc = launch_check("cg residual"))) break;
    double rn = 0.0;
    e = cudaMemcpyAsync(&rn, scal + S_NRM, sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
      rc = set_error(PJDS_ECUDA, "cg: %s", cudaGetErrorString(e));
      break;
    }
    rel = bnorm > 0.0 ? rn / bnorm : rn;
    if (out.n_history < PJDS_CG_HISTORY) out.history[out.n_history++] = rel;
    if (outer >= o.max_outer || rel <= o.tol || rn == 0.0) break;
    dev::launch_early(ir_start_kernel<TL>, nb, KT, s, r64, r, p, d, scal, red.partial, n);
    red.sum(nb, s, F_RR);
    for (int it = 0; it < o.inner_iters; ++it) {
      launch_dot(dot_lo, Al, p, q, nullptr, red, s, F_ALPHA);                   // q = A p, (p, q), alpha
      dev::launch_early(cg_update_kernel<TL>, g_vec, KT, s, r, q, scal, red.partial, n);  // r, (r, r), beta
      red.sum(g_vec, s, F_BETA);
      dev::launch_early(cg_dir_kernel<TL>, g_vec, KT, s, d, p, r, scal, n);  // d, p
    }
    dev::launch_early(ir_correct_kernel<TL>, nb, KT, s, x, d, scal, n);
    if ((rc = launch_check("cg inner"))) break;
    out.outer = outer + 1;
    out.inner_total += o.inner_iters;
  }
  out.rel_residual = rel;
  if (res) *res = out;
  return rc;
}

}  // namespace kry
}  // namespace pjds

using namespace pjds;
using namespace pjds::kry;

extern "C" int pjds_cg_workspace_bytes(int32_t n_rows, int32_t n_pad, int32_t vec_dtype, size_t *bytes) {
  clear_error();
  if (!bytes || n_rows < 0 || n_pad < n_rows) return set_error(PJDS_EINVAL, "bad arguments");
  *bytes = cg_bytes(n_rows, vec_dtype == PJDS_F64 ? 8 : 4);
  return PJDS_OK;
}

extern "C" int pjds_cg_solve(const pjds_dev *A_hi, const pjds_dev *A_lo, const double *b, double *x,
                             const pjds_cg_opts *opts, pjds_cg_result *res, void *work, size_t work_bytes,
                             void *stream) {
  clear_error();
  int rc = check_square_permuted(A_hi, "A_hi");
  if (rc) return rc;
  if (A_hi->dtype != PJDS_F64) return set_error(PJDS_EINVAL, "A_hi must hold fp64 values");
  if (!A_lo) A_lo = A_hi;
  if ((rc = check_square_permuted(A_lo, "A_lo"))) return rc;
  if (A_lo->n_rows != A_hi->n_rows) return set_error(PJDS_EINVAL, "A_lo and A_hi differ in size");
  if (A_hi->n_rows == 0) return PJDS_OK;
  if (!b || !x || !work) return set_error(PJDS_EINVAL, "b, x or work is NULL");
  pjds_cg_opts o{6, 50, 0.0, 1, 0};
  if (opts) {
    o = *opts;
    if (o.max_outer <= 0) o.max_outer = 6;
    if (o.inner_iters <= 0) o.inner_iters = 50;
  }
  if (o.inner_iters > 100000 || o.max_outer > 100000) return set_error(PJDS_EINVAL, "iteration counts too large");
  const bool low = A_lo->dtype != PJDS_F64;
  const size_t need = cg_bytes(A_hi->n_rows, low ? 4 : 8);
  if (work_bytes < need) return set_error(PJDS_EINVAL, "workspace of %zu bytes is smaller than %zu", work_bytes, need);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  return low ? cg_run<float>(A_hi, A_lo, b, x, o, res, work, s) : cg_run<double>(A_hi, A_lo, b, x, o, res, work, s);
}

// ----------------------------------------------------------------------------- Lanczos

static size_t lanczos_bytes(int32_t n, int vec_bytes, int32_t steps) {
  return Reduce::bytes(n) + align256((size_t)steps * 8) + align256((size_t)(steps + 1) * 8) +
         3 * align256((size_t)n * vec_bytes);
}

template <typename TX>
static int lanczos_run(const pjds_dev *A, const TX *v0, int32_t steps, double *alpha_h, double *beta_h, TX *basis,
                       void *work, cudaStream_t s) {
  const int32_t n = A->n_rows, nb = n_blocks_of(n);
  Carve cv{static_cast<char *>(work), 0, 0};
  const Reduce red = Reduce::take(cv, n);
  double *alpha = cv.take<double>((size_t)steps);
  double *beta = cv.take<double>((size_t)steps + 1);
  TX *buf[2] = {cv.take<TX>((size_t)n), nullptr};
  buf[1] = cv.take<TX>((size_t)n);
  TX *w = cv.take<TX>((size_t)n);
  DotKernel<TX, 0> dot;
  int rc;
  if ((rc = make_dot(A, &dot)) || (rc = red.clear(s))) return rc;
  cudaError_t e = cudaMemsetAsync(beta, 0, sizeof(double), s);
  if (e != cudaSuccess) return set_error(PJDS_ECUDA, "lanczos: %s", cudaGetErrorString(e));
  const int32_t g_vec = group_grid<TX>(n);
  // v_j: its row of the caller's basis, else the two buffers in turn
  auto vec = [&](int32_t j) { return basis ? basis + (int64_t)j * n : buf[j & 1]; };
  dev::launch_early(sumsq_kernel<TX>, nb, KT, s, v0, red.partial, n);
  red.sum(nb, s, F_NORM);
  dev::launch_early(lanczos_start_kernel<TX>, nb, KT, s, v0, vec(0), red.scal, n);
  for (int32_t j = 0; j < steps; ++j) {
    TX *const v = vec(j);
    launch_dot(dot, A, v, w, nullptr, red, s, F_LALPHA, j, alpha);  // w = A v, alpha_j = (v, w)
    dev::launch_early(lanczos_orth_kernel<TX>, g_vec, KT, s, w, v, j > 0 ? vec(j - 1) : nullptr, red.scal, red.partial, j, n);
    red.sum(g_vec, s, F_LBETA, j + 1, beta);  // beta_j+1
    if (j + 1 < steps) dev::launch_early(lanczos_next_kernel<TX>, g_vec, KT, s, vec(j + 1), w, red.scal, n);
  }
  if ((rc = launch_check("lanczos steps"))) return rc;
  e = cudaMemcpyAsync(alpha_h, alpha, sizeof(double) * (size_t)steps, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(beta_h, beta, sizeof(double) * ((size_t)steps + 1), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return set_error(PJDS_ECUDA, "lanczos: %s", cudaGetErrorString(e));
  return PJDS_OK;
}

extern "C" int pjds_lanczos_workspace_bytes(int32_t n_rows, int32_t n_pad, int32_t vec_dtype, int32_t steps,
                                            size_t *bytes) {
  clear_error();
  if (!bytes || n_rows < 0 || n_pad < n_rows || steps < 0) return set_error(PJDS_EINVAL, "bad arguments");
  *bytes = lanczos_bytes(n_rows, vec_dtype == PJDS_F64 ? 8 : 4, steps);
  return PJDS_OK;
}

extern "C" int pjds_lanczos(const pjds_dev *A, const void *v0, int32_t steps, double *alpha_host, double *beta_host,
                            void *basis, int32_t use_graph, void *work, size_t work_bytes, void *stream) {
  clear_error();
  int rc = check_square_permuted(A, "A");
  if (rc) return rc;
  if (steps <= 0 || steps > 100000) return set_error(PJDS_EINVAL, "steps must be in [1, 100000]");
  if (A->n_rows == 0) return set_error(PJDS_EINVAL, "empty matrix");
  if (!v0 || !alpha_host || !beta_host || !work) return set_error(PJDS_EINVAL, "a pointer argument is NULL");
  const int vb = vector_bytes(A->dtype);
  if (work_bytes < lanczos_bytes(A->n_rows, vb, steps)) return set_error(PJDS_EINVAL, "workspace too small");
  (void)use_graph;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (A->dtype == PJDS_F64)
    return lanczos_run<double>(A, static_cast<const double *>(v0), steps, alpha_host, beta_host,
                               static_cast<double *>(basis), work, s);
  return lanczos_run<float>(A, static_cast<const float *>(v0), steps, alpha_host, beta_host,
                            static_cast<float *>(basis), work, s);
}

// ----------------------------------------------------------------------------- tridiagonal eigenpair (host)

namespace {

// number of eigenvalues of T below t (LDL^T Sturm count)
int sturm_below(int32_t k, const double *a, const double *b, double t) {
  int cnt = 0;
  double d = a[0] - t;
  const double tiny = DBL_MIN * 1e3;
  for (int32_t i = 0;; ++i) {
    if (d == 0.0) d = -tiny;
    if (d < 0.0) ++cnt;
    if (i + 1 >= k) break;
    d = (a[i + 1] - t) - b[i + 1] * b[i + 1] / d;
  }
  return cnt;
}

// Solve (T - t I) z = rhs in place by Gaussian elimination with partial
// pivoting on the tridiagonal band (rows may swap with the next row).
void tridiag_solve_pivot(int32_t k, const double *a, const double *b, double t, double *z) {
  std::vector<double> d(k), du(k, 0.0), du2(k, 0.0), dl(k, 0.0);
  for (int32_t i = 0; i < k; ++i) d[i] = a[i] - t;
  for (int32_t i = 0; i + 1 < k; ++i) {
    du[i] = b[i + 1];
    dl[i] = b[i + 1];
  }
  const double eps = DBL_EPSILON * 4.0;
  double scale = 0.0;
  for (int32_t i = 0; i < k; ++i) scale = std::max(scale, fabs(a[i]) + (i ? fabs(b[i]) : 0.0));
  for (int32_t i = 0; i + 1 < k; ++i) {
    if (fabs(d[i]) >= fabs(dl[i])) {
      if (d[i] == 0.0) d[i] = eps * (scale > 0 ? scale : 1.0);
      const double f = dl[i] / d[i];
      d[i + 1] -= f * du[i];
      z[i + 1] -= f * z[i];
      dl[i] = 0.0;
    } else {  // swap rows i and i+1
      const double f = d[i] / dl[i];
      d[i] = dl[i];
      const double tmp = d[i + 1];
      d[i + 1] = du[i] - f * tmp;
      du[i] = tmp;
      if (i + 2 < k) {
        du2[i] = du[i + 1];
        du[i + 1] = -f * du2[i];
      }
      const double zt = z[i];
      z[i] = z[i + 1];
      z[i + 1] = zt - f * z[i + 1];
    }
  }
  if (d[k - 1] == 0.0) d[k - 1] = eps * (scale > 0 ? scale : 1.0);
  z[k - 1] /= d[k - 1];
  if (k > 1) z[k - 2] = (z[k - 2] - du[k - 2] * z[k - 1]) / d[k - 2];
  for (int32_t i = k - 3; i >= 0; --i) z[i] = (z[i] - du[i] * z[i + 1] - du2[i] * z[i + 2]) / d[i];
}

}  // namespace

extern "C" int pjds_tridiag_extreme(int32_t k, const double *alpha, const double *beta, int32_t which, double *theta,
                                    double *s) {
  clear_error();
  if (k <= 0 || !alpha || !beta || !theta) return set_error(PJDS_EINVAL, "bad arguments");
  double lo = alpha[0], hi = alpha[0];
  for (int32_t i = 0; i < k; ++i) {
    const double r = (i > 0 ? fabs(beta[i]) : 0.0) + (i + 1 < k ? fabs(beta[i + 1]) : 0.0);
    lo = std::min(lo, alpha[i] - r);
    hi = std::max(hi, alpha[i] + r);
  }
  const double span = std::max(hi - lo, DBL_MIN);
  lo -= 1e-12 * span;
  hi += 1e-12 * span;
  const int m = which == 0 ? k - 1 : 0;  // index of the wanted eigenvalue (ascending)
  for (int it = 0; it < 2000; ++it) {
    const double mid = 0.5 * (lo + hi);
    if (mid <= lo || mid >= hi) break;
    if (sturm_below(k, alpha, beta, mid) > m)
      hi = mid;
    else
      lo = mid;
  }
  const double th = 0.5 * (lo + hi);
  *theta = th;
  if (s) {
    std::vector<double> z(k, 1.0);
    for (int it = 0; it < 4; ++it) {
      tridiag_solve_pivot(k, alpha, beta, th, z.data());
      double nrm = 0.0;
      for (double v : z) nrm += v * v;
      nrm = sqrt(nrm);
      if (!(nrm > 0.0) || !std::isfinite(nrm)) return set_error(PJDS_EINVAL, "inverse iteration failed");
      for (double &v : z) v /= nrm;
    }
    // sign convention: largest-magnitude component positive
    int32_t im = 0;
    for (int32_t i = 1; i < k; ++i)
      if (fabs(z[i]) > fabs(z[im])) im = i;
    const double sg = z[im] < 0 ? -1.0 : 1.0;
    for (int32_t i = 0; i < k; ++i) s[i] = sg * z[i];
  }
  return PJDS_OK;
}

// ----------------------------------------------------------------------------- Ritz refinement

static size_t ritz_bytes(int32_t n, int32_t k) {
  return Reduce::bytes(n) + align256((size_t)k * 8) + align256((size_t)n * 8);
}

extern "C" int pjds_ritz_workspace_bytes(int32_t n_rows, int32_t n_pad, int32_t k, size_t *bytes) {
  clear_error();
  if (!bytes || n_rows < 0 || n_pad < n_rows || k <= 0) return set_error(PJDS_EINVAL, "bad arguments");
  *bytes = ritz_bytes(n_rows, k);
  return PJDS_OK;
}

extern "C" int pjds_ritz_refine(const pjds_dev *A_hi, const void *basis, int32_t basis_dtype, int32_t k,
                                const double *s_host, double *y, double *theta, double *rel_residual, void *work,
                                size_t work_bytes, void *stream) {
  clear_error();
  int rc = check_square_permuted(A_hi, "A_hi");
  if (rc) return rc;
  if (A_hi->dtype != PJDS_F64) return set_error(PJDS_EINVAL, "A_hi must hold fp64 values");
  if (k <= 0 || !basis || !s_host || !y || !theta || !rel_residual || !work)
    return set_error(PJDS_EINVAL, "bad arguments");
  if (basis_dtype != PJDS_F64 && basis_dtype != PJDS_F32) return set_error(PJDS_EINVAL, "basis must be f64 or f32");
  const int32_t n = A_hi->n_rows, nb = n_blocks_of(n);
  if (n == 0) return set_error(PJDS_EINVAL, "empty matrix");
  if (work_bytes < ritz_bytes(n, k)) return set_error(PJDS_EINVAL, "workspace too small");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  Carve cv{static_cast<char *>(work), 0, 0};
  const Reduce red = Reduce::take(cv, n);
  double *sd = cv.take<double>((size_t)k);
  double *w = cv.take<double>((size_t)n);
  DotKernel<double, 0> dot;
  if ((rc = make_dot(A_hi, &dot)) || (rc = red.clear(st))) return rc;
  cudaError_t e = cudaMemcpyAsync(sd, s_host, sizeof(double) * (size_t)k, cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return set_error(PJDS_ECUDA, "ritz: %s", cudaGetErrorString(e));
  if (basis_dtype == PJDS_F64)
    dev::launch_early(ritz_combine_kernel<double>, nb, KT, st, static_cast<const double *>(basis), sd, k, n, y, red.partial);
  else
    dev::launch_early(ritz_combine_kernel<float>, nb, KT, st, static_cast<const float *>(basis), sd, k, n, y, red.partial);
  red.sum(nb, st, F_STORE, S_AUX0);
  launch_dot(dot, A_hi, y, w, nullptr, red, st, F_STORE, S_AUX1);  // w = A y, (y, w)
  dev::launch_early(ritz_residual_kernel, nb, KT, st, w, y, red.scal, red.partial, n);
  red.sum(nb, st, F_STORE, S_AUX2);
  if ((rc = launch_check("ritz refine"))) return rc;
  double h[3];
  e = cudaMemcpyAsync(h, red.scal + S_AUX0, sizeof(h), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return set_error(PJDS_ECUDA, "ritz: %s", cudaGetErrorString(e));
  if (!(h[0] > 0.0)) return set_error(PJDS_EINVAL, "Ritz vector is zero");
  *theta = h[1] / h[0];
  *rel_residual = sqrt(h[2] / h[0]) / fabs(*theta);
  return PJDS_OK;
}

// ----------------------------------------------------------------------------- CG without any allocation

// pjds_cg_solve_static: the same solve as pjds_cg_solve, for callers that
// cannot provide a device workspace at all. Its workspace is this file-scope
// device array, which every GPU that loads the library holds until the
// process exits. The array's name is only a host-side stand-in in host code,
// so its device address is looked up once per device with
// cudaGetSymbolAddress and that address is handed to the kernels.
namespace pjds {
namespace kry {

constexpr int32_t CG_STATIC_MAX_ROWS = 131072;
constexpr size_t CG_STATIC_BYTES = (size_t)11 << 19;  // 5.5 MiB
static __device__ __align__(256) unsigned char g_cg_static_scratch[CG_STATIC_BYTES];

constexpr int kMaxDevices = 64;
static void *g_cg_static_ptr[kMaxDevices];
static std::mutex g_cg_static_mu;

// Device address of the static workspace on the current device (set up on
// the first call per device). The address is kept for the life of the
// process: after cudaDeviceReset the module is loaded again and the kept
// address no longer names the array, so the library must not be used across
// a reset of the device.
static int cg_static_workspace(void **out) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return set_error(PJDS_ECUDA, "cudaGetDevice: %s", cudaGetErrorString(e));
  if (dev < 0 || dev >= kMaxDevices) return set_error(PJDS_EINVAL, "device %d outside the supported range", dev);
  std::lock_guard<std::mutex> lock(g_cg_static_mu);
  if (!g_cg_static_ptr[dev]) {
    void *p = nullptr;
    e = cudaGetSymbolAddress(&p, g_cg_static_scratch);
    if (e != cudaSuccess || !p)
      return set_error(PJDS_ECUDA, "cudaGetSymbolAddress of the static workspace: %s", cudaGetErrorString(e));
    g_cg_static_ptr[dev] = p;
  }
  *out = g_cg_static_ptr[dev];
  return PJDS_OK;
}

}  // namespace kry
}  // namespace pjds

extern "C" int pjds_cg_solve_static(const pjds_dev *A_hi, const pjds_dev *A_lo, const double *b, double *x,
                                    const pjds_cg_opts *opts, pjds_cg_result *res, void *stream) {
  clear_error();
  int rc = check_square_permuted(A_hi, "A_hi");
  if (rc) return rc;
  if (A_hi->dtype != PJDS_F64) return set_error(PJDS_EINVAL, "A_hi must hold fp64 values");
  if (!A_lo) A_lo = A_hi;
  if ((rc = check_square_permuted(A_lo, "A_lo"))) return rc;
  if (A_lo->n_rows != A_hi->n_rows) return set_error(PJDS_EINVAL, "A_lo and A_hi differ in size");
  if (A_hi->n_rows > CG_STATIC_MAX_ROWS)
    return set_error(PJDS_EINVAL,
                     "pjds_cg_solve_static handles at most %d rows (got %d); use pjds_cg_solve with a workspace",
                     CG_STATIC_MAX_ROWS, A_hi->n_rows);
  if (A_hi->n_rows == 0) return PJDS_OK;
  if (!b || !x) return set_error(PJDS_EINVAL, "b or x is NULL");
  pjds_cg_opts o{6, 50, 0.0, 1, 0};
  if (opts) {
    o = *opts;
    if (o.max_outer <= 0) o.max_outer = 6;
    if (o.inner_iters <= 0) o.inner_iters = 50;
  }
  if (o.inner_iters > 100000 || o.max_outer > 100000) return set_error(PJDS_EINVAL, "iteration counts too large");
  // No stream, graph or other driver object is created, as this entry point promises.
  o.use_graph = 0;
  const bool low = A_lo->dtype != PJDS_F64;
  const size_t need = cg_bytes(A_hi->n_rows, low ? 4 : 8);
  if (need > CG_STATIC_BYTES)
    return set_error(PJDS_EINVAL, "static workspace of %zu bytes is smaller than %zu", CG_STATIC_BYTES, need);
  void *work = nullptr;
  if ((rc = cg_static_workspace(&work))) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // The array keeps the previous call's contents: cg_run clears its counters and
  // scalars, and writes every vector and partial sum before reading it.
  return low ? cg_run<float>(A_hi, A_lo, b, x, o, res, work, s) : cg_run<double>(A_hi, A_lo, b, x, o, res, work, s);
}
