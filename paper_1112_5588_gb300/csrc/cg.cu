// Small systems of pjds_cg_solve: the whole solve in one cooperative launch.
//
// Bound by latency: a step is two grid-wide exchanges (2.0 and 2.6 us with 152
// CTAs, gridsum.cuh) and a product of one or two L2 latencies a round, the
// matrix coming from shared memory. Against three launches per step from a
// recorded graph (a graph is recorded for every solve, a reducing launch ends
// with 4.5 us of fp64 trees and a last CTA's pass over the partial sums): 300
// steps on the 27-point stencil, 6 refinements, 1,000 rows fp64 5.6 -> 2.3 ms,
// 4,096 rows fp32 5.2 -> 2.5, 19,683 rows fp32 6.2 -> 2.8 and fp64 5.6 -> 3.2,
// 125,000 rows fp32 7.8 -> 4.6 ms.
#include <math.h>
#include <string.h>

#include "cg.h"
#include "solver.cuh"

namespace pjds {
namespace kry {

template <typename TL>
struct CgArgs {
  Mat hi, lo;
  const double *b;
  double *x, *r64;
  TL *r, *p[2];  // gathered by the products: r and, in turn, the old and the new p
  GridSlots *slots;
  CgOut *out;
  int32_t n, max_outer, inner, n_max;  // n_max: of lo
  double tol;
};

// A step's vectors: p = r + beta p is not published before the product that
// gathers it; the product gathers r and the old p and forms p's elements itself
// (the same rounding, the same bits), so a step has two grid-wide exchanges:
// (p, A p) and (r, r), the second of which also publishes r and the new p.
template <typename TV, typename TL, int T, bool TILE>
__global__ void __launch_bounds__(SOLVER_THREADS, 1) cg_kernel(const __grid_constant__ CgArgs<TL> a) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int U = TILE ? 8 : 4;
  const Rows<T> rows(a.n);
  TL *const lr = reinterpret_cast<TL *>(smem), *const lp = lr + rows.local(), *const lq = lp + rows.local(),
           *const ld = lq + rows.local();
  const int32_t units = rows.local() / rows.UR;
  const Tile<TV, T> tile(smem + ((size_t)rows.local() * 4 * sizeof(TL) + 15) / 16 * 16, units, a.n_max);
  if constexpr (TILE) tile.load(a.lo, rows, units);
  GridSum sum{a.slots, 0};
  double bn2, c = 0.0;
  rows.own([&](int32_t i, int32_t) { c += a.b[i] * a.b[i]; });
  if (!sum.operator()<false>(c, bn2)) return;
  const double bnorm = sqrt(bn2);

  int32_t outer = 0, n_history = 0;
  double nrm;
  for (;; ++outer) {
    // r64 = b - A x, ||r64||
    c = 0.0;
    rows.all([&](int32_t i, int32_t, int32_t) {
      const double acc = row_product_t<double, T, 4>(a.hi, i, rows.s, i < a.n, [&](int32_t k) { return a.x[k]; });
      if (rows.s == 0 && i < a.n) {
        const double v = a.b[i] - acc;
        a.r64[i] = v;
        c += v * v;
      }
    });
    double n2;
    if (!sum.operator()<false>(c, n2)) return;
    nrm = sqrt(n2);
    if (blockIdx.x == 0 && threadIdx.x == 0 && n_history < PJDS_CG_HISTORY) a.out->history[n_history] = nrm;
    if (n_history < PJDS_CG_HISTORY) ++n_history;
    const double rel = bnorm > 0.0 ? nrm / bnorm : nrm;
    if (outer >= a.max_outer || rel <= a.tol || nrm == 0.0) break;

    // r = r64 / ||r64|| in the inner type, d = 0
    const double inv = nrm > 0.0 ? 1.0 / nrm : 0.0;
    double rr;
    c = 0.0;
    rows.own([&](int32_t i, int32_t at) {
      const TL v = (TL)(a.r64[i] * inv);
      lr[at] = a.r[i] = v;
      ld[at] = TL(0);
      c += (double)v * (double)v;
    });
    if (!sum.operator()<true>(c, rr)) return;

    TL be = TL(0);
    for (int32_t it = 0; it < a.inner; ++it) {
      // p = r + beta p, q = A p, alpha = (r, r) / (p, q)
      const TL *const r = a.r, *const old = a.p[(it & 1) ^ 1];
      TL *const now = a.p[it & 1];
      double pq, alpha;
      c = 0.0;
      auto product = [&](int32_t i, int32_t k, auto x) {
        if constexpr (TILE)
          return tile.template product<U>(rows, k, x);
        else
          return row_product_t<TV, T, U>(a.lo, i, rows.s, i < a.n, x);
      };
      rows.all([&](int32_t i, int32_t at, int32_t k) {
        const bool live = i < a.n;
        const auto acc = it == 0 ? product(i, k, [&](int32_t c) { return r[c]; })
                                 : product(i, k, [&](int32_t c) { return dev::fma_acc(be, old[c], r[c]); });
        if (rows.s == 0 && live) {
          const TL p = it == 0 ? lr[at] : dev::fma_acc(be, lp[at], lr[at]);
          lp[at] = now[i] = p;
          lq[at] = (TL)acc;
          c += (double)p * (double)(TL)acc;
        }
      });
      if (!sum.operator()<false>(c, pq, alpha, [&](double t) { return t != 0.0 ? rr / t : 0.0; })) return;
      const TL al = (TL)alpha;

      // d += alpha p, r -= alpha q, beta = (r, r) / (r, r) before
      double rn, beta;
      c = 0.0;
      rows.own([&](int32_t i, int32_t at) {
        ld[at] = dev::fma_acc(al, lp[at], ld[at]);
        const TL v = dev::fma_acc(-al, lq[at], lr[at]);
        lr[at] = a.r[i] = v;
        c += (double)v * (double)v;
      });
      if (!sum.operator()<true>(c, rn, beta, [&](double t) { return rr != 0.0 ? t / rr : 0.0; })) return;
      be = (TL)beta;
      rr = rn;
    }

    // x += ||r64|| d
    rows.own([&](int32_t i, int32_t at) { a.x[i] = fma(nrm, (double)ld[at], a.x[i]); });
    double none;
    if (!sum.operator()<true>(0.0, none)) return;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    a.out->bnorm2 = bn2;
    a.out->norm = nrm;
    a.out->outer = outer;
    a.out->n_history = n_history;
  }
}

template <typename TV, typename TL, int T>
static int launch(const SolverShape &p, CgArgs<TL> &a, bool *fits, cudaStream_t s) {
  return p.tile ? launch_solver(cg_kernel<TV, TL, T, true>, p, a, fits, s)
                : launch_solver(cg_kernel<TV, TL, T, false>, p, a, fits, s);
}

template <typename TV, typename TL>
static int run(const pjds_dev *Ah, const pjds_dev *Al, const CgSystem &c, const SolverShape &p, bool *fits,
               cudaStream_t s) {
  CgArgs<TL> a;
  a.hi = mat_of(Ah), a.lo = mat_of(Al);
  a.b = c.b, a.x = c.x, a.r64 = c.r64;
  a.r = static_cast<TL *>(c.r), a.p[0] = static_cast<TL *>(c.p), a.p[1] = static_cast<TL *>(c.q);
  a.slots = static_cast<GridSlots *>(c.slots), a.out = c.out;
  a.n = Ah->n_rows, a.max_outer = c.max_outer, a.inner = c.inner, a.tol = c.tol;
  a.n_max = Al->n_max;
  switch (p.T) {
    case 4: return launch<TV, TL, 4>(p, a, fits, s);
    case 2: return launch<TV, TL, 2>(p, a, fits, s);
    default: return launch<TV, TL, 1>(p, a, fits, s);
  }
}

size_t cg_slots_bytes() { return sizeof(GridSlots); }

int cg_small(const pjds_dev *Ah, const pjds_dev *Al, const CgSystem &c, bool *taken, cudaStream_t s) {
  *taken = false;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return set_error(PJDS_ECUDA, "device query: %s", cudaGetErrorString(e));
  const SolverShape p = solver_shape(Al, 4, vector_bytes(Al->dtype), sms);
  if (!solver_takes(p, Ah->n_rows, sms)) return PJDS_OK;
  e = cudaMemsetAsync(c.out, 0, sizeof(CgOut), s);
  if (e == cudaSuccess) e = cudaMemsetAsync(c.slots, 0, sizeof(GridSlots), s);
  if (e != cudaSuccess) return set_error(PJDS_ECUDA, "cg: %s", cudaGetErrorString(e));
  int rc = Al->dtype == PJDS_F64   ? run<double, double>(Ah, Al, c, p, taken, s)
           : Al->dtype == PJDS_F32 ? run<float, float>(Ah, Al, c, p, taken, s)
                                   : run<dev::bf16_t, float>(Ah, Al, c, p, taken, s);
  if (rc || !*taken) return rc;
  CgOut h;
  unsigned long long error = 0;
  e = cudaMemcpyAsync(&h, c.out, sizeof(h), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(&error, &static_cast<GridSlots *>(c.slots)->error, sizeof(error), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return set_error(PJDS_ECUDA, "cg: %s", cudaGetErrorString(e));
  if (error) return set_error(PJDS_ECUDA, "cg: a wait between CTAs ran out");
  const double bnorm = sqrt(h.bnorm2);
  auto rel = [&](double v) { return bnorm > 0.0 ? v / bnorm : v; };
  memset(c.res, 0, sizeof(*c.res));
  c.res->outer = h.outer;
  c.res->inner_total = h.outer * c.inner;
  c.res->rel_residual = rel(h.norm);
  c.res->n_history = h.n_history;
  for (int32_t k = 0; k < h.n_history; ++k) c.res->history[k] = rel(h.history[k]);
  return PJDS_OK;
}

}  // namespace kry
}  // namespace pjds
