// Parts of a solver kernel that runs a whole solve in one cooperative launch, for
// systems small enough that a step's kernels are bound by latency (cg_kernel,
// cg.cu). The CTAs keep their rows for the whole run:
// every vector but those that the next product gathers stays in shared memory,
// and the step's scalars reach all CTAs through grid-wide sums (gridsum.cuh),
// so nothing is launched, recorded or read back per step.
//
// Unit u is 32 / T consecutive sorted rows, one warp's rows with T threads per
// row. CTA c keeps units c, c + G, c + 2G, ... (G CTAs), so that long and short
// rows spread over all CTAs; its warps take them in turn.
#pragma once

#include <algorithm>

#include "common.h"
#include "cooperative.h"
#include "gridsum.cuh"
#include "spmv_kernels.cuh"

namespace pjds {
namespace kry {

constexpr int SOLVER_THREADS = 512;          // at most; one CTA per SM
constexpr int SOLVER_SMEM = 208 * 1024;      // of vectors and matrix, at most

struct Mat {
  const void *val;
  const int32_t *col;
  const int64_t *col_start;
  const int32_t *block_len;
  int32_t b;
};

inline Mat mat_of(const pjds_dev *A) { return Mat{A->val, A->col, A->col_start, A->block_len, A->b}; }

// Product of row i with the vector whose element c is x(c), T lanes (s: this
// lane's place) per row, complete in every lane of the row. Per row the order
// of pjds_spmv_cfg with the same threads per row.
template <typename TV, int T, int U, typename F>
__device__ __forceinline__ typename dev::Acc<TV>::T row_product_t(const Mat &A, int32_t i, int32_t s, bool active,
                                                                  F x) {
  using TA = typename dev::Acc<TV>::T;
  const TV *__restrict__ val = static_cast<const TV *>(A.val);
  const int32_t *__restrict__ col = A.col;
  const int64_t *__restrict__ start = A.col_start;
  const int32_t L = active ? __ldg(A.block_len + (uint32_t)i / (uint32_t)A.b) : 0;
  TA acc = TA(0);
  for (int32_t j = s; j < L; j += U * T) {
    int32_t c[U];
    TV v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (j + u * T < L) {
        const int64_t o = __ldg(start + j + u * T) + i;
        c[u] = __ldg(col + o);
        if constexpr (sizeof(TV) == 2)
          v[u].bits = __ldg(reinterpret_cast<const unsigned short *>(val + o));
        else
          v[u] = __ldg(val + o);
      } else {
        c[u] = -1;
        v[u] = TV{};
      }
    }
    decltype(x(0)) xv[U];
#pragma unroll
    for (int u = 0; u < U; ++u) xv[u] = c[u] >= 0 ? x(c[u]) : decltype(x(0))(0);
#pragma unroll
    for (int u = 0; u < U; ++u) acc = c[u] >= 0 ? dev::fma_acc(dev::to_acc(v[u]), (TA)xv[u], acc) : acc;
  }
#pragma unroll
  for (int o = T / 2; o >= 1; o /= 2) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  return acc;
}

// This thread's rows.
template <int T>
struct Rows {
  static constexpr int UR = 32 / T;  // rows of a unit
  int32_t n, n_units, w, nw, sub, s;

  __device__ __forceinline__ explicit Rows(int32_t n_)
      : n(n_), n_units((n_ + UR - 1) / UR), w(threadIdx.x >> 5), nw(blockDim.x >> 5), sub((threadIdx.x & 31) / T),
        s((threadIdx.x & 31) % T) {}

  // rows of a CTA's vectors
  __device__ __forceinline__ int32_t local() const {
    return (n_units + (int32_t)gridDim.x - 1) / (int32_t)gridDim.x * UR;
  }

  // f(row, its index in the CTA's vectors, unit of the CTA) for each row of the warp's units, by
  // every lane of the row (row >= n: a lane without a row)
  template <typename F>
  __device__ __forceinline__ void all(F f) const {
    for (int32_t k = w, u = w * (int32_t)gridDim.x + (int32_t)blockIdx.x; u < n_units;
         k += nw, u += nw * (int32_t)gridDim.x)
      f(u * UR + sub, k * UR + sub, k);
  }

  // f(row, its index) by the first lane of each row
  template <typename F>
  __device__ __forceinline__ void own(F f) const {
    all([&](int32_t i, int32_t at, int32_t) {
      if (s == 0 && i < n) f(i, at);
    });
  }
};

// A CTA's rows of a matrix in shared memory: entry j of the r-th row of unit k
// at base[k] + j UR + r, so that a warp's lanes read consecutive elements. A
// grid-wide exchange drops the SM's L1 (its acquire), so a product from global
// memory would take the matrix from L2 again at every step, two dependent loads
// before each gather.
template <typename TV, int T>
struct Tile {
  static constexpr int UR = 32 / T;
  int32_t *base;  // [units + 1]
  int32_t *col;
  TV *val;

  __device__ __forceinline__ Tile(unsigned char *p, int32_t units, int32_t n_max) {
    const int64_t e = (int64_t)units * UR * n_max;
    val = reinterpret_cast<TV *>(p);
    p += (e * (int64_t)sizeof(TV) + 15) / 16 * 16;
    col = reinterpret_cast<int32_t *>(p);
    p += (e + 3) / 4 * 16;
    base = reinterpret_cast<int32_t *>(p);
  }

  __device__ __forceinline__ void load(const Mat &A, const Rows<T> &rows, int32_t units) const {
    for (int32_t k = threadIdx.x; k < units; k += blockDim.x) {
      const int64_t i = ((int64_t)k * gridDim.x + blockIdx.x) * UR;
      base[k + 1] = i < rows.n ? __ldg(A.block_len + (uint32_t)i / (uint32_t)A.b) * UR : 0;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      int32_t at = 0;
      base[0] = 0;
      for (int32_t k = 0; k < units; ++k) base[k + 1] = at += base[k + 1];
    }
    __syncthreads();
    const TV *__restrict__ gval = static_cast<const TV *>(A.val);
    for (int32_t k = rows.w; k < units; k += rows.nw) {
      const int64_t i = ((int64_t)k * gridDim.x + blockIdx.x) * UR + rows.sub;
      const int32_t L = (base[k + 1] - base[k]) / UR;
      for (int32_t j = rows.s; j < L; j += T) {
        const int64_t o = __ldg(A.col_start + j) + i;
        col[base[k] + j * UR + rows.sub] = __ldcs(A.col + o);
        val[base[k] + j * UR + rows.sub] = dev::ld_stream1(gval + o);
      }
    }
    __syncthreads();
  }

  // the product of the row of unit k that this lane shares, as row_product_t
  template <int U, typename F>
  __device__ __forceinline__ typename dev::Acc<TV>::T product(const Rows<T> &rows, int32_t k, F x) const {
    using TA = typename dev::Acc<TV>::T;
    const int32_t end = base[k + 1];
    TA acc = TA(0);
    for (int32_t j = base[k] + rows.s * UR + rows.sub; j < end; j += U * 32) {
      int32_t c[U];
      decltype(x(0)) xv[U];
#pragma unroll
      for (int u = 0; u < U; ++u) c[u] = j + u * 32 < end ? col[j + u * 32] : -1;
#pragma unroll
      for (int u = 0; u < U; ++u) xv[u] = c[u] >= 0 ? x(c[u]) : decltype(x(0))(0);
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (c[u] >= 0) acc = dev::fma_acc(dev::to_acc(val[j + u * 32]), (TA)xv[u], acc);
    }
#pragma unroll
    for (int o = T / 2; o >= 1; o /= 2) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    return acc;
  }
};

// bytes of a Tile of `units` units of `ur` rows of at most n_max entries
inline size_t tile_bytes(int64_t units, int64_t ur, int64_t n_max, int value_bytes) {
  const int64_t e = units * ur * n_max;
  return (size_t)((units + 1 + 3) / 4 * 16 + (e + 3) / 4 * 16 + (e * value_bytes + 15) / 16 * 16);
}

struct SolverShape {
  int32_t T, grid, threads;
  size_t smem;    // of the vectors, and of the matrix if tile
  bool tile;      // the matrix is in shared memory
};

// Shape for the steps' matrix, with `vectors` vectors of vec_bytes per row in
// shared memory, and the matrix too if it fits: up to 4 threads per row while the rows
// alone leave the GPU's threads idle and a row has entries for them (27-point
// stencil, fp32 CG of 300 steps: 4,096 rows T = 1 / 2 / 4 / 8 2.75 / 2.48 / 2.37
// / 2.45 ms, 19,683 rows 3.02 / 2.74 / 2.88 / 3.23 ms, 125,000 rows 4.57 / 4.99 /
// 5.59 / 7.48 ms).
inline SolverShape solver_shape(const pjds_dev *A, int vectors, int vec_bytes, int sms) {
  const int32_t n = A->n_rows;
  const double mean = (double)A->nnz / n;
  SolverShape p{1, 1, 32, 0, false};
  while (p.T < 4 && (int64_t)n * p.T * 2 <= (int64_t)sms * SOLVER_THREADS && mean >= 2.0 * p.T) p.T *= 2;
  const int64_t ur = 32 / p.T, units = (n + ur - 1) / ur;
  p.grid = (int32_t)std::min<int64_t>(std::min(sms, GS_MAX_CTAS), std::max<int64_t>(1, (units + 3) / 4));
  const int64_t per = (units + p.grid - 1) / p.grid;
  p.threads = 32 * (int32_t)std::min<int64_t>(SOLVER_THREADS / 32, std::max<int64_t>(per, 4));
  p.smem = (size_t)((per * ur * vectors * vec_bytes + 15) / 16 * 16);
  const size_t tile = tile_bytes(per, ur, A->n_max, value_bytes(A->dtype));
  if (p.smem + tile <= SOLVER_SMEM) {
    p.tile = true;
    p.smem += tile;
  }
  return p;
}

// Whether to take a system of n rows: while the matrix fits in the SMs' shared
// memory, else up to one row per thread. Beyond, the launches of krylov.cu keep
// more loads in flight (27-point stencil, fp32 CG of 300 steps from global
// memory: 64,000 rows 5.7 against 7.5 ms, 125,000 rows 8.6 against 7.8, 216,000
// rows 11.8 against 9.0). Short rows fit up to several times as many (CG of 200
// steps, one launch / a launch for every step: rows of 3 entries fp32 100,000 rows
// 2.0 / 3.4 ms, 300,000 2.5 / 3.8, 800,000 4.2 / 5.4, fp64 300,000 rows 4.0 / 4.3;
// rows of 7 fp32 300,000 rows 2.7 / 3.9, fp64 200,000 rows 3.2 / 4.3).
inline bool solver_takes(const SolverShape &p, int32_t n, int sms) { return p.tile || n <= sms * SOLVER_THREADS; }

// Launch a solver kernel; all its CTAs are resident, as they wait for one another.
// *fits: false where the context does not hold so many (it may be limited to some
// of the SMs); nothing ran then.
template <typename Args>
int launch_solver(void (*kernel)(const Args), const SolverShape &p, Args &a, bool *fits, cudaStream_t s) {
  void *args[] = {&a};
  cudaError_t e = cudaSuccess;
  if (p.smem > 40 * 1024)
    e = cudaFuncSetAttribute((const void *)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SOLVER_SMEM);
  if (e == cudaSuccess)
    e = launch_cooperative((const void *)kernel, (unsigned)p.grid, (unsigned)p.threads, args, p.smem, s);
  *fits = e != cudaErrorCooperativeLaunchTooLarge;
  return e == cudaSuccess || !*fits ? PJDS_OK : set_error(PJDS_ECUDA, "solver launch: %s", cudaGetErrorString(e));
}

}  // namespace kry
}  // namespace pjds
