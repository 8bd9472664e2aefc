// The small-system CG solve (cg.cu) as krylov.cu calls it.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

#include "common.h"
#include "pjds_krylov.h"

namespace pjds {
namespace kry {

// Results of a solve in device memory.
struct CgOut {
  double bnorm2, norm;
  int32_t outer, n_history;
  double history[PJDS_CG_HISTORY];  // ||r|| before each outer step, then the final one
};

// A solve: the caller's vectors and the workspace's.
struct CgSystem {
  const double *b;
  double *x, *r64;
  void *r, *p, *q;  // of the inner type
  void *slots;      // cg_slots_bytes()
  CgOut *out;
  pjds_cg_result *res;
  int32_t max_outer, inner;
  double tol;
};

size_t cg_slots_bytes();

// The whole solve in one cooperative launch, if the system is small enough for it
// and the context holds all its CTAs at once (*taken); waits for the stream then.
int cg_small(const pjds_dev *Ah, const pjds_dev *Al, const CgSystem &c, bool *taken, cudaStream_t s);

}  // namespace kry
}  // namespace pjds
