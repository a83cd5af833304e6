// Batched solve (see batch.cu): the per-LP result record the device writes,
// and the handle it finishes handed-off LPs on.
#pragma once
#include <stdint.h>

struct pdhgc_lp;

namespace pdhgc {

// pdhgc_lp_create; own_gpu = false keeps the handle on the per-pass kernels,
// which share the GPU with other work: a step kernel's grid (steps.cuh) starts
// only once all of its CTAs fit, so LPs finished beside a running batch would
// wait for it and for each other
int lp_create(pdhgc_lp** out, int32_t m, int32_t n, int64_t nnz, const int64_t* row_ptr, const int32_t* col_idx,
              const double* val, const double* b, const double* c, const double* lb, const double* ub,
              const int8_t* sense, int inputs_on_device, void* cuda_stream, bool own_gpu);

struct BatchReport {
  int32_t status, chosen;
  int64_t iters, restarts;
  double rP2, rD2, rPinf, rDinf, pobj, dobj;
  double p, dd, cand;  // metric counts (off bound, zero reduced cost, candidates)
  double omega, eta, sigma_max, seconds;
};

}  // namespace pdhgc
