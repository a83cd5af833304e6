// pdhgc_kkt_eval: Section 2 optimality numbers and the Section 2.1 / 4.2
// metrics of a user-supplied point (x, y) on an LP given as a device CSR,
// without a handle.  The kernels need scratch memory beyond the inputs and
// outputs: an accumulator for A'y (n doubles) and per-block partial sums.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <mutex>
#include <string>

#include "../../include/pdhgc.h"
#include "kkt_eval.h"

namespace pdhgc {

namespace {

__device__ __forceinline__ double proj_dual_ev(double lam, double l, double u) {
  const bool lf = l != -INFINITY, uf = u != INFINITY;
  if (lf && uf) return lam;
  if (lf) return fmax(lam, 0.0);
  if (uf) return fmin(lam, 0.0);
  return 0.0;
}

// Per-block partials of NQ <= 8 quantities (a maximum where the bit of
// kMaxMask is set), in a fixed order: the threads' values go through shared
// memory and warp k folds quantity k.  An FP64 operation costs a scheduler 64
// cycles whatever its active lanes, so 12 warp operations a quantity count
// against the 104 of a shuffle tree in each of the 8 warps and an 8-term sum in
// every thread.
template <int NQ, unsigned kMaxMask>
__device__ void fold_block(const double (&v)[NQ], double* __restrict__ part) {
  static_assert(NQ <= kEvThreads / 32, "a warp per quantity");
  __shared__ double s[NQ][kEvThreads];
#pragma unroll
  for (int k = 0; k < NQ; ++k) s[k][threadIdx.x] = v[k];
  __syncthreads();
  const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (k >= NQ) return;
  const bool is_max = (kMaxMask >> k) & 1u;
  double x = s[k][lane];
  for (int i = lane + 32; i < kEvThreads; i += 32) x = is_max ? fmax(x, s[k][i]) : x + s[k][i];
  for (int off = 16; off > 0; off >>= 1) {
    const double o = __shfl_xor_sync(0xffffffffu, x, off);
    x = is_max ? fmax(x, o) : x + o;
  }
  if (lane == 0) part[k * kEvBlocks + blockIdx.x] = x;
}

// Rows: (Ax)_i, the residual of each row under its sense, b'y, the slack
// metrics of inequality rows, and the scatter of y_i a_ij into A'y.
// Partials (kEvRowQ per block): sum r^2, max |r|, sum b y, off, zero, cand,
// sum b^2.  1 << lg lanes per row, 32 >> lg rows a warp at a time: the lane
// reduction and the row's own operations are warp operations of the FP64 unit
// shared by those rows; a row longer than kEvLong << lg is left to the whole
// warp.  100k x 400k power law, 3.2M nonzeros, the whole evaluation: 996 us
// with a warp per row, single-block norms and 1024 blocks folding with shuffles.
constexpr int kEvLong = 64;
__global__ void __launch_bounds__(kEvThreads) k_ev_rows(EvalInput in, int lg, double* __restrict__ aty,
                                                        double* __restrict__ part) {
  const int lane = threadIdx.x & 31, L = 1 << lg, sub = lane & (L - 1);
  const int rows_per = 32 >> lg;
  const int warps = gridDim.x * (blockDim.x >> 5);
  double q[kEvRowQ] = {0, 0, 0, 0, 0, 0, 0};
  int n_off = 0, n_zero = 0, n_cand = 0;  // off the FP64 unit
  const long long groups = ((long long)in.m + rows_per - 1) / rows_per;
  for (long long g = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); g < groups; g += warps) {
    const long long i = g * rows_per + (lane >> lg);
    const bool has = i < in.m;
    const long long e0 = has ? in.row_ptr[i] : 0, e1 = has ? in.row_ptr[i + 1] : 0;
    const double yi = has ? in.y[i] : 0.0;
    const bool is_long = e1 - e0 > (long long)kEvLong * L;
    double s = 0.0;
    if (!is_long) {
      for (long long e = e0 + sub; e < e1; e += L) {
        const double a = in.val[e];
        const int j = in.col_idx[e];
        s = fma(a, in.x[j], s);
        atomicAdd(aty + j, a * yi);
      }
    }
    for (int off = L >> 1; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    for (unsigned todo = __ballot_sync(0xffffffffu, is_long && sub == 0); todo; todo &= todo - 1) {
      const int from = __ffs(todo) - 1;
      const long long f0 = __shfl_sync(0xffffffffu, e0, from), f1 = __shfl_sync(0xffffffffu, e1, from);
      const double yl = __shfl_sync(0xffffffffu, yi, from);
      double t = 0.0;
      for (long long e = f0 + lane; e < f1; e += 32) {
        const double a = in.val[e];
        const int j = in.col_idx[e];
        t = fma(a, in.x[j], t);
        atomicAdd(aty + j, a * yl);
      }
      for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
      if (lane == from) s = t;
    }
    if (has && sub == 0) {
      const char sn = in.sense ? (char)in.sense[i] : '=';
      const double bi = in.b[i];
      double r = bi - s;
      if (sn == '<') r = fmin(r, 0.0);
      if (sn == '>') r = fmax(r, 0.0);
      q[0] += r * r;
      q[1] = fmax(q[1], fabs(r));
      q[2] += bi * yi;
      q[6] += bi * bi;
      if (sn != '=') {
        const double slack = sn == '<' ? bi - s : s - bi;
        const bool off = slack > 1e-6, zero = fabs(yi) <= 1e-6;
        n_off += off;
        n_zero += zero;
        n_cand += off && zero;
      }
    }
  }
  q[3] = n_off;
  q[4] = n_zero;
  q[5] = n_cand;
  fold_block<kEvRowQ, 2u>(q, part);
}

// columns: lam = c - A'y, z = proj(lam), r_D = lam - z, c'x, the bound part
// of the dual objective and the structural metrics.  Partials (kEvColQ per
// block): sum r_D^2, max |r_D|, c x, l z+ - u z-, off, zero, cand, sum c^2.
__global__ void __launch_bounds__(kEvThreads) k_ev_cols(EvalInput in, const double* __restrict__ aty,
                                                        double* __restrict__ part) {
  double q[kEvColQ] = {0, 0, 0, 0, 0, 0, 0, 0};
  int n_off = 0, n_zero = 0, n_cand = 0;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < in.n; j += gridDim.x * blockDim.x) {
    const double l = in.lb ? in.lb[j] : 0.0;
    const double u = in.ub ? in.ub[j] : INFINITY;
    const double cj = in.c[j];
    const double lam = cj - aty[j];
    const double z = proj_dual_ev(lam, l, u);
    const double rd = lam - z;
    const double xj = in.x[j];
    q[0] += rd * rd;
    q[1] = fmax(q[1], fabs(rd));
    q[2] += cj * xj;
    q[3] += (l != -INFINITY ? l * fmax(z, 0.0) : 0.0) - (u != INFINITY ? u * fmax(-z, 0.0) : 0.0);
    const bool off = fmin(xj - l, u - xj) > 1e-6, zero = fabs(z) <= 1e-6;
    n_off += off;
    n_zero += zero;
    n_cand += off && zero;
    q[7] += cj * cj;
  }
  q[4] = n_off;
  q[5] = n_zero;
  q[6] = n_cand;
  fold_block<kEvColQ, 2u>(q, part);
}

// one CTA, a warp per quantity: fold the partials (lane t takes blocks t, t +
// 32, ... in order) and assemble the numbers
constexpr int kEvFinalThreads = 32 * (kEvRowQ + kEvColQ);
__global__ void __launch_bounds__(kEvFinalThreads) k_ev_final(const double* __restrict__ rpart,
                                                              const double* __restrict__ cpart,
                                                              double* __restrict__ out) {
  __shared__ double q[kEvRowQ + kEvColQ];
  const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const double* p = k < kEvRowQ ? rpart + k * kEvBlocks : cpart + (k - kEvRowQ) * kEvBlocks;
  const bool is_max = k == 1 || k == kEvRowQ + 1;
  double v = 0.0;
#pragma unroll 19
  for (int b = lane; b < kEvBlocks; b += 32) v = is_max ? fmax(v, p[b]) : v + p[b];
  for (int off = 16; off > 0; off >>= 1) {
    const double o = __shfl_xor_sync(0xffffffffu, v, off);
    v = is_max ? fmax(v, o) : v + o;
  }
  if (lane == 0) q[k] = v;
  __syncthreads();
  if (threadIdx.x != 0) return;
  const double* c = q + kEvRowQ;
  const double rP2 = sqrt(q[0]), rD2 = sqrt(c[0]);
  const double nb = sqrt(q[6]), nc = sqrt(c[7]);
  const double pobj = c[2], dobj = q[2] + c[3];
  out[0] = rP2;
  out[1] = rD2;
  out[2] = q[1];
  out[3] = c[1];
  out[4] = pobj;
  out[5] = dobj;
  out[6] = pobj - dobj;
  out[7] = rP2 / (1.0 + nb);
  out[8] = rD2 / (1.0 + nc);
  out[9] = fabs(pobj - dobj) / (1.0 + fabs(pobj) + fabs(dobj));
  out[10] = q[3] + c[4];  // p
  out[11] = q[4] + c[5];  // d
  out[12] = q[5] + c[6];  // candidates
}

}  // namespace

size_t kkt_eval_scratch_doubles(int32_t n) {
  return (size_t)n + (size_t)(kEvRowQ + kEvColQ) * kEvBlocks + kEvOut;
}

int kkt_eval_check(int32_t m, int32_t n, int64_t nnz, const void* row_ptr, const void* col_idx, const void* val,
                   const void* b, const void* c, const void* x, const void* y, const pdhgc_report* out,
                   std::string& detail) {
  if (m < 1 || n < 1 || nnz < 0) {
    detail = "m and n must be >= 1, nnz >= 0";
    return PDHGC_ERR_INVALID_ARG;
  }
  if (!row_ptr || !b || !c || !x || !y || !out || (nnz > 0 && (!col_idx || !val))) {
    detail = "NULL argument";
    return PDHGC_ERR_INVALID_ARG;
  }
  return PDHGC_OK;
}

int kkt_eval_run(const EvalInput& in, double* scratch, cudaStream_t st, pdhgc_report* out, std::string& detail) {
  double* aty = scratch;
  double* rpart = aty + in.n;
  double* cpart = rpart + (size_t)kEvRowQ * kEvBlocks;
  double* res = cpart + (size_t)kEvColQ * kEvBlocks;
  auto fail = [&](cudaError_t e, const char* what) {
    detail = std::string(what) + ": " + cudaGetErrorString(e);
    return e == cudaErrorMemoryAllocation ? PDHGC_ERR_OOM : PDHGC_ERR_CUDA;
  };
  cudaError_t e = cudaMemsetAsync(aty, 0, sizeof(double) * (size_t)in.n, st);
  if (e != cudaSuccess) return fail(e, "kkt_eval clear");
  // lanes per row: about 8 entries a lane of a mean row
  int lg = 0;
  while (lg < 5 && ((int64_t)in.m << (lg + 3)) < in.nnz) ++lg;
  k_ev_rows<<<kEvBlocks, kEvThreads, 0, st>>>(in, lg, aty, rpart);
  k_ev_cols<<<kEvBlocks, kEvThreads, 0, st>>>(in, aty, cpart);
  k_ev_final<<<1, kEvFinalThreads, 0, st>>>(rpart, cpart, res);
  e = cudaGetLastError();
  if (e != cudaSuccess) return fail(e, "kkt_eval launch");
  double h[kEvOut];
  e = cudaMemcpyAsync(h, res, 13 * sizeof(double), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return fail(e, "kkt_eval");
  std::memset(out, 0, sizeof(*out));
  out->rP2 = h[0];
  out->rD2 = h[1];
  out->rPinf = h[2];
  out->rDinf = h[3];
  out->pobj = h[4];
  out->dobj = h[5];
  out->gap = h[6];
  out->rel_p = h[7];
  out->rel_d = h[8];
  out->rel_gap = h[9];
  out->rel_kkt = std::fmax(h[7], std::fmax(h[8], h[9]));
  const int64_t mm = in.m;
  out->off_bound_p = (int64_t)std::llround(h[10]);
  out->zero_rc_d = (int64_t)std::llround(h[11]);
  out->candidates = (int64_t)std::llround(h[12]);
  out->corner_measure = out->candidates > mm ? out->candidates - mm : 0;
  out->primal_push_est = out->off_bound_p > mm ? out->off_bound_p - mm : 0;
  out->dual_push_est = mm > out->zero_rc_d ? mm - out->zero_rc_d : 0;
  const int64_t thr = 2 * mm > 100000 ? 2 * mm : 100000;
  out->should_corner = out->candidates >= thr ? 1 : 0;
  return PDHGC_OK;
}

}  // namespace pdhgc

extern "C" int pdhgc_kkt_eval(int32_t m, int32_t n, int64_t nnz, const int64_t* row_ptr, const int32_t* col_idx,
                              const double* val, const double* b, const double* c, const double* lb,
                              const double* ub, const int8_t* sense, const double* x, const double* y,
                              pdhgc_report* out, void* cuda_stream) {
  std::string detail;
  int rc = pdhgc::kkt_eval_check(m, n, nnz, row_ptr, col_idx, val, b, c, x, y, out, detail);
  if (rc != PDHGC_OK) return pdhgc::set_error_detail(rc, detail);
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const size_t bytes = pdhgc::kkt_eval_scratch_doubles(n) * sizeof(double);
  void* scratch = nullptr;
  cudaError_t e = cudaMallocAsync(&scratch, bytes, st);
  if (e != cudaSuccess)
    return pdhgc::set_error_detail(PDHGC_ERR_OOM, std::string("cudaMallocAsync: ") + cudaGetErrorString(e));
  pdhgc::EvalInput in{m, n, nnz, row_ptr, col_idx, val, b, c, lb, ub, sense, x, y};
  rc = pdhgc::kkt_eval_run(in, static_cast<double*>(scratch), st, out, detail);
  // The evaluation has ended (its results were read): no synchronisation behind
  // the free, at which the device's default pool would unmap the scratch for the
  // next call to map it again.  100k x 400k LP, us a call, new inputs each time:
  // 123 one after another, 230 where the caller synchronises before each, 320
  // with the caller's synchronisation behind it counted in; with a
  // synchronisation here 300 in every case; 990 to 1,010 before the kernels of
  // this file.  Inputs out of L2 add 10
  cudaFreeAsync(scratch, st);
  if (rc != PDHGC_OK) return pdhgc::set_error_detail(rc, detail);
  return PDHGC_OK;
}

// ---------------------------------------------------------------------------
// pdhgc_kkt_eval_noalloc: the same evaluation with its scratch in a
// file-scope device array instead of cudaMallocAsync, for callers that must
// not allocate device memory (see include/pdhgc.h).
// ---------------------------------------------------------------------------
namespace {

constexpr int32_t kNoAllocMaxN = 1 << 18;  // largest n the static scratch holds
constexpr size_t kNoAllocDoubles = (size_t)kNoAllocMaxN + (size_t)(pdhgc::kEvRowQ + pdhgc::kEvColQ) *
                                                               pdhgc::kEvBlocks + pdhgc::kEvOut;

// Shared by every call on a device and kept until the process exits; each call
// overwrites all of it that it reads (the A'y accumulator is zeroed first).
static __device__ __align__(256) double g_kkt_eval_scratch[kNoAllocDoubles];

constexpr int kMaxDevices = 64;
std::mutex g_scratch_mu;
double* g_scratch_ptr[kMaxDevices] = {};

// true when p is device memory of device `dev` in the current context (a
// cached address stays valid until cudaDeviceReset replaces the context)
bool still_device_memory(const void* p, int dev) {
  cudaPointerAttributes a{};
  const cudaError_t e = cudaPointerGetAttributes(&a, p);
  if (e != cudaSuccess) {
    cudaGetLastError();  // not a pointer of this context: clear the error it set
    return false;
  }
  return a.type == cudaMemoryTypeDevice && a.device == dev;
}

// device address of g_kkt_eval_scratch for the current device, looked up
// with that device current on its first call, and again whenever the cached
// address no longer belongs to the device's current context
int scratch_for_current_device(double** out, std::string& detail) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) {
    detail = std::string("cudaGetDevice: ") + cudaGetErrorString(e);
    return PDHGC_ERR_CUDA;
  }
  if (dev < 0 || dev >= kMaxDevices) {
    detail = "device ordinal out of range";
    return PDHGC_ERR_INVALID_ARG;
  }
  std::lock_guard<std::mutex> lock(g_scratch_mu);
  if (!g_scratch_ptr[dev] || !still_device_memory(g_scratch_ptr[dev], dev)) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_kkt_eval_scratch);
    if (e != cudaSuccess || !p) {
      detail = std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e);
      return PDHGC_ERR_CUDA;
    }
    g_scratch_ptr[dev] = static_cast<double*>(p);
  }
  *out = g_scratch_ptr[dev];
  return PDHGC_OK;
}

}  // namespace

extern "C" int pdhgc_kkt_eval_noalloc(int32_t m, int32_t n, int64_t nnz, const int64_t* row_ptr,
                                      const int32_t* col_idx, const double* val, const double* b, const double* c,
                                      const double* lb, const double* ub, const int8_t* sense, const double* x,
                                      const double* y, pdhgc_report* out, void* cuda_stream) {
  std::string detail;
  int rc = pdhgc::kkt_eval_check(m, n, nnz, row_ptr, col_idx, val, b, c, x, y, out, detail);
  if (rc != PDHGC_OK) return pdhgc::set_error_detail(rc, detail);
  if (n > kNoAllocMaxN)
    return pdhgc::set_error_detail(PDHGC_ERR_TOO_LARGE,
                                   "pdhgc_kkt_eval_noalloc: n = " + std::to_string(n) +
                                       " exceeds the static scratch capacity of " +
                                       std::to_string(kNoAllocMaxN) + " columns; use pdhgc_kkt_eval");
  double* scratch = nullptr;
  rc = scratch_for_current_device(&scratch, detail);
  if (rc != PDHGC_OK) return pdhgc::set_error_detail(rc, detail);
  pdhgc::EvalInput in{m, n, nnz, row_ptr, col_idx, val, b, c, lb, ub, sense, x, y};
  rc = pdhgc::kkt_eval_run(in, scratch, static_cast<cudaStream_t>(cuda_stream), out, detail);
  if (rc != PDHGC_OK) return pdhgc::set_error_detail(rc, detail);
  return PDHGC_OK;
}
