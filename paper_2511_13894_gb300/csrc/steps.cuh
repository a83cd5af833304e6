// The persistent step kernel: one launch runs all iterations of a chunk (the
// check_period steps between two KKT checks), two matrix passes each; and the
// power iteration on the same passes.
//
// What bounds the per-pass kernels on LPs of up to about a million nonzeros is
// latency: 4 to 5 us per launch inside the graph, then per warp a chain of
// dependent (matrix entry, gather, FP64) operations as long as its rows.  On
// GB300 a load from L2 takes 380 cycles, an FP64 operation 64 (one warp
// instruction per 64 cycles and scheduler, whatever its active lanes), a grid
// barrier with its fences 2,300 to 2,700.  Here
//   - the rows are cut into units of even work (StepPlan) that keep the FP64
//     units of all SMs busy;
//   - the matrix entries of a CTA's units stay in its shared memory for the
//     whole launch, two columns a lane (the kernel runs where they fit);
//   - the passes are ordered in one of two ways.  Barrier: a grid barrier after
//     each pass, gathers through L1 (rows with many nonzeros make a few entries
//     of the gathered vector hot).  Flow: no barrier at all; every entry of the
//     gathered vectors is written together with its step number in one access
//     (16 bytes, FP32: 8), and a gather repeats its load until it finds the
//     number it waits for.  An entry is only overwritten after all its readers
//     have read it: column j gathers y from the rows that hold j, and these are
//     the rows that gather x_bar_j.  Entries of long rows, which most SMs read,
//     are copied to shared memory once per CTA and pass.
// Loop time per iteration, before (two launches) and now, us (GB300, Halpern):
//   FP64  200 x 500 random face 7.9 -> 3.4 (flow), 5000 x 17500 with bounds
//         (averaged) 10.3 -> 5.1 (flow), 2000 x 8000 power law 13.8 -> 6.5 to 9.2
//         (flow; it depends on where the entries lie in L2), 20k x 80k power law
//         18.7 -> 12.7 (barrier)
//   FP32  20k x 80k power law (averaged) 17.7 -> 12.4 (barrier)
#pragma once
#include "kernels.cuh"

namespace pdhgc {

template <class VT>
struct StepMat {
  const VT* __restrict__ val;        // slots (pairs of columns interleaved per lane)
  const int* __restrict__ col;       // slots; -1 = padding
  const StepTask* __restrict__ tasks;
  const StepEpi* __restrict__ epis;
  const int* __restrict__ warp_ptr;  // ctas * kStepWarps + 1
  const int* __restrict__ epi_ptr;   // ctas + 1
  const int* __restrict__ slot_ptr;
  int max_tasks, max_epis, max_part, max_slots;  // per CTA (shared-memory layout)
};

// entries (value, step number) of the gathered vectors: 16 bytes (FP64), 8 (FP32)
template <class GT>
struct StepEntry;
template <>
struct StepEntry<double> {
  using type = ulonglong2;
};
template <>
struct StepEntry<float> {
  using type = unsigned long long;
};

struct StepFlow {
  void* fy;             // m entries: y, gathered by the pass over A'
  void* fx;             // n entries: x_bar, gathered by the pass over A
  const unsigned* seq;  // number of this launch's first step; 1 at a phase's start, where all entries are 0
  unsigned* bar;        // barrier mode: arrivals, 0 at launch
  int* err;             // set when a bounded wait ran out
  int limit;            // polls of one wait before that
  int hot_y, hot_x;     // leading entries of y / x_bar that every CTA copies to shared memory
};

template <class T>
struct Vec2;
template <>
struct Vec2<double> {
  using type = double2;
};
template <>
struct Vec2<float> {
  using type = float2;
};

__device__ __forceinline__ double2 ld_stream2(const double2* p) {
  double2 v;
  asm("ld.global.nc.L1::no_allocate.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ float2 ld_stream2(const float2* p) {
  float2 v;
  asm("ld.global.nc.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ int2 ld_stream2(const int2* p) {
  int2 v;
  asm("ld.global.nc.L1::no_allocate.v2.s32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
  return v;
}

// Gathers of a vector that this kernel itself rewrites between passes: plain
// (coherent) loads, never the read-only path; the barrier's acquire drops the
// lines of the previous pass from L1
__device__ __forceinline__ double ld_iter(const double* p) {
  double v;
  asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ float ld_iter(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}

// Pairs of steps whose gathers a lane keeps in flight.  FP64 tasks are short (4
// to 8 steps on the LPs measured, kStepMaxCols at most): 4 pairs instead of 2 measured 14.1 against 12.8 us per iteration
// on the 20k x 80k power law.  FP32 tasks have up to 32 steps in SELL rows and
// 128 in long ones: 8 pairs (4 in flow order, whose entries take twice the
// registers) are what 128 registers hold without spilling.
template <bool kFlow, class VT>
constexpr int kStepPairs = std::is_same<VT, float>::value ? (kFlow ? 4 : 8) : 2;
constexpr int kStepWaitLimit = 1 << 21;        // polls of one wait (about a second); a handle can set fewer

__device__ __forceinline__ void ld_entry(const ulonglong2* p, double& v, unsigned& seq) {
  unsigned long long a, b;
  asm volatile("{\n\t.reg .b128 q;\n\tld.relaxed.gpu.global.b128 q, [%2];\n\tmov.b128 {%0, %1}, q;\n\t}"
               : "=l"(a), "=l"(b)
               : "l"(p));
  v = __longlong_as_double((long long)a);
  seq = (unsigned)b;
}
__device__ __forceinline__ void st_entry(ulonglong2* p, double v, unsigned seq) {
  asm volatile("{\n\t.reg .b128 q;\n\tmov.b128 q, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], q;\n\t}" ::"l"(p),
               "l"((unsigned long long)__double_as_longlong(v)), "l"((unsigned long long)seq)
               : "memory");
}
__device__ __forceinline__ void ld_entry(const unsigned long long* p, float& v, unsigned& seq) {
  unsigned long long a;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(a) : "l"(p));
  v = __uint_as_float((unsigned)a);
  seq = (unsigned)(a >> 32);
}
__device__ __forceinline__ void st_entry(unsigned long long* p, float v, unsigned seq) {
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p),
               "l"((unsigned long long)__float_as_uint(v) | ((unsigned long long)seq << 32))
               : "memory");
}

// matrix entries of one batch of PB pairs
template <class VT, int PB>
struct StepHead {
  typename Vec2<VT>::type v[PB];
  int2 c[PB];
};

template <class VT, int PB>
__device__ __forceinline__ void step_load(StepHead<VT, PB>& h, const typename Vec2<VT>::type* vp, const int2* cp,
                                          int p, int np) {
#pragma unroll
  for (int u = 0; u < PB; ++u) {
    if (p + u < np) {
      h.c[u] = cp[(p + u) * 32];
      h.v[u] = vp[(p + u) * 32];
    } else {
      h.c[u] = make_int2(-1, -1);
    }
  }
}

// the vector a pass gathers: entries of step `want` (wait), or the plain vector
// that the previous kernel left (the first pass of a launch)
template <class GT>
struct StepSrc {
  const typename StepEntry<GT>::type* entries;
  unsigned want;
  bool wait;
  GT* hot;   // the CTA's copy of the first n_hot values in shared memory (wait only)
  int n_hot;
};

// copies the hot values of step `want` into shared memory
template <class GT>
__device__ __forceinline__ void step_fetch_hot(const StepSrc<GT>& src, bool& failed, int* err, int limit) {
  for (int j = threadIdx.x; j < src.n_hot; j += kStepThreads) {
    GT v;
    unsigned q;
    for (int i = 0;; ++i) {
      ld_entry(src.entries + j, v, q);
      if ((int)(q - src.want) >= 0 || failed) break;  // newer: all rows that read entry j are done
      if (i > 256) __nanosleep(100);
      if (i >= limit) {
        failed = true;
        atomicExch(err, 2);
      }
    }
    src.hot[j] = v;
  }
  failed = __any_sync(0xffffffffu, failed);
}

template <bool kFlow, int PB, class Op>
__device__ __forceinline__ void step_consume(const Op& op, typename Op::Acc& acc,
                                             const StepHead<typename Op::VT, PB>& h,
                                             const StepSrc<typename Op::GT>& src, bool& failed, int* err,
                                             int limit) {
  using GT = typename Op::GT;
  constexpr int B = 2 * PB;
  GV<GT, 1> g[B];
  int c[B];
#pragma unroll
  for (int u = 0; u < PB; ++u) {
    c[2 * u] = h.c[u].x;
    c[2 * u + 1] = h.c[u].y;
  }
  if (kFlow && src.wait) {
    unsigned q[B];
#pragma unroll
    for (int u = 0; u < B; ++u) {
      q[u] = src.want;
      if (c[u] >= src.n_hot) ld_entry(src.entries + c[u], g[u].v[0], q[u]);
    }
#pragma unroll
    for (int u = 0; u < B; ++u)
      if (c[u] >= 0 && c[u] < src.n_hot) g[u].v[0] = src.hot[c[u]];
    bool stale = false;
#pragma unroll
    for (int u = 0; u < B; ++u) stale |= q[u] != src.want;
    for (int i = 0; __any_sync(0xffffffffu, stale) && !failed; ++i) {
      if (i > 256) __nanosleep(100);
#pragma unroll
      for (int u = 0; u < B; ++u)
        if (q[u] != src.want) ld_entry(src.entries + c[u], g[u].v[0], q[u]);
      stale = false;
#pragma unroll
      for (int u = 0; u < B; ++u) stale |= q[u] != src.want;
      if (i >= limit) {  // uniform in the warp: it waits no more in this launch
        failed = true;
        if ((threadIdx.x & 31) == 0) atomicExch(err, 2);
      }
    }
  } else {
#pragma unroll
    for (int u = 0; u < B; ++u)
      if (c[u] >= 0) g[u].v[0] = ld_iter(op.gsrc(0) + c[u]);
  }
#pragma unroll
  for (int u = 0; u < PB; ++u) {
    if (h.c[u].x >= 0) op.accum(acc, 0.0, h.v[u].x, g[2 * u]);
    if (h.c[u].y >= 0) op.accum(acc, 0.0, h.v[u].y, g[2 * u + 1]);
  }
}

// what a CTA keeps of one matrix in shared memory
template <class VT>
struct StepLocal {
  const StepTask* tasks;  // of the CTA
  const StepEpi* epis;
  const typename Vec2<VT>::type* val;
  const int2* col;
  int t0, t1, nepis;  // tasks of this warp; CTA rows
};

// the grid's barrier (barrier mode): `target` arrivals in all.  A wait that
// runs out sets the error word, and the CTA waits no more in this launch
__device__ __forceinline__ void step_barrier(const StepFlow& flow, unsigned target, bool& failed) {
  __syncthreads();
  if (threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(flow.bar) : "memory");
    for (int i = 0; !failed; ++i) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(flow.bar) : "memory");
      if (v >= target) break;
      if (i >= flow.limit) {
        failed = true;
        atomicExch(flow.err, 2);
      }
    }
  }
  __syncthreads();
}

// One matrix pass of this CTA.  s_part (the parts of split rows) alternates
// between two buffers from step to step: a warp may be a step ahead of another
// that still adds parts, but not two (the barrier below).
template <bool kFlow, class Op>
__device__ __forceinline__ void step_pass(const Op& op, const StepLocal<typename Op::VT>& L,
                                          typename Op::Acc* __restrict__ s_part, const StepSrc<typename Op::GT>& src,
                                          typename StepEntry<typename Op::GT>::type* __restrict__ dst, unsigned seq,
                                          bool& failed, int* err, int limit, double* part) {
  using VT = typename Op::VT;
  using V2 = typename Vec2<VT>::type;
  using PF = Prefetcher<Op>;
  constexpr int PB = kStepPairs<kFlow, VT>;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (kFlow && src.wait && src.n_hot > 0) {  // uniform over the grid
    step_fetch_hot(src, failed, err, limit);
    __syncthreads();
  }
  // the inputs of this warp's first joined rows: in barrier order they come from
  // L2 (the barrier drops L1), which would follow the join
  StepEpi ep{};
  typename PF::Pre epre{};
  if (!kFlow && warp < L.nepis) {
    ep = L.epis[warp];
    if (lane < ep.nrows) epre = PF::get(op, ep.row + lane);
  }
  for (int t = L.t0; t < L.t1; ++t) {
    const StepTask k = L.tasks[t];
    const int np = k.np;
    const bool split = (k.flags & kStepSplit) != 0;
    const bool lead = lane < k.nrows && !split;  // runs a row's epilogue
    const V2* vp = L.val + (k.base >> 1) + lane;
    const int2* cp = L.col + (k.base >> 1) + lane;
    StepHead<VT, PB> head;
    typename Op::Acc acc;
    acc.zero();
    typename PF::Pre pre{};
    if (lead) pre = PF::get(op, k.row + lane);
    for (int p = 0; p < np; p += PB) {
      step_load<VT, PB>(head, vp, cp, p, np);
      step_consume<kFlow, PB>(op, acc, head, src, failed, err, limit);
    }
    // lanes 0 .. R - 1 hold the rows' parts 0, the next R their parts 1 ...
    const int lg = k.flags & kStepLgMask, R = 32 >> lg;
    if (std::is_same<VT, float>::value && lg < 5) {  // SELL parts: in part order
      const typename Op::Acc own = acc;
      for (int q = 1; q < (1 << lg); ++q) acc.add(own.shfl_down(0xffffffffu, q * R));
    } else {
      for (int off = 16; off >= R; off >>= 1) acc.add(acc.shfl_xor(0xffffffffu, off));
    }
    if (lead) {
      const typename Op::GT v = PF::epilogue_val(op, k.row + lane, acc, pre, part);
      if constexpr (kFlow) st_entry(dst + k.row + lane, v, seq);
    } else if (split && lane < k.nrows) {
      s_part[k.slot + lane] = acc;
    }
  }
  if (L.nepis > 0) {  // uniform over the CTA
    __syncthreads();
    for (int e = warp; e < L.nepis; e += kStepWarps) {
      if (kFlow || e != warp) {
        ep = L.epis[e];
        if (lane < ep.nrows) epre = PF::get(op, ep.row + lane);
      }
      const int R = 32 >> ep.lg, r = lane & (R - 1);
      const bool has = r < ep.nrows;
      typename Op::Acc acc;
      acc.zero();
      if constexpr (std::is_same<VT, float>::value) {
        if (has && lane < R)  // in part order
          for (int q = 0; q < ep.k; ++q) acc.add(s_part[ep.slot + q * ep.nrows + r]);
      } else {
        if (has)
          for (int q = lane >> (5 - ep.lg); q < ep.k; q += 1 << ep.lg) acc.add(s_part[ep.slot + q * ep.nrows + r]);
        for (int off = 16; off >= R; off >>= 1) acc.add(acc.shfl_xor(0xffffffffu, off));
      }
      if (has && lane < R) {
        const typename Op::GT v = PF::epilogue_val(op, ep.row + r, acc, epre, part);
        if constexpr (kFlow) st_entry(dst + ep.row + r, v, seq);
      }
    }
  }
}

// copies this CTA's share of a matrix into shared memory
template <class VT>
__device__ __forceinline__ StepLocal<VT> step_stage(const StepMat<VT>& M, unsigned char*& sp) {
  using V2 = typename Vec2<VT>::type;
  StepLocal<VT> L;
  const int b = blockIdx.x, warp = threadIdx.x >> 5;
  const int* wp = M.warp_ptr + b * kStepWarps;
  const int t0 = wp[0], ntasks = wp[kStepWarps] - t0;
  const int e0 = M.epi_ptr[b], s0 = M.slot_ptr[b], ns = M.slot_ptr[b + 1] - s0;
  L.t0 = wp[warp] - t0;
  L.t1 = wp[warp + 1] - t0;
  L.nepis = M.epi_ptr[b + 1] - e0;
  StepTask* st = reinterpret_cast<StepTask*>(sp);
  sp += sizeof(StepTask) * M.max_tasks;
  StepEpi* se = reinterpret_cast<StepEpi*>(sp);
  sp += sizeof(StepEpi) * M.max_epis;
  V2* sv = reinterpret_cast<V2*>(sp);
  sp += sizeof(VT) * M.max_slots;
  int2* sc = reinterpret_cast<int2*>(sp);
  sp += sizeof(int) * M.max_slots;
  for (int t = threadIdx.x; t < ntasks; t += kStepThreads) st[t] = M.tasks[t0 + t];
  for (int t = threadIdx.x; t < L.nepis; t += kStepThreads) se[t] = M.epis[e0 + t];
  const V2* gv = reinterpret_cast<const V2*>(M.val + s0);  // s0: a multiple of 64
  const int2* gc = reinterpret_cast<const int2*>(M.col + s0);
  for (int t = threadIdx.x; t < (ns >> 1); t += kStepThreads) {
    sv[t] = ld_stream2(gv + t);
    sc[t] = ld_stream2(gc + t);
  }
  L.tasks = st;
  L.epis = se;
  L.val = sv;
  L.col = sc;
  return L;
}

// The steps of one chunk.  which: bit 0 the pass over A' (OpT), bit 1 the
// pass over A (OpA); both in a solve, one of them when a pass is timed (it
// then gathers the plain vector every time).  All CTAs must be resident
// (cooperative launch): they wait for each other.
template <bool kFlow, class OpT, class OpA>
__global__ void __launch_bounds__(kStepThreads, 1)
    k_steps(StepMat<typename OpT::VT> T, StepMat<typename OpA::VT> A, OpT opT, OpA opA, StepFlow flow, int period,
            int which) {
  using VT = typename OpT::VT;
  using GT = typename OpT::GT;
  using Entry = typename StepEntry<GT>::type;
  static_assert(std::is_same<typename OpT::Acc, typename OpA::Acc>::value && sizeof(typename OpT::Acc) == 8,
                "partial sums are 8 bytes in both passes");
  extern __shared__ __align__(16) unsigned char s_steps[];
  const Scalars* S = opT.S;
  if (S->done) return;  // uniform over the grid
  const long long left = S->max_iters - S->k;
  const int n_it = left < period ? (int)left : period;
  unsigned char* sp = s_steps;
  const StepLocal<VT> LT = step_stage(T, sp);
  const StepLocal<VT> LA = step_stage(A, sp);
  typename OpT::Acc* part_t = reinterpret_cast<typename OpT::Acc*>(sp);
  typename OpT::Acc* part_a = part_t + 2 * T.max_part;
  GT* s_hy = reinterpret_cast<GT*>(part_a + 2 * A.max_part);
  GT* s_hx = s_hy + flow.hot_y;
  Entry *fx = static_cast<Entry*>(flow.fx), *fy = static_cast<Entry*>(flow.fy);
  const unsigned seq0 = *flow.seq;
  const bool both = which == 3;
  bool failed = false;
  unsigned target = 0;
  __syncthreads();
  for (int i = 0; i < n_it; ++i) {
    opT.it = both ? i : 0;  // a timed pass replays a step inside a chunk: the Halpern weights end with the chunk
    opA.it = opT.it;
    const unsigned seq = both ? seq0 + (unsigned)i : 0u;
    if (which & 1) {
      if (!kFlow && target) step_barrier(flow, target, failed);
      target += gridDim.x;
      step_pass<kFlow>(opT, LT, part_t + (i & 1) * T.max_part, StepSrc<GT>{fy, seq - 1, both && i > 0, s_hy, flow.hot_y},
                       fx, seq, failed, flow.err, flow.limit, nullptr);
    }
    if (which & 2) {
      if (!kFlow && target) step_barrier(flow, target, failed);
      target += gridDim.x;
      step_pass<kFlow>(opA, LA, part_a + (i & 1) * A.max_part, StepSrc<GT>{fx, seq, both, s_hx, flow.hot_x}, fy, seq,
                       failed, flow.err, flow.limit, nullptr);
    }
  }
}

// ---- power iteration ---------------------------------------------------------

// out = scale * (matrix v); the caller's partial gets the sum of out^2
struct PowerOp {
  using Acc = SumD<1>;
  static constexpr int NG = 1;
  using VT = double;
  using GT = double;
  const double* v;
  double* out;
  double scale;
  struct Pre {};
  __device__ const double* gsrc(int) const { return v; }
  __device__ void accum(Acc& a, double, double val, const GV<double, 1>& g) const { a.v[0] = fma(val, g.v[0], a.v[0]); }
  __device__ Pre prefetch(int) const { return Pre{}; }
  __device__ double epilogue_pre(int r, const Acc& a, const Pre&, double* part) const {
    const double x = scale * a.v[0];
    out[r] = x;
    *part += x * x;
    return x;
  }
};

// `iters` steps of u = A v / |v'|, v' = A' u from `v` (of norm 1), then
// partials[b] = CTA b's part of |A v / |v||^2.  The per-pass form takes four
// launches a step (two passes, the norm, the division): 31 us on a 200 x 500
// LP and 45 us on 20k x 80k; here two passes and two barriers.  v is not divided
// by its norm: the next row sums are (m divisions and a pass over v less).
// norm_part: one double per CTA.
__global__ void __launch_bounds__(kStepThreads, 1)
    k_power(StepMat<double> T, StepMat<double> A, Scalars* S, const double* v, double* u, double* w,
            double* __restrict__ norm_part, double* __restrict__ partials, StepFlow flow, int iters) {
  extern __shared__ __align__(16) unsigned char s_steps[];
  __shared__ double s_red[kStepWarps];
  __shared__ double s_norm;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned char* sp = s_steps;
  const StepLocal<double> LT = step_stage(T, sp);
  const StepLocal<double> LA = step_stage(A, sp);
  SumD<1>* part_t = reinterpret_cast<SumD<1>*>(sp);
  SumD<1>* part_a = part_t + T.max_part;
  bool failed = false;
  unsigned target = 0;
  double scale = 1.0;
  __syncthreads();
  // this CTA's sum of squares, in a fixed order
  auto block_sum = [&](double x, double* out) {
    for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
    if (lane == 0) s_red[warp] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int q = 1; q < kStepWarps; ++q) x += s_red[q];
      out[blockIdx.x] = x;
    }
  };
  const StepSrc<double> plain{nullptr, 0u, false, nullptr, 0};
  ulonglong2* const none = nullptr;
  for (int k = 0; k <= iters; ++k) {
    double sq = 0.0;
    step_pass<false>(PowerOp{k == 0 ? v : w, u, scale}, LA, part_a, plain, none, 0u, failed, flow.err, flow.limit, &sq);
    if (k == iters) {
      block_sum(sq, partials);
      return;
    }
    step_barrier(flow, target += gridDim.x, failed);
    sq = 0.0;
    step_pass<false>(PowerOp{u, w, 1.0}, LT, part_t, plain, none, 0u, failed, flow.err, flow.limit, &sq);
    block_sum(sq, norm_part);
    step_barrier(flow, target += gridDim.x, failed);
    if (warp == 0) {
      double x = 0.0;
      for (int b = lane; b < (int)gridDim.x; b += 32) x += __ldcg(norm_part + b);
      for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
      if (lane == 0) s_norm = sqrt(x);
    }
    __syncthreads();
    if (s_norm == 0.0) {  // A_hat v = 0: the same in every CTA
      if (blockIdx.x == 0 && threadIdx.x == 0) S->pi_zero = 1;
      return;
    }
    scale = 1.0 / s_norm;
  }
}

// Slots of the step layout from CSR arrays: a warp per task.  Step j of a
// task: pair j / 2, element j % 2, at base + (j / 2) * 64 + 2 * lane + j % 2.
template <class VT>
__global__ void k_step_fill(const StepTask* __restrict__ tasks, const StepSrcMap* __restrict__ map,
                            const int* __restrict__ slot0, int ntasks, const int* __restrict__ rp,
                            const int* __restrict__ col, const double* __restrict__ val, int* __restrict__ pcol,
                            VT* __restrict__ pval) {
  const int t = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (t >= ntasks) return;
  const StepTask k = tasks[t];
  const StepSrcMap mp = map[t];
  const int R = 32 >> (k.flags & kStepLgMask), r = lane & (R - 1), q = lane / R;
  const bool has = r < k.nrows;
  const int e0 = has ? rp[k.row + r] : 0, len = has ? rp[k.row + r + 1] - e0 : 0;
  const long long base = (long long)slot0[t] + k.base;
  for (int j = 0; j < 2 * k.np; ++j) {
    const long long e = (long long)j * mp.sj + (long long)q * mp.sq + mp.off;
    const bool in = j < mp.jmax && e < len;
    const long long s = base + (long long)(j >> 1) * 64 + 2 * lane + (j & 1);
    if (pcol) pcol[s] = in ? col[e0 + e] : -1;
    if (pval) pval[s] = in ? (VT)val[e0 + e] : VT(0);
  }
}

}  // namespace pdhgc
