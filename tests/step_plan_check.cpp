// Checks plan_steps on the CPU: the slots that the fill kernel writes and the
// sums that the step kernel forms are replayed from the plan.  Reads an LP
// (int64 m, n, nnz; row_ptr; int32 col; double val), prints "ok" or the fault.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <string>
#include <vector>

#include "../paper_2511_13894_gb300/csrc/host_prep.h"

using namespace pdhgc;

namespace {

#define REQUIRE(c)                                       \
  do {                                                   \
    if (!(c)) {                                          \
      std::printf("line %d: %s\n", __LINE__, #c);        \
      std::exit(1);                                      \
    }                                                    \
  } while (0)

// the row sum in the per-pass kernel's order (plan_segments), products rounded
double segment_sum(const Csr& C, int32_t r) {
  const int32_t e0 = C.row_ptr[r], len = C.row_ptr[r + 1] - e0;
  auto strided = [&](int32_t first, int32_t step) {
    std::vector<double> lane(32, 0.0);
    for (int l = 0; l < 32; ++l)
      for (int32_t j = first + l; j < len; j += step) lane[l] += C.val[e0 + j];
    for (int off = 16; off > 0; off >>= 1) {
      std::vector<double> t(lane);
      for (int l = 0; l < 32; ++l) lane[l] = t[l] + t[l ^ off];
    }
    return lane[0];
  };
  if (r < C.cta_rows) {
    double s = strided(0, kBlock);
    for (int w = 1; w < kWarpsPerBlock; ++w) s += strided(32 * w, kBlock);
    return s;
  }
  if (r < C.long_rows) return strided(0, 32);
  const int32_t w = C.slice_w[(r - C.long_rows) / kSellH];
  int32_t K = 1;
  while (K < kWarpsPerBlock && K * kColsPerWarp < w) K <<= 1;
  const int32_t cw = (w + K - 1) / K;
  double s = 0.0;
  for (int32_t q = 0; q < K; ++q) {
    double p = 0.0;
    for (int32_t j = q * cw; j < std::min(len, (q + 1) * cw); ++j) p += C.val[e0 + j];
    s = q ? s + p : p;
  }
  return s;
}

void check(const Csr& C, int32_t ctas, bool bulk) {
  StepPlan P;
  plan_steps(C, ctas, bulk, P);
  REQUIRE(P.ok && P.ctas == ctas);
  REQUIRE((int32_t)P.warp_ptr.size() == ctas * kStepWarps + 1 && (int32_t)P.epi_ptr.size() == ctas + 1);
  REQUIRE(P.tasks.size() == P.map.size() && P.tasks.size() == P.slot0.size());
  std::vector<int> used(C.nnz, 0), epilogues(C.rows, 0);
  std::vector<char> slot(P.nslots, 0);
  std::vector<double> sum(C.rows, 0.0);
  for (int32_t b = 0; b < ctas; ++b) {
    const int32_t t0 = P.warp_ptr[b * kStepWarps], t1 = P.warp_ptr[(b + 1) * kStepWarps];
    REQUIRE(t1 - t0 <= P.max_tasks && P.slot_ptr[b + 1] - P.slot_ptr[b] <= P.max_slots);
    std::vector<double> part(P.max_part, 0.0);
    std::vector<int> written(P.max_part, 0);
    for (int32_t t = t0; t < t1; ++t) {
      const StepTask& k = P.tasks[t];
      const StepSrcMap& m = P.map[t];
      const int lg = k.flags & kStepLgMask, R = 32 >> lg;
      REQUIRE(P.slot0[t] == P.slot_ptr[b] && k.base % 64 == 0 && k.nrows <= R && k.row + k.nrows <= C.rows);
      REQUIRE(k.base + 64 * (int64_t)k.np <= P.slot_ptr[b + 1] - P.slot_ptr[b]);
      std::vector<double> lane(32, 0.0);
      for (int l = 0; l < 32; ++l) {
        const int r = l & (R - 1), q = l / R;
        const int32_t e0 = r < k.nrows ? C.row_ptr[k.row + r] : 0;
        const int64_t len = r < k.nrows ? C.row_ptr[k.row + r + 1] - e0 : 0;
        for (int j = 0; j < 2 * k.np; ++j) {
          const int64_t s = (int64_t)P.slot0[t] + k.base + (j >> 1) * 64 + 2 * l + (j & 1);
          REQUIRE(s >= 0 && s < P.nslots && !slot[s]);
          slot[s] = 1;
          const int64_t e = (int64_t)j * m.sj + (int64_t)q * m.sq + m.off;
          if (j < m.jmax && e < len) {
            used[e0 + e]++;
            lane[l] += C.val[e0 + e];
          }
        }
      }
      if (bulk && lg < 5) {
        const std::vector<double> own(lane);
        for (int l = 0; l < R; ++l)
          for (int q = 1; q < (1 << lg); ++q) lane[l] += own[l + q * R];
      } else {
        for (int off = 16; off >= R; off >>= 1) {
          const std::vector<double> t2(lane);
          for (int l = 0; l < 32; ++l) lane[l] = t2[l] + t2[l ^ off];
        }
      }
      for (int r = 0; r < k.nrows; ++r) {
        if (k.flags & kStepSplit) {
          REQUIRE(k.slot >= 0 && k.slot + r < P.max_part && !written[k.slot + r]);
          written[k.slot + r] = 1;
          part[k.slot + r] = lane[r];
        } else {
          epilogues[k.row + r]++;
          sum[k.row + r] = lane[r];
        }
      }
    }
    REQUIRE(P.epi_ptr[b + 1] - P.epi_ptr[b] <= P.max_epis);
    for (int32_t e = P.epi_ptr[b]; e < P.epi_ptr[b + 1]; ++e) {
      const StepEpi& ep = P.epis[e];
      for (int r = 0; r < ep.nrows; ++r) {
        double s = 0.0;
        for (int q = 0; q < ep.k; ++q) {
          const int32_t i = ep.slot + q * ep.nrows + r;
          REQUIRE(i < P.max_part && written[i] == 1);
          written[i] = 2;
          s = q ? s + part[i] : part[i];
        }
        epilogues[ep.row + r]++;
        sum[ep.row + r] = s;
      }
    }
    for (int w : written) REQUIRE(w != 1);
  }
  for (int u : used) REQUIRE(u == 1);
  for (char s : slot) REQUIRE(s == 1);
  for (int32_t r = 0; r < C.rows; ++r) {
    REQUIRE(epilogues[r] == 1);
    const double want = segment_sum(C, r);
    if (bulk)
      REQUIRE(sum[r] == want);  // the same order: the same bits
    else
      REQUIRE(std::abs(sum[r] - want) <= 1e-9);
  }
}

}  // namespace

int main(int, char** argv) {
  FILE* f = std::fopen(argv[1], "rb");
  int64_t h[3];
  REQUIRE(f && std::fread(h, 8, 3, f) == 3);
  const int64_t m = h[0], n = h[1], nnz = h[2];
  std::vector<int64_t> rp(m + 1);
  std::vector<int32_t> col(nnz);
  std::vector<double> val(nnz), b(m, 1.0), c(n, 1.0);
  REQUIRE(std::fread(rp.data(), 8, m + 1, f) == (size_t)m + 1);
  REQUIRE(std::fread(col.data(), 4, nnz, f) == (size_t)nnz && std::fread(val.data(), 8, nnz, f) == (size_t)nnz);
  std::fclose(f);
  Prepared P;
  std::string detail;
  REQUIRE(prepare_lp(P, (int32_t)m, (int32_t)n, nnz, rp.data(), col.data(), val.data(), b.data(), c.data(), nullptr,
                     nullptr, nullptr, detail) == 0);
  for (int32_t ctas : {1, 3, 152})
    for (bool bulk : {false, true}) {
      check(P.A, ctas, bulk);
      check(P.AT, ctas, bulk);
    }
  std::printf("ok\n");
  return 0;
}
