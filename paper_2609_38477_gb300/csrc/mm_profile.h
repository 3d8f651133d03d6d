// Work profile of the tensor-core batch products (gemm_mma.cuh), from which the
// host cuts a launch into ranges of equal modeled cost.  Host code only.
#pragma once

#include <cstdint>

namespace seedq {

constexpr int kMaxJ = 9;        // hull rungs (App. B.3: four to eight on the paper's grids)
constexpr int kCostStage = 24;  // stage width (blocks) the profiles assume
constexpr int kProfile = 16;    // columns at which a superblock's profile is kept
constexpr int kMmGroups = 4;    // row groups of a superblock
// Time of a superblock's column that an idle group saves none of, as a share of
// a busy group's.  Measured at 0 / 0.3 / 0.5 / 0.65 / 0.8 / 0.95, b8: 5000 x 5008
// (its last superblock holds 8 rows) 103 / 60 / 48 / 46.6 / 45.5 / 46.5 us, 38408
// x 5008 252 / 227 / 213 / 203 / 197 / 197; 5120 x 5008 45.4.
constexpr double kIdleGroup = 0.8;
constexpr int kProfileFloats = 2 * (kProfile + 1);

// For each set of sixteen rows the kernel passes over every column one of them
// has at a rung; a pass of the group's 32 rows over a stage costs about five
// columns more (fitted to per-CTA times).  Rows missing from a group count as
// its first: the kernel's lanes repeat it.
class MmProfile {
 public:
  MmProfile(int nb, int J, const int32_t *k) : nb_(nb), J_(J), k_(k) {}

  // One group of nr rows, row i's J - 1 breakpoints at rowb[i]: its passes and
  // the sum of k over them in P and K; both, before column nb * i / kProfile,
  // are added to prof[i] and prof[kProfile + 1 + i].
  void add(const int32_t *const *rowb, int nr, float *prof, double &P, double &K) {
    // A group whose rows all have the last one's breakpoints repeats its
    // profile (tensors without a row factor: every group).
    bool same = have_;
    for (int i = 0; i < nr && same; ++i) same = equal(rowb[i], bk_);
    if (!same) {
      measure(rowb, nr);
      have_ = true;
      for (int i = 1; i < nr && have_; ++i) have_ = equal(rowb[i], rowb[0]);
      for (int j = 0; j < J_ - 1; ++j) bk_[j] = rowb[0][j];
    }
    repeat(prof, P, K);
  }
  // The same for a group known to have the breakpoints of the last one.
  void repeat(float *prof, double &P, double &K) const {
    P = P_;
    K = K_;
    for (int i = 0; i < kProfileFloats; ++i) prof[i] += own_[i];
  }

  // Makes a superblock of fewer groups cost what it takes: its columns pass
  // through a CTA hardly faster than a whole one's, the warps of the missing
  // groups idle.  P and K: its groups' sums.
  static void partial(int groups, float *prof, double &P, double &K) {
    const double f = 1.0 + kIdleGroup * (kMmGroups - groups) / groups;
    P *= f;
    K *= f;
    for (int i = 0; i < kProfileFloats; ++i) prof[i] = (float)(prof[i] * f);
  }

 private:
  bool equal(const int32_t *a, const int32_t *b) const {
    for (int j = 0; j < J_ - 1; ++j)
      if (a[j] != b[j]) return false;
    return true;
  }
  void span(int from, int to, double wp, double wk) {
    P_ += wp * (to - from);
    K_ += wk * (to - from);
    for (int i = 1; i <= kProfile; ++i) {
      const int c = (int)((int64_t)nb_ * i / kProfile), n = (c < to ? c : to) - from;
      if (n <= 0) continue;
      own_[i] += (float)(wp * n);
      own_[kProfile + 1 + i] += (float)(wk * n);
    }
  }
  void measure(const int32_t *const *rowb, int nr) {
    constexpr double kPass = 5.0;
    P_ = K_ = 0.0;
    for (float &v : own_) v = 0.f;
    for (int j = 0; j < J_; ++j) {
      int from32 = nb_, to32 = 0;
      for (int s0 = 0; s0 < 32; s0 += 16) {
        int from = nb_, to = 0;
        for (int i = s0; i < s0 + 16; ++i) {
          const int32_t *b = rowb[i < nr ? i : 0];
          const int a = (j > 0) ? b[j - 1] : 0, z = (j < J_ - 1) ? b[j] : nb_;
          if (a < z) {
            from = a < from ? a : from;
            to = z > to ? z : to;
          }
        }
        if (from < to) span(from, to, 0.5, 0.5 * k_[j]);
        from32 = from < from32 ? from : from32;
        to32 = to > to32 ? to : to32;
      }
      // One pass per stage it touches: len / 24 of them, and one more.
      if (from32 < to32) span(from32, to32, kPass / kCostStage + kPass / (to32 - from32), 0.0);
    }
  }

  int nb_, J_;
  const int32_t *k_;
  // The last group measured: its profile, and its breakpoints if they are all
  // its rows' (have_).
  bool have_ = false;
  int32_t bk_[kMaxJ] = {0};
  double P_ = 0.0, K_ = 0.0;
  float own_[kProfileFloats] = {0.f};
};

}  // namespace seedq
