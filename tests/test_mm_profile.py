"""The host-side work profile of the tensor-core products (csrc/mm_profile.h),
compiled for the host: a superblock's profile is the sum of its groups' own,
whichever of them repeat the group before, and ends at the passes and the sum
of k that the groups report."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2609_38477_gb300", "csrc")

PROGRAM = r"""
#include "mm_profile.h"
#include <cmath>
#include <cstdio>
#include <vector>
using namespace seedq;

#define CHECK(c) do { if (!(c)) { std::printf("FAIL line %d: %s\n", __LINE__, #c); return 1; } } while (0)

int main() {
  const int nb = 500, J = 4;
  const int32_t k[J] = {2, 3, 4, 6};
  // Rows of two kinds, in groups that repeat (A A, B B), alternate, mix and end short.
  const int32_t A[3] = {40, 200, 480}, B[3] = {300, 310, 310}, C[3] = {0, 0, 500};
  struct Group { const int32_t *first, *second; int nr; };
  const std::vector<Group> kinds = {{A, A, 32}, {B, B, 32}, {B, B, 32}, {B, B, 32},
                                    {C, C, 32}, {A, A, 32}, {A, A, 32}, {C, C, 32},
                                    {A, B, 32}, {A, B, 32}, {A, A, 32}, {A, A, 7},
                                    {A, A, 7}, {A, A, 32}};
  auto rows = [&](const Group &g, const int32_t **rowb) {
    for (int i = 0; i < g.nr; ++i) rowb[i] = i % 3 == 1 ? g.second : g.first;
  };
  MmProfile all(nb, J, k);
  for (size_t s0 = 0; s0 < kinds.size(); s0 += kMmGroups) {
    float prof[kProfileFloats] = {0.f};
    double want[kProfileFloats] = {0.0}, P = 0.0, K = 0.0;
    for (size_t g = s0; g < kinds.size() && g < s0 + kMmGroups; ++g) {
      const int32_t *rowb[32];
      rows(kinds[g], rowb);
      double p, q, p1, q1;
      all.add(rowb, kinds[g].nr, prof, p, q);
      float own[kProfileFloats] = {0.f};
      MmProfile fresh(nb, J, k);
      fresh.add(rowb, kinds[g].nr, own, p1, q1);
      CHECK(p == p1 && q == q1);
      for (int i = 0; i < kProfileFloats; ++i) want[i] += own[i];
      P += p;
      K += q;
    }
    for (int i = 0; i < kProfileFloats; ++i) CHECK(std::fabs(prof[i] - want[i]) <= 1e-5 * (1.0 + want[i]));
    CHECK(std::fabs(prof[kProfile] - P) <= 1e-5 * P);
    CHECK(std::fabs(prof[2 * kProfile + 1] - K) <= 1e-5 * K);
    for (int i = 0; i < kProfile; ++i) CHECK(prof[i] <= prof[i + 1]);
  }
  std::printf("ok\n");
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_superblock_profile_is_the_sum_of_its_groups(tmp_path):
    src = tmp_path / "profile.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "profile"
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr


PARTIAL = r"""
#include "mm_profile.h"
#include <cmath>
#include <cstdio>
using namespace seedq;

int main() {
  for (int groups = 1; groups <= kMmGroups; ++groups) {
    float prof[kProfileFloats];
    for (int i = 0; i < kProfileFloats; ++i) prof[i] = (float)(i * groups);
    double P = 10.0 * groups, K = 30.0 * groups;
    MmProfile::partial(groups, prof, P, K);
    // Between its groups' own cost and a whole superblock's; the profile in step.
    if (P < 10.0 * groups || P > 10.0 * kMmGroups + 1e-9 || std::fabs(K - 3 * P) > 1e-9) return 1;
    for (int i = 0; i < kProfileFloats; ++i)
      if (std::fabs(prof[i] - i * P / 10.0) > 1e-4 * (1 + prof[i])) return 2;
  }
  std::printf("ok\n");
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_partial_superblock(tmp_path):
    src = tmp_path / "partial.cpp"
    src.write_text(PARTIAL)
    exe = tmp_path / "partial"
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
