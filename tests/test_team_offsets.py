"""The areas of a team's shared memory (csrc/kin_team.cuh) that are in use at
the same time do not overlap: computed on the host, for every species count,
by a small program built from the header itself."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1607_03884_gb300", "csrc")
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

PROGRAM = r"""
#include <cstdio>
#include "kin_team.cuh"
using namespace kin;
struct Area { const char *name; const unsigned char *a, *b; };
template <typename LT> void check(int ns, int nr) {
  MechLayout L{};
  L.ns = ns; L.nr = nr; L.nslots = 6 * nr; L.neff = nr;
  static unsigned char buf[1 << 20];
  const size_t bytes = team_bytes(L, ns, sizeof(LT));
  const TeamBuf<LT> t = carve_team<LT>(L, buf, 0, ns, nullptr);
  const size_t w = t.wstride * sizeof(double);
  auto U = [](const void *p) { return (const unsigned char *)p; };
  // a difference Jacobian with a state per warp: three rate buffers, each
  // warp's vectors, the control block
  Area A[8] = {{"ctl", U(t.ctl), U(t.ctl) + sizeof(TeamCtl)}};
  for (int q = 0; q < 3; ++q) {
    A[1 + q] = {"rates", U(t.C(q)), U(t.C(q)) + w};
    A[4 + q] = {"vectors", U(t.fd(q)), U(t.fd(q)) + 3 * t.nv * sizeof(double)};
  }
  A[7] = {"permutations", U(t.p1), U(t.p1) + 128};
  for (int i = 0; i < 8; ++i) {
    if (A[i].a < buf || A[i].b > buf + bytes) printf("%d species: %s outside\n", ns, A[i].name);
    for (int j = 0; j < i; ++j)
      if (A[i].a < A[j].b && A[j].a < A[i].b)
        printf("%d species, %d reactions: %s over %s\n", ns, nr, A[i].name, A[j].name);
  }
  if (!team_fd_fits(ns)) printf("%d species: not taken\n", ns);
}
int main() {
  for (int ns = 17; ns < 64; ++ns)
    for (int nr : {1, 27, 325}) check<float>(ns, nr);
  printf("done\n");
}
"""


@pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc")
def test_buffers_in_use_together_do_not_overlap(tmp_path):
    src, exe = tmp_path / "areas.cu", tmp_path / "areas"
    src.write_text(PROGRAM)
    subprocess.run([NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-I", CSRC,
                    "-o", str(exe), str(src)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    assert out == "done\n", out
