"""Every shared-memory index of the staged S_r products (gram_stage.cuh, used by gram_s in chains.cu), enumerated on the
host over all subspaces p + q <= 48 and cluster sizes that reach them: no lane reads a vector beyond a chunk's own, both
buffers end within the staging area, and the vectors a lane is responsible for are its own."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1202_0098_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "gram_stage.cuh"
using namespace mka;

static long bad = 0, calls = 0;

// One gram_s call over vectors [n0, n1) with the staging area of a CTA whose work vectors have m_cap rows.
static void call(int p, int q, int atoms, int n0, int n1, int floats) {
  ++calls;
  const int nvec = chunk_vectors(n0, n1), rc = chunk_rows(nvec, floats), vs = chunk_stride(rc);
  const int na = n1 <= 32 ? 4 : 6;              // the kernel's NA
  bool ok = rc >= 4 && rc % 4 == 0 && 2 * nvec * vs <= floats && 4 * rc <= vs;
  for (int nn = n0; nn < n1; nn += 2) {
    const int nb = nn + 1 < n1 ? nn + 1 : n1 - 1, cnt = nb / 8 + 1;
    ok = ok && cnt <= na;
    for (int i = 0; i < cnt; ++i)
      for (int t = 0; t < 8; ++t) {
        const int v = lane_vector(t, i, nb);
        ok = ok && v >= 0 && v < nvec && nvec * vs + v * vs + 4 * (rc - 1) + 3 < floats;
        if (t + 8 * i <= nb) ok = ok && v == t + 8 * i;
      }
    ok = ok && n1 + nb - n0 < nvec;             // the pair's own S W
  }
  if (!ok && ++bad <= 5) std::printf("p=%d q=%d atoms=%d [%d,%d)\n", p, q, atoms, n0, n1);
}

int main() {
  for (int p = 1; p <= 48; ++p)
    for (int q = 0; p + q <= 48; ++q)
      for (int atoms = 1; atoms <= 512; ++atoms) {
        const int nu = p + q, m = 4 * atoms, floats = 12 * m;
        if (m < 6 * nu || !chains_fit(m, p, nu, true)) continue;
        if (q > 0) {
          call(p, q, atoms, 0, p, floats - gs_floats(p));   // the seam
          call(p, q, atoms, p, nu, floats);                 // the second chain
        }
        call(p, q, atoms, 0, nu, floats);                   // one chain alone, or s_j dropped
      }
  std::printf("calls %ld bad %ld\n", calls, bad);
  return bad != 0;
}
"""


def test_no_index_leaves_the_staging_area(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "stage.cpp", tmp_path / "stage"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I" + CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout.split()[1]) > 100000
