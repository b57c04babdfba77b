"""Host-side rules of the library's headers, compiled into a small program and run here (no GPU)."""
import os
import subprocess

import pytest

from conftest import ROOT
from paper_1611_06765_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include "pnm_context.cuh"

static int failed = 0;
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); failed = 1; } } while (0)

// n systems finish an update, c of them converged: the count is complete after the last one only
static void counts(unsigned long long n, unsigned long long c) {
  const UpdCount all{(n - c) * UpdCount::one(false) + c * UpdCount::one(true)};
  CHECK(all.finished() == n && all.converged() == c);
  const UpdCount before{all.v - UpdCount::one(c == n)};
  CHECK(before.finished() == n - 1);
}

// no size that a 32-bit map indexes may pass it
static void maps() {
  const long ok = (1L << 31) - 3, over = (1L << 31) - 2;
  CHECK(fits_maps(ok, ok, ok, ok) && fits_maps(0, 0, 0, 0));
  CHECK(!fits_maps(over, 1, 1, 1) && !fits_maps(1, over, 1, 1) && !fits_maps(1, 1, over, 1) && !fits_maps(1, 1, 1, 2 * over) && fits_maps(1, 1, 1, over));
  // S_z > 0 channels of one row and one column (two states of a shell): one element each, a row of
  // formed_width(1) as laid out; 2^30 of them have 2^30 elements and 2^32 as laid out
  const long channels = 1L << 30;
  CHECK(fits_maps(1, channels, 1, 1) && !fits_maps(1, channels, channels * formed_width(1), channels * formed_width(1)));
}

// the channels that have always been refused: three 8-byte matrices per problem, in tiles of four, and
// index tables past 227 KB
static void channels() {
  for (int cls = -1; cls <= 1; cls++)
    for (int d = 1; d <= 300; d++) {
      const int nm = cls == 0 ? 2 : 1, h = d / nm;
      const size_t m4 = (h + 3) & ~3, staged = 4 * m4 * sizeof(int) + sizeof(double) * 3 * nm * m4 * m4;
      const bool refused = cls >= 0 && h > 16 && staged > 227 * 1024;
      CHECK(ph_fits(d, 1, cls) == !refused && ph_fits(1, d, cls) == !refused);
    }
}

// contexts whose channels differ do not share what the autotuners measured; densities and twists do
static std::string key(int n, int z, int n2max, double rho, double phi) {
  pnm_ctx c;
  c.sys.resize(1);
  c.sys[0].N = n + z;
  c.sys[0].Z = z;
  c.sys[0].n2max = n2max;
  c.sys[0].rho = rho;
  for (double& p : c.sys[0].phi) p = 0.0;
  c.sys[0].phi[1] = phi;
  return pnm_shape_key(&c);
}
static void keys() {
  const std::string k = key(14, 0, 20, 0.08, 0.0);
  CHECK(k == key(14, 0, 20, 0.16, 0.0) && key(14, 0, 20, 0.08, 0.1) == key(14, 0, 20, 0.08, 0.3));
  CHECK(k != key(14, 0, 20, 0.08, 0.1) && k != key(0, 14, 20, 0.08, 0.0) && k != key(7, 7, 20, 0.08, 0.0));
  CHECK(k != key(14, 0, 21, 0.08, 0.0) && k != key(38, 0, 20, 0.08, 0.0));
}

int main() {
  keys();
  channels();
  maps();
  for (unsigned long long n : {2ull, 3ull, (1ull << 21) - 1, 1ull << 21, (1ull << 21) + 5, (1ull << 31) - 1})
    for (unsigned long long c : {0ull, 1ull, n - 1, n}) counts(n, c);
  return failed;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    src, exe = str(d / "rules.cu"), str(d / "rules")
    open(src, "w").write(PROGRAM)
    cmd = [build.nvcc()] + build.ARCH + ["-std=c++17", "--expt-relaxed-constexpr", "-cudart", "static", "-I" + build.CSRC,
                                         "-I" + os.path.join(ROOT, "include"), src, "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


def test_rules(program):
    r = subprocess.run([program], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
