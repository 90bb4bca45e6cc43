"""Choice of the cluster width of the one-kernel coarse end, with fakes of the CUDA calls: after a
failing one the narrower cluster is taken and no error is left for the next launch to find."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include "rmg_cluster.h"
// argv: opt-in succeeds, then for 16 and 8 blocks whether the query succeeds and what it finds
int main(int, char** v) {
  int pending = 0;
  const int got = rmg::widest_cluster(
      [&] { const bool ok = atoi(v[1]); pending |= !ok; return ok; },
      [&](int n, int* count) {
        const int at = n == 16 ? 2 : 4;
        const bool ok = atoi(v[at]);
        pending |= !ok;
        if (ok) *count = atoi(v[at + 1]);
        return ok;
      },
      [&] { pending = 0; });
  printf("%d %d\n", got, pending);
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("cluster")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-I",
                    os.path.join(ROOT, "paper_2103_11962_gb300", "csrc"), "-o", str(d / "h"),
                    str(d / "h.cpp")], check=True)
    return str(d / "h")


@pytest.mark.parametrize("wide,q16,n16,q8,n8,expect", [
    (1, 1, 9, 1, 19, 16),
    (1, 1, 0, 1, 19, 8),          # 16 do not fit
    (0, 1, 9, 1, 19, 8),          # the opt-in fails
    (1, 0, 0, 1, 19, 8),          # the query for 16 fails
    (0, 1, 9, 0, 0, 0),           # everything fails
    (1, 1, 0, 1, 0, 0),
])
def test_widest_cluster(harness, wide, q16, n16, q8, n8, expect):
    args = [str(a) for a in (wide, q16, n16, q8, n8)]
    out = subprocess.run([harness] + args, check=True, capture_output=True, text=True).stdout
    assert out.split() == [str(expect), "0"]
