"""The memory estimate that decides automatic streaming counts every array that
mra_build allocates for the factors, in each precision form: the doubles of every
form, the column scales of G and H where the Gram products run on the emulation
engine, the row scales of the emulated form.  No GPU: the host header alone."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "mra_sizes.h"
int main(int, char** a) {
  const int M = atoi(a[1]);
  int64_t rc[16];
  for (int m = 0; m < M; ++m) rc[m] = atoll(a[8 + m]);
  printf("%.17g\n", mra::factor_bytes(M, atoi(a[2]), atoi(a[3]), atoi(a[4]), rc, atoll(a[5]), atoll(a[6]), atoll(a[7])));
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    d = tmp_path_factory.mktemp("sizes")
    (d / "main.cpp").write_text(MAIN)
    out = str(d / "sizes")
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_1507_04789_gb300", "csrc"),
                    str(d / "main.cpp"), "-o", out], check=True)
    return out


def arrays(M, r, emu, gram, rc, obs, ls, leaves):
    """Bytes of the factor arrays as mra_build asks for them, one by one."""
    groups = lambda k: (k + 127) // 128
    b = 0
    for m, R in enumerate(rc):
        V, Li, Acc, Om, Lt, G, g = r * m * r, r * r, (m + 1) * (m + 2) // 2 * r * r, (m + 1) * r, r * r, r * m * r, r
        b += 8 * R * (V + Li + Acc + Om + Lt + G + g)
        vexp, liexp, gcol = groups(m * r) * r, r, m * r
        b += 4 * R * (emu * (vexp + liexp) + gram * gcol)
    H, z = obs * M * r, obs
    hcol, hrow = leaves * M * r, obs * groups(M * r)
    return b + 8 * (H + z + ls) + 4 * (gram * hcol + emu * hrow)


# n, M, r: ordinary leaves, sparse leaves of a complete tree, one level
@pytest.mark.parametrize("n,M,r", [(100003, 5, 49), (3000, 7, 32), (60, 1, 64), (5000, 6, 17)])
@pytest.mark.parametrize("form", ["fp64", "mixed", "emu"])
def test_estimate_counts_every_array(exe, n, M, r, form):
    emu, gram = form == "emu", form != "fp64"
    rc = [4 ** m for m in range(M)]
    ls, leaves = n * max(1, n // 4 ** M), 4 ** M
    args = [M, r, int(emu), int(gram), n, ls, leaves, *rc]
    got = float(subprocess.run([exe, *map(str, args)], check=True, capture_output=True, text=True).stdout)
    assert got == arrays(M, r, emu, gram, rc, n, ls, leaves)
    if form == "mixed" and n < leaves:   # the table of H outweighs half of H there
        assert got - arrays(M, r, False, False, rc, n, ls, leaves) > 4 * n * M * r
