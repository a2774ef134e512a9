"""The FP64-emulation engine's tile product against extended-precision sums.

Edges of its tiles: one row and column, slots of 16 rows, K steps of 16, scale
groups of 128, scale passes of 512 columns, the three operand layouts, scales
from tables and from its own pass, elements spread over 60 binary orders.

Bound per entry: every operand is rounded to 2^-49 of its group's scale (two
operands), the dropped digit pairs are below 5 * 2^14 * 2^-64, so a term is off
by at most (2^-48 + 2^-47.6) 2^(e + f) < 2^-46.5 2^(e + f); the double-float sums
and the final rounding add at most 2^-44 of sum |a b| over a few groups.
"""
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHAPES = [(1, 1, 1), (16, 16, 16), (17, 15, 17), (64, 64, 64), (128, 64, 127), (128, 64, 128), (127, 63, 129),
          (100, 33, 448), (128, 64, 512), (33, 49, 513), (128, 64, 1100), (5, 64, 15), (128, 1, 31)]


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("engine") / "emu_engine_check")
    from paper_1507_04789_gb300 import build
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, os.path.join(ROOT, "tests", "emu_engine_check.cu"),
                    "-o", out], check=True)
    return out


def operand(rng, n, K, kind):
    x = rng.standard_normal((n, K))
    if kind == 1:                                # rows and columns of very different size, zeros
        x *= 2.0 ** rng.integers(-30, 30, (n, 1)) * 2.0 ** rng.integers(-30, 1, (1, K))
        x[rng.random((n, K)) < 0.1] = 0.0
        x[0] = 0.0
    if kind == 2:                                # digits at their limits: powers of two and their neighbours
        x = rng.choice([1.0, -1.0, np.nextafter(2.0, 1.0), -np.nextafter(2.0, 1.0), 1.0 + 2.0 ** -9, 0.5], (n, K))
    return x


@pytest.mark.parametrize("kind", [0, 1, 2])
def test_products(exe, kind):
    rng = np.random.default_rng(17 + kind)
    cases, data = [], b""
    for na, nb, K in SHAPES:
        for la, lb, tab in ((0, 0, 1), (1, 2, 0), (2, 2, 1), (2, 1, 0)):
            A, B = operand(rng, na, K, kind), operand(rng, nb, K, kind)
            cases.append((A, B))
            data += np.array([na, nb, K, la, lb, tab], dtype=np.int32).tobytes() + A.tobytes() + B.tobytes()
    res = subprocess.run([exe], input=data, capture_output=True, timeout=300)
    assert res.returncode == 0, (res.returncode, res.stderr)
    out, pos, worst, rms = np.frombuffer(res.stdout), 0, 0.0, 0.0
    for A, B in cases:
        na, K = A.shape
        nb = B.shape[0]
        got = out[pos:pos + na * nb].reshape(na, nb)
        pos += na * nb
        Al, Bl = A.astype(np.longdouble), B.astype(np.longdouble)
        err = np.abs((got - np.einsum("ik,jk->ij", Al, Bl)).astype(np.float64))
        absum = np.abs(A) @ np.abs(B).T
        bound = 2.0 ** -44 * absum
        for k in range(0, K, 128):
            ma, mb = np.abs(A[:, k:k + 128]).max(1), np.abs(B[:, k:k + 128]).max(1)
            ea, eb = (np.where(m > 0, 2.0 ** np.frexp(m)[1], 0.0) for m in (ma, mb))
            bound += 2.0 ** -46.5 * min(128, K - k) * ea[:, None] * eb[None, :]
        assert (err <= bound).all(), (A.shape, B.shape, (err / np.maximum(bound, 1e-300)).max())
        rel = err / np.maximum(absum, 1e-300)
        worst, rms = max(worst, rel.max()), max(rms, np.sqrt((rel ** 2).mean()))
    assert pos == out.size
    print(f"kind {kind}: max error / sum |ab| {worst:.2e}, largest rms of a product {rms:.2e}")
