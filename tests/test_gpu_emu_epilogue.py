"""Rows of the FP64-emulation engine's products as its kernels write them.

Every row and column of ragged tiles, strides and offsets of every alignment
(rows of one warp then differ in theirs), the product stored and subtracted, by
the inlined helpers and by the call, in global and in shared memory; whatever
lies around and between the rows stays as it was.  Bounds of the values as in
test_gpu_emu_engine.py, plus the subtraction's rounding; the exponents are those
of the rows written.
"""
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
GUARD, POISON = 4096, -1.2345678901234567e+250

# na, nb, K
SHAPES = [(1, 1, 1), (31, 16, 16), (33, 17, 40), (64, 32, 64), (70, 49, 70), (97, 63, 98), (127, 64, 130), (128, 64, 448)]


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("epilogue") / "emu_epilogue_check")
    from paper_1507_04789_gb300 import build
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, os.path.join(ROOT, "tests", "emu_epilogue_check.cu"),
                    "-o", out], check=True)
    return out


@pytest.mark.parametrize("form", ["inlined", "call", "call, shared"])
def test_rows(exe, form):
    form = ["inlined", "call", "call, shared"].index(form)
    rng = np.random.default_rng(29 + form)
    cases, data = [], b""
    for na, nb, K in SHAPES:
        for pad in (0, 1, 2, 3, 4):
            for off in (0, 1, 2, 3):
                sub, xe0 = int(rng.integers(2)), int(rng.integers(0, nb))
                gcol = int(rng.integers(0, 257 - nb))
                A, B = rng.standard_normal((na, K)), rng.standard_normal((nb, K))
                C = rng.standard_normal((na, nb)) * np.sqrt(K)
                cases.append((A, B, C, nb + pad, off, sub, xe0, gcol))
                data += np.array([na, nb, K, nb + pad, off, sub, form, xe0, gcol], dtype=np.int32).tobytes()
                data += A.tobytes() + B.tobytes() + C.tobytes()
    res = subprocess.run([exe], input=data, capture_output=True, timeout=300)
    assert res.returncode == 0, (res.returncode, res.stderr)
    pos = 0
    for A, B, C, ldo, off, sub, xe0, gcol in cases:
        (na, K), nb = A.shape, B.shape[0]
        size = 2 * GUARD + 4 + na * ldo
        buf = np.frombuffer(res.stdout, count=size, offset=pos)
        pos += 8 * size
        xe = np.frombuffer(res.stdout, dtype=np.int32, count=384, offset=pos).reshape(3, 128)
        pos += 4 * 384
        what = (A.shape, B.shape, ldo, off, sub)
        rows = buf[GUARD + off:GUARD + off + na * ldo].reshape(na, ldo)
        got = rows[:, :nb]
        want = np.einsum("ik,jk->ij", A.astype(np.longdouble), B.astype(np.longdouble))
        bound = 2.0 ** -44 * (np.abs(A) @ np.abs(B).T)
        for k in range(0, K, 128):
            ea, eb = (2.0 ** np.frexp(np.abs(X[:, k:k + 128]).max(1))[1] for X in (A, B))
            bound += 2.0 ** -46.5 * min(128, K - k) * ea[:, None] * eb[None, :]
        if sub:
            want = C - want
            bound += 2.0 ** -52 * np.abs(want).astype(np.float64)
        err = np.abs((got - want).astype(np.float64))
        assert (err <= bound).all(), (what, np.argwhere(~(err <= bound))[:8])
        assert (rows[:, nb:] == POISON).all(), what
        assert (buf[:GUARD + off] == POISON).all() and (buf[GUARD + off + na * ldo:] == POISON).all(), what
        if form:
            e = np.where(got != 0.0, np.frexp(got)[1], -2000)
            group = (gcol + np.arange(nb)) // 128
            for table, cols in ((xe[0], np.arange(nb) >= xe0), (xe[1], group == 0), (xe[2], group == 1)):
                ref = np.full(128, -2000)
                if cols.any():
                    ref[:na] = e[:, cols].max(1)
                np.testing.assert_array_equal(table, ref, err_msg=str(what))
    assert pos == len(res.stdout)
