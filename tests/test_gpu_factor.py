"""Panel Cholesky and triangular inverse in shared memory, single and block-diagonal.

Orders around the panel width (4), empty and one-row blocks, the largest order
(128), both thread counts, stacked storage, and a matrix that is not positive
definite.  Bounds: the computed factor satisfies |L L' - A| <= (n + 1) u |L| |L'|
and the computed inverse |X L - I| <= n u |X| |L| entrywise (Higham, "Accuracy
and Stability of Numerical Algorithms", Theorems 10.3 and 8.5, u = 2^-53); twice
that covers the products formed here.
"""
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
BLOCKS = [(1,), (3,), (4,), (5,), (16,), (49,), (64,), (127,), (128,), (64, 64), (17, 1, 30), (30, 34, 0, 22), (0, 3),
          (32, 32, 32, 32), (25, 25, 25)]


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    from paper_1507_04789_gb300 import build
    out = str(tmp_path_factory.mktemp("factor") / "factor_check")
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, os.path.join(ROOT, "tests", "factor_check.cu"),
                    "-o", out], check=True)
    return out


def matrix(rng, lens):
    n = sum(lens)
    A, s = np.zeros((n, n)), 0
    for m in lens:
        x = rng.random((m, 2))
        d = np.sqrt(((x[:, None] - x[None]) ** 2).sum(2))
        A[s:s + m, s:s + m] = np.exp(-d / 0.3) + 0.02 * np.eye(m)
        s += m
    return A


def call(exe, jobs):
    data = b"".join(np.array([len(l), stk, th, *l, *[0] * (4 - len(l))], dtype=np.int32).tobytes() + A.tobytes()
                    for l, stk, th, A in jobs)
    res = subprocess.run([exe], input=data, capture_output=True, timeout=120)
    assert res.returncode == 0, res.returncode
    out, pos = [], 0
    for l, _, _, A in jobs:
        n = A.shape[0]
        a = np.frombuffer(res.stdout, count=2 * n * n, offset=pos).reshape(2, n, n)
        pos += 16 * n * n
        out.append((a[0], a[1], int(np.frombuffer(res.stdout, dtype=np.int32, count=1, offset=pos)[0])))
        pos += 4
    assert pos == len(res.stdout)
    return out


def test_factor_and_inverse(exe):
    rng = np.random.default_rng(5)
    jobs = []
    for l in BLOCKS:
        A = matrix(rng, l)
        for th in (256, 512):
            jobs.append((l, 0, th, A))
            if len(l) > 1:
                jobs.append((l, 1, th, A))
    u = 2.0 ** -53
    for (l, stk, th, A), (L, X, bad) in zip(jobs, call(exe, jobs)):
        n = A.shape[0]
        assert bad == 0
        Ll, Xl = L.astype(np.longdouble), X.astype(np.longdouble)
        r1, b1 = np.abs(Ll @ Ll.T - A), (n + 1) * u * (np.abs(L) @ np.abs(L).T)
        r2, b2 = np.abs(Xl @ Ll - np.eye(n)), n * u * (np.abs(X) @ np.abs(L))
        assert (r1 <= 2 * b1).all() and (r2 <= 2 * b2).all(), (l, stk, th)


def test_not_positive_definite_is_flagged(exe):
    rng = np.random.default_rng(6)
    jobs = []
    for l, row in (((64,), 20), ((5, 9, 33, 40), 13), ((16,), 0)):
        A = matrix(rng, l)
        A[row, row] = -2.0
        jobs.append((l, 0, 256, A))
    for (l, _, _, A), (L, X, bad) in zip(jobs, call(exe, jobs)):
        assert bad == 1 and np.isfinite(L).all() and np.isfinite(X).all()
