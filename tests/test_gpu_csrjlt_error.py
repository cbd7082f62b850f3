"""csrjlt (Alg. 4) in FP32: the error of long sums against 64 bits, and slices of
every size."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from oracle import gaussian as oga

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,nz,m", [(500_000, 32, 1, 400), (300_000, 17, 2, 200), (200_000, 200, 4, 400),
                                      (150_000, 64, 3, 64)])
def test_error_of_long_sums(n, d, nz, m):
    """nz entries of +-1 a row, so that C's entries are sums of draws; the first
    eight rows of G in 64 bits.  An FP32 draw is off by up to 1.5 x 2^-24 in the
    mean.  A chain of L FP32 additions, whose sum grows as a random walk, is off by
    2^-24 x 0.3 sqrt(L) of it (a rounding 0.29 ulp, an ulp 0.72 x 2^-23 in the mean);
    L: the nonzeros of a column within a partial, of which there are as many as
    160 KB an SM hold, with some 1,000 rows each or more."""
    import paper_2203_02798_gb300 as lsk
    rng = np.random.default_rng(n)
    J = rng.integers(0, d, size=n * nz).astype(np.int32)
    V = rng.choice(np.array([-1.0, 1.0], dtype=np.float32), size=n * nz)
    I = np.arange(n + 1, dtype=np.int64) * nz
    C = lsk.csrjlt(lsk.csr_from_numpy(V, J, I, d), m, 21, "fp32").cpu().numpy().astype(np.float64)[:8]
    rows = np.repeat(np.arange(n), nz)
    want = np.zeros((8, d))
    for i in range(0, n, 100_000):
        G = oga.gaussian_columns(8, i, min(n, i + 100_000), 21, oga.PREC_FP32, oga.STREAM_JLT) * np.sqrt(8 / m)
        blk = slice(i * nz, min(n, i + 100_000) * nz)
        for j in range(8):
            want[j] += np.bincount(J[blk], weights=V[blk] * G[j, rows[blk] - i], minlength=d)
    L = n * nz / (d * min(n // 1024, 152 * (160 << 10) // (d * m * 4)))
    assert np.linalg.norm(C - want) <= 2.0 ** -24 * np.sqrt(2.25 + 0.11 * L) * np.linalg.norm(want)


@pytest.mark.parametrize("d,m", [(120, 60), (128, 221), (256, 73), (1100, 8)])
def test_first_call_of_a_process(d, m):
    """Slices of C just below 48 KB, as the first call of a process (a larger one
    before it would have raised the kernel's limit)."""
    code = f"""
import numpy as np, paper_2203_02798_gb300 as lsk
from oracle import gaussian as oga
n, d, m = 3000, {d}, {m}
rng = np.random.default_rng(d)
J = rng.integers(0, d, size=n).astype(np.int32)
V = rng.standard_normal(n).astype(np.float32)
C = lsk.csrjlt(lsk.csr_from_numpy(V, J, np.arange(n + 1, dtype=np.int64), d), m, 3, "fp32").cpu().numpy()
G = oga.gaussian_columns(m, 0, n, 3, oga.PREC_FP32, oga.STREAM_JLT)
A = np.zeros((n, d))
A[np.arange(n), J] = V
assert np.linalg.norm(C - G @ A) <= 1e-6 * np.linalg.norm(G @ A)
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    p = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stderr[-2000:]
