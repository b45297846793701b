"""Step 1's overlap counts at the sizes where they change path: columns of up to
and more than 256 rows (sorted lists or not), rows whose candidates outgrow the
on-chip table, cosines at and next to tau."""
import numpy as np
import pytest

import oracle
from gpu_helpers import as_dict, compare_vb, cuda_ok, gpu_compress
from paper_1508_02219_gb300 import synth

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]


def _check(a, tau):
    m = synth.from_dense(a)
    c = oracle.compress(m.n, m.rowptr, m.colind, m.val, tau)
    A = gpu_compress(m, tau)
    g = A.export()
    assert np.array_equal(g["perm"], c.perm) and np.array_equal(g["bsz"], c.bsz)
    compare_vb(dict(rsz=g["bsz"], csz=g["bsz"], **{k: g[k] for k in ("bptr", "bcol", "voff", "val")}), as_dict(c.A),
               "VBCSR")


@pytest.mark.parametrize("tall", [1, 31, 33, 255, 256, 257, 600])
@pytest.mark.parametrize("tau", [0.7, 1.0])
def test_column_lengths(tall, tau):
    """Some columns hold `tall` rows, the others few; n = 900 also makes rows of
    more than 640 candidates."""
    n = 900
    rng = np.random.default_rng(tall)
    a = np.where(rng.random((n, n)) < 0.006, rng.standard_normal((n, n)), 0.0)
    for c in rng.choice(n, 12, replace=False):
        a[:, c] = 0.0
        a[rng.choice(n, tall, replace=False), c] = 1.0
    a[::3] = a[1::3]  # equal rows
    a[np.arange(n), np.arange(n)] = 4.0
    _check(a, tau)


@pytest.mark.parametrize("tau", [0.5, 0.6, 0.75, 0.8, np.sqrt(0.5), 1.0])
def test_cosines_at_tau(tau):
    """Rows of 1 to 40 columns nested in one another: overlaps c with c^2 equal
    to, just below and just above tau^2 |P_i| |P_j|."""
    n = 120
    a = np.zeros((n, n))
    for i in range(n):
        a[i, : 1 + i % 40] = 1.0 + i
        if i % 5 == 0:
            a[i, 60 + i % 7] = 2.0
    _check(a, float(tau))
