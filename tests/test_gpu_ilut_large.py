"""The last-level block ILUT on pivot blocks of more than 32 rows: factored on chip
beside a row in global memory, or in global memory; permutations of up to and more
than 64 and 128 places in cycles of every length."""
import numpy as np
import pytest

import oracle
from gpu_helpers import compare_factor, cuda_ok, vb
from test_gpu_sweeps import _matrix

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]

SIZES = [(31, 34), (40, 44), (50, 56), (63, 65), (100, 104), (126, 131)]


@pytest.mark.parametrize("lo,hi", SIZES)
def test_fp64_random_pivot_blocks(lo, hi):
    """Diagonal blocks without any dominance of their own: every row moves."""
    m = list(_matrix(lo, hi, 9, 2, seed=lo))
    bsz, bptr, bcol, voff, val = m
    rng = np.random.default_rng(hi)
    for i in range(9):
        b = int(bptr[i] + np.searchsorted(bcol[bptr[i]:bptr[i + 1]], i))
        val[voff[b]:voff[b + 1]] = rng.standard_normal(bsz[i] * bsz[i]) * 10.0
    V = vb()
    A = V.vbarms_vbsr_from_blocks(*m)
    Am = oracle.VBMat(m[0], m[0], *m[1:])
    for t, lfil in ((0.0, -1), (1e-4, 1)):
        Po = oracle.Prec(Am, 0, t, lfil)
        piv = Po.vec(0, "piv")
        assert (piv[: int(bsz[0])] != np.arange(bsz[0])).sum() > bsz[0] // 2
        compare_factor(V.vbarms_factor(A, 0, t, lfil), Po)


@pytest.mark.parametrize("lo,hi", SIZES)
def test_mixed_factors_close(lo, hi):
    m = _matrix(lo, hi, 9, 2, seed=20 + lo)
    P = vb().vbarms_factor(vb().vbarms_vbsr_from_blocks(*m), 0, 0.0, -1, precision="fp32")
    Po = oracle.Prec(oracle.VBMat(m[0], m[0], *m[1:]), 0, 0.0, -1)
    # u = 2^-24: the no-drop factors of a dominant matrix, |dLU| <= 3 n u |L||U|
    for w in ("L", "U", "D"):
        g, o = P.export(0, w), Po.mat(0, w)
        assert np.linalg.norm(g["val"] - o.val) <= 3 * int(m[0].sum()) * 2.0 ** -24 * np.linalg.norm(o.val), w
    assert np.array_equal(P.vector(0, "piv"), Po.vec(0, "piv"))
    assert np.array_equal(P.vector(0, "ptag")[m[0] > 32], np.ones((m[0] > 32).sum()))
