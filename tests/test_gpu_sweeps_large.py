"""The last level's triangular sweeps on block rows of more than 16 scalars whose
1 025 to 1 536 values take the whole on-chip space of a warp: pivot blocks of more
than 32 rows, and FP64 pivot blocks of 17 to 32 rows in a mixed factor."""
import numpy as np
import pytest

import oracle
from gpu_helpers import cuda_ok, vb
from test_gpu_sweeps import _apply, _matrix

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]


def _check(lo, hi, nb, band, seed, precision, **opt):
    m = _matrix(lo, hi, nb, band, seed=seed)
    V = vb()
    P = V.vbarms_factor(V.vbarms_vbsr_from_blocks(*m), 0, 0.0, -1, precision=precision, **opt)
    for w in ("L", "U"):
        o = P.export(0, w)
        nv = np.diff(o["voff"][o["bptr"]])
        assert ((nv > 1024) & (nv <= 1536)).sum() >= nb // 2, w
    n = int(m[0].sum())
    x = np.random.default_rng(seed).standard_normal(n)
    yo = oracle.Prec(oracle.VBMat(m[0], m[0], *m[1:]), 0, 0.0, -1).apply(x)
    y = _apply(V, P, x)
    # FP64: the solve's parity bound.  FP32 factor and solve: 3 n u |L||U| each
    # way, |A^-1||L||U| <= 3 on these dominant matrices, u = 2^-24
    tol = 1e-12 if precision == "fp64" else 9 * n * 2.0 ** -24
    assert np.linalg.norm(y - yo) <= tol * np.linalg.norm(yo)
    return P


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("lo,hi", [(33, 33), (33, 38), (38, 39)])
def test_pivot_blocks_of_more_than_32_rows(lo, hi, precision):
    for seed in range(4):
        _check(lo, hi, 24, 1, seed, precision)


@pytest.mark.parametrize("lo,hi,band", [(17, 18, 4), (20, 21, 3), (24, 27, 2)])
def test_fp64_pivot_blocks_of_17_to_32_rows_in_a_mixed_factor(lo, hi, band):
    for seed in range(4):
        P = _check(lo, hi, 40, band, seed, "fp32", fp64_pivot_cond=1.0)
        assert P.vector(0, "ptag").all()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("lo,hi,band", [(17, 18, 4), (20, 21, 3), (24, 27, 2)])
def test_rows_of_17_to_32_scalars(lo, hi, band, precision):
    """The pivot block's own space lies right behind the values."""
    _check(lo, hi, 40, band, 7, precision)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_columns_that_every_lane_loads_again(precision):
    """Dependencies of more than 8 unknowns: the first 8 come from the lane that
    polled them, the others from each lane's own loads."""
    V = vb()
    m = _matrix(17, 40, 30, 5, seed=2)
    P = V.vbarms_factor(V.vbarms_vbsr_from_blocks(*m), 0, 0.0, -1, precision=precision)
    n = int(m[0].sum())
    Po = oracle.Prec(oracle.VBMat(m[0], m[0], *m[1:]), 0, 0.0, -1)
    for k in range(8):
        x = np.random.default_rng(k).standard_normal(n)
        yo = Po.apply(x)
        tol = 1e-12 if precision == "fp64" else 9 * n * 2.0 ** -24
        assert np.linalg.norm(_apply(V, P, x) - yo) <= tol * np.linalg.norm(yo)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("lo,hi", [(33, 33), (63, 65), (95, 98), (120, 128)])
def test_pivot_blocks_of_up_to_128_rows(lo, hi, precision):
    """Blocks of one to four rows a lane, interchanges in every third and in random
    ones."""
    V = vb()
    m = list(_matrix(lo, hi, 8, 1, seed=lo))
    bsz, bptr, bcol, voff, val = m
    rng = np.random.default_rng(hi)
    for i in range(1, 8, 2):
        b = int(bptr[i] + np.searchsorted(bcol[bptr[i]:bptr[i + 1]], i))
        d = val[voff[b]:voff[b + 1]].reshape(bsz[i], bsz[i])
        d[:] = d[rng.permutation(bsz[i])]
    n = int(bsz.sum())
    P = V.vbarms_factor(V.vbarms_vbsr_from_blocks(*m), 0, 0.0, -1, precision=precision)
    x = np.random.default_rng(3).standard_normal(n)
    yo = oracle.Prec(oracle.VBMat(m[0], m[0], *m[1:]), 0, 0.0, -1).apply(x)
    # the bounds above
    tol = 1e-12 if precision == "fp64" else 9 * n * 2.0 ** -24
    assert np.linalg.norm(_apply(V, P, x) - yo) <= tol * np.linalg.norm(yo)
