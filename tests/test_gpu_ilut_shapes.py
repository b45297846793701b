"""The last-level block ILUT at the sizes where it changes path: pivot blocks of
1-8, 9-16, 17-32 and more rows, multipliers taken in chunks of rows, records
larger than one and than both stage buffers, working rows that outgrow the
on-chip workspace, lfil cuts in registers and by radix selection, equal norms,
equal pivots, and FP64 pivot blocks inside a mixed factor."""
import numpy as np
import pytest

import oracle
from gpu_helpers import compare_factor, cuda_ok, torch, vb
from test_gpu_sweeps import CASES, _matrix

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]


def _factors(m, t, lfil, precision, nlev=0):
    V = vb()
    P = V.vbarms_factor(V.vbarms_vbsr_from_blocks(*m), nlev, t, lfil, precision=precision)
    return V, P, oracle.Prec(oracle.VBMat(m[0], m[0], *m[1:]), nlev, t, lfil)


@pytest.mark.parametrize("t,lfil", [(0.0, -1), (2e-4, -1), (1e-4, 4)])
@pytest.mark.parametrize("name", CASES)
def test_fp64_factors_bit_exact(name, t, lfil):
    _, P, Po = _factors(_matrix(*CASES[name], seed=40 + sorted(CASES).index(name)), t, lfil, "fp64")
    compare_factor(P, Po)


@pytest.mark.parametrize("name", CASES)
def test_mixed_factors_close(name):
    m = _matrix(*CASES[name], seed=60 + sorted(CASES).index(name))
    V, P, Po = _factors(m, 0.0, -1, "fp32")
    n = int(m[0].sum())
    # u = 2^-24: the no-drop factors of a dominant matrix, |dLU| <= 3 n u |L||U|
    for w in ("L", "U", "D"):
        g, o = P.export(0, w), Po.mat(0, w)
        assert np.array_equal(g["bcol"], o.bcol) and np.array_equal(g["voff"], o.voff)
        assert np.linalg.norm(g["val"] - o.val) <= 3 * n * 2.0 ** -24 * np.linalg.norm(o.val), w
    assert np.array_equal(P.vector(0, "piv"), Po.vec(0, "piv"))


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 6, 7, 8, 9])
def test_mixed_factors_of_one_block_size(n):
    m = _matrix(n, n, 30, 6, seed=90 + n)
    V, P, Po = _factors(m, 0.0, -1, "fp32")
    # the bound of the test above
    for w in ("L", "U", "D"):
        g, o = P.export(0, w), Po.mat(0, w)
        assert np.linalg.norm(g["val"] - o.val) <= 3 * 30 * n * 2.0 ** -24 * np.linalg.norm(o.val), w
    assert np.array_equal(P.vector(0, "piv"), Po.vec(0, "piv"))


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nb,band,lfil", [(420, 190, 12), (700, 340, 9)])
def test_lfil_cuts_of_many_candidates(nb, band, lfil, precision):
    """More than 64 and more than 256 candidates a row; small whole values make
    equal norms, which the lower column wins."""
    m = list(_matrix(1, 2, nb, band, seed=5))
    rng = np.random.default_rng(6)
    m[4] = np.where(np.abs(m[4]) < 1.0, rng.integers(-2, 3, m[4].size) * 0.0625, m[4])
    V, P, Po = _factors(tuple(m), 0.0, lfil, precision)
    if precision == "fp64":
        compare_factor(P, Po)
    else:
        for w in ("L", "U"):
            counts = np.diff(P.export(0, w)["bptr"])
            assert np.array_equal(counts, np.diff(Po.mat(0, w).bptr)) and counts.max() == lfil


def test_equal_pivots_and_tagged_blocks():
    """Blocks whose pivot column holds equal magnitudes take the first row, as
    the oracle does; blocks whose condition exceeds the threshold keep an FP64
    pivot in the mixed factor and the others do not."""
    m = list(_matrix(2, 24, 60, 3, seed=9))
    bsz, bptr, bcol, voff, val = m
    ill = np.arange(60) % 4 == 1
    for i in range(60):
        b = int(bptr[i] + np.searchsorted(bcol[bptr[i]:bptr[i + 1]], i))
        d = val[voff[b]:voff[b + 1]].reshape(bsz[i], bsz[i])
        if ill[i]:
            d[-1] = d[0] * (1.0 + 1e-6)
            d[-1, -1] += 1e-5 * np.abs(d[0]).max()
        else:
            d[:] = np.where(np.arange(bsz[i])[:, None] >= np.arange(bsz[i]), 1.0, 0.0) * 40.0 + np.eye(bsz[i])
            d[:, 0] = 40.0
    V, P, Po = _factors(tuple(m), 0.0, -1, "fp64")
    compare_factor(P, Po)
    Pm = V.vbarms_factor(V.vbarms_vbsr_from_blocks(*m), 0, 0.0, -1, precision="fp32")
    # the condition of every block as it was factored, from the FP64 factors; the
    # FP32 estimate is within kappa 2^-24 n of it, far less than the factor two
    tags, D, piv = Pm.vector(0, "ptag"), Po.mat(0, "D"), Po.vec(0, "piv")
    off = np.concatenate([[0], np.cumsum(bsz)])
    for i in range(60):
        n = int(bsz[i])
        lu = D.val[D.voff[i]:D.voff[i + 1]].reshape(n, n)
        a = (np.tril(lu, -1) + np.eye(n)) @ np.triu(lu)
        for k in range(n - 1, -1, -1):
            a[[k, piv[off[i] + k]]] = a[[piv[off[i] + k], k]]
        kappa = np.linalg.cond(a, 1)
        assert tags[i] == 1 if kappa > 2e4 else tags[i] == 0 or kappa > 5e3, (i, n, kappa)
    assert tags.any() and not tags.all()
    x = np.random.default_rng(3).standard_normal(int(bsz.sum()))
    y = torch.zeros(len(x), dtype=torch.float64, device="cuda")
    V.vbarms_apply(Pm, torch.from_numpy(x).cuda(), y)
    assert np.isfinite(y.cpu().numpy()).all()
