"""Products with a block matrix at the block sizes where they change path: blocks all
of one size (a plain loop up to 7 columns), of up to, exactly and more than 8
columns, and of mixed sizes."""
import numpy as np
import pytest

import oracle
from gpu_helpers import cuda_ok, torch, vb
from test_gpu_sweeps import _matrix

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]

SIZES = [(s, s) for s in (1, 2, 5, 6, 7, 8, 9, 15, 16, 17, 33)] + [(1, 7), (1, 9), (6, 8), (7, 24)]


@pytest.mark.parametrize("lo,hi", SIZES)
def test_matrix_times_vector(lo, hi):
    """One step of GMRES(1) without a preconditioner: x = b (Ab, b) / (Ab, Ab)."""
    V = vb()
    bsz, bptr, bcol, voff, val = m = _matrix(lo, hi, 45, 4, seed=lo + hi)
    n, off = int(bsz.sum()), np.concatenate([[0], np.cumsum(bsz)])
    a = np.zeros((n, n))
    for i in range(45):
        for b in range(bptr[i], bptr[i + 1]):
            j = bcol[b]
            a[off[i]:off[i + 1], off[j]:off[j + 1]] = val[voff[b]:voff[b + 1]].reshape(bsz[i], bsz[j])
    b = np.random.default_rng(1).standard_normal(n)
    ab = a @ b
    x = torch.zeros(n, dtype=torch.float64, device="cuda")
    V.fgmres_solve(V.vbarms_vbsr_from_blocks(*m), None, torch.from_numpy(b).cuda(), x, rtol=0.0, restart=1, maxit=1)
    # products and sums of n terms each way, u = 2^-53, and the step's few operations
    tol = 8 * n * 2.0 ** -53 * np.linalg.norm(np.abs(a) @ np.abs(b)) / np.linalg.norm(ab)
    xo = b * (ab @ b) / (ab @ ab)
    assert np.linalg.norm(x.cpu().numpy() - xo) <= tol * np.linalg.norm(xo)


@pytest.mark.parametrize("lo,hi", SIZES)
def test_level_products(lo, hi):
    """G and W of one reduction level."""
    V = vb()
    m = _matrix(lo, hi, 45, 4, seed=50 + lo + hi)
    x = np.random.default_rng(2).standard_normal(int(m[0].sum()))
    yo = oracle.Prec(oracle.VBMat(m[0], m[0], *m[1:]), 1, 0.0, -1).apply(x)
    xd = torch.from_numpy(x).cuda()
    y = torch.zeros_like(xd)
    # FP64: the solve's parity bound; FP32: 9 n u, u = 2^-24, for these dominant matrices
    for precision, tol in (("fp64", 1e-12), ("fp32", 9 * len(x) * 2.0 ** -24)):
        V.vbarms_apply(V.vbarms_factor(V.vbarms_vbsr_from_blocks(*m), 1, 0.0, -1, precision=precision), xd, y)
        assert np.linalg.norm(y.cpu().numpy() - yo) <= tol * np.linalg.norm(yo), precision
