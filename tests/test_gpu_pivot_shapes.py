"""The reduction levels' pivot solves at the numbers of blocks where a launch deals
them out differently: one, two, four, eight and 32 to a warp, and a thread for each
block where most are large."""
import numpy as np
import pytest

import oracle
from gpu_helpers import cuda_ok, torch, vb
from test_gpu_sweeps import _matrix

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("lo,hi,nb", [(9, 9, 300), (9, 9, 3000), (9, 9, 6000), (9, 9, 11000), (8, 10, 11000),
                                      (1, 12, 11000), (17, 18, 11000), (1, 9, 70000)])
def test_level_solves(lo, hi, nb):
    V = vb()
    m = _matrix(lo, hi, nb, 1, seed=nb + lo)
    A = V.vbarms_vbsr_from_blocks(*m)
    Po = oracle.Prec(oracle.VBMat(m[0], m[0], *m[1:]), 1, 1e-3, 4)
    x = np.random.default_rng(4).standard_normal(int(m[0].sum()))
    yo = Po.apply(x)
    xd = torch.from_numpy(x).cuda()
    y = torch.zeros_like(xd)
    # FP64: the solve's parity bound; FP32: 9 n u for the rows of a block and of
    # its few neighbours (n = 8 hi), u = 2^-24
    for precision, tol in (("fp64", 1e-12), ("fp32", 9 * 8 * hi * 2.0 ** -24)):
        P = V.vbarms_factor(A, 1, 1e-3, 4, precision=precision)
        V.vbarms_apply(P, xd, y)
        assert np.linalg.norm(y.cpu().numpy() - yo) <= tol * np.linalg.norm(yo), precision
        V.vbarms_apply(P, torch.zeros_like(xd), y)
        assert not y.any(), precision
