"""The greedy of Step 3 with groups beside the warp that reads ahead of it: orders of
many 32s in which nearly nothing is eligible (the greedy overtakes the reader), all
is, or only a stretch is."""
import numpy as np
import pytest

import oracle
from gpu_helpers import compare_factor, cuda_ok, vb
from test_gpu_sweeps import _matrix

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("share", [0.002, 0.3, 1.0])
@pytest.mark.parametrize("nb", [33, 2048, 6001])
def test_orders_of_few_and_many_eligible_supernodes(nb, share):
    m = _matrix(1, 2, nb, 3, seed=nb)
    Am = oracle.VBMat(m[0], m[0], *m[1:])
    w = oracle.Prec(Am, 1, 1e-3, 6, gs=4).vec(0, "w")
    tol = float(np.quantile(w, 1.0 - share)) if share < 1.0 else 0.0
    P = vb().vbarms_factor(vb().vbarms_vbsr_from_blocks(*m), 1, 1e-3, 6, group_size=4, ddtol=tol)
    Po = oracle.Prec(Am, 1, 1e-3, 6, gs=4, ddtol=tol)
    if Po.levels:
        assert np.array_equal(P.vector(0, "gptr"), Po.gptr(0))
    compare_factor(P, Po)
