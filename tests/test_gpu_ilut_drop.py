"""The drop rule of the FP64 last-level ILUT on blocks that are exactly zero: dropped
for every positive tolerance whose squared threshold is positive, also below the
range of FP32, and kept for tolerance zero."""
import numpy as np
import pytest

import oracle
from gpu_helpers import compare_factor, cuda_ok, vb
from test_gpu_sweeps import _matrix

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("lo,hi", [(1, 6), (9, 20)])
@pytest.mark.parametrize("t", [0.0, 1e-200, 1e-120, 1e-50, 7e-46, 1e-44, 1e-38, 1e-20, 1e-8])
def test_zero_blocks(t, lo, hi):
    bsz, bptr, bcol, voff, val = _matrix(lo, hi, 40, 1, seed=12)
    for i in range(40):
        for b in range(bptr[i], bptr[i + 1]):
            if bcol[b] != i and (i + bcol[b]) % 3 == 0:
                val[voff[b]:voff[b + 1]] = 0.0
    V = vb()
    P = V.vbarms_factor(V.vbarms_vbsr_from_blocks(bsz, bptr, bcol, voff, val), 0, t, -1)
    Po = oracle.Prec(oracle.VBMat(bsz, bsz, bptr, bcol, voff, val), 0, t, -1)
    zeros = sum(not np.any(o.val[o.voff[b]:o.voff[b + 1]])
                for o in (Po.mat(0, "L"), Po.mat(0, "U")) for b in range(len(o.bcol)))
    assert (zeros > 0) == (t * t == 0.0)
    compare_factor(P, Po)
