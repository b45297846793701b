"""The time limit of a device wait in the triangular sweeps covers one wait: a row
whose dependencies keep arriving may take longer than the limit altogether."""
import numpy as np
import pytest

from gpu_helpers import cuda_ok, torch, vb

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]

NB, HUB = 1100, 8


def _chain(ni):
    """Row i depends on row i - 1 and on every HUB-th row before it, so that each row
    takes something new every HUB links of the chain; all rows of the forward sweep
    are in flight at once."""
    rng = np.random.default_rng(ni)
    bptr, bcol = [0], []
    for i in range(NB):
        bcol.extend(sorted({k for k in range(0, i, HUB)} | ({i - 1} if i else set()) | {i}))
        bptr.append(len(bcol))
    bptr, bcol = np.array(bptr, np.int64), np.array(bcol, np.int32)
    val = rng.standard_normal((len(bcol), ni, ni)) * (0.1 / ni)
    rows = np.repeat(np.arange(NB), np.diff(bptr))
    val[rows == bcol] += 2.0 * np.eye(ni)
    return (np.full(NB, ni, np.int32), bptr, bcol, np.arange(len(bcol) + 1, dtype=np.int64) * ni * ni, val.ravel())


@pytest.mark.parametrize("ni", [6, 14, 18])
def test_a_row_that_progresses_does_not_time_out(ni):
    V = vb()
    A = V.vbarms_vbsr_from_blocks(*_chain(ni))
    x = torch.from_numpy(np.random.default_rng(1).standard_normal(NB * ni)).cuda()
    y, z = torch.zeros_like(x), torch.zeros_like(x)
    P = V.vbarms_factor(A, 0, 0.0, -1)
    ms = []
    for _ in range(4):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        V.vbarms_apply(P, x, y)
        e1.record()
        torch.cuda.synchronize()
        ms.append(e0.elapsed_time(e1))
    # a third of what the sweep of the chain takes, some 350 links; a wait takes at most HUB
    Q = V.vbarms_factor(A, 0, 0.0, -1, wait_limit=int(min(ms) * 1e6 / 3))
    V.vbarms_apply(Q, x, z)
    assert torch.equal(y, z)
