"""vbarms_memory_trim empties the pool while handles live; what they hold stays."""
import numpy as np
import pytest

from gpu_helpers import cuda_ok, gpu_compress, torch, vb
from paper_1508_02219_gb300 import synth

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]


def test_trim_gives_unused_memory_back():
    V = vb()
    m = synth.geometric(40000, 6, seed=1)
    A = gpu_compress(m, 0.8)
    P = V.vbarms_factor(A, 2, 1e-3, 20)
    x = torch.from_numpy(np.random.default_rng(0).standard_normal(m.n)).cuda()
    y, z = torch.zeros_like(x), torch.zeros_like(x)
    V.vbarms_apply(P, x, y)
    V.memory_trim()
    free0 = torch.cuda.mem_get_info()[0]
    V.vbarms_factor(A, 2, 1e-3, 20)  # its memory stays in the pool
    torch.cuda.synchronize()
    assert free0 - torch.cuda.mem_get_info()[0] > 256 << 20
    V.memory_trim(128 << 20)
    # a page of what the driver maps at once beside what is to stay
    assert free0 - torch.cuda.mem_get_info()[0] <= 192 << 20
    V.memory_trim()
    assert free0 - torch.cuda.mem_get_info()[0] <= 64 << 20
    V.vbarms_apply(P, x, z)
    assert torch.equal(y, z)
