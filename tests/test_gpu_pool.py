"""The library's device memory pool: what it keeps is bounded and given back, and
several threads on their own streams get their own results."""
import gc
import threading

import numpy as np
import pytest

from gpu_helpers import cuda_ok, gpu_compress, torch, vb
from paper_1508_02219_gb300 import synth

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]


def test_memory_is_given_back_after_the_last_handle():
    V = vb()
    gc.collect()
    torch.cuda.synchronize()
    m = synth.geometric(40000, 6, seed=1)
    free0, total = torch.cuda.mem_get_info()
    A = gpu_compress(m, 0.8)
    P = V.vbarms_factor(A, 2, 1e-3, 20)
    del P
    torch.cuda.synchronize()
    assert free0 - torch.cuda.mem_get_info()[0] <= total // 8 + A.query()["nval"] * 8 + (1 << 30)
    del A
    gc.collect()
    torch.cuda.synchronize()
    # a 256th of the device, and what the CUDA context itself took meanwhile
    assert free0 - torch.cuda.mem_get_info()[0] <= total // 256 + (256 << 20)


def test_threads_on_their_own_streams():
    V = vb()
    mats = [synth.geometric(1500 + 400 * k, 4 + k % 3, seed=30 + k) for k in range(4)]
    xs = [np.random.default_rng(k).standard_normal(m.n) for k, m in enumerate(mats)]

    def work(k, stream, out):
        m = mats[k]
        for _ in range(3):
            with torch.cuda.stream(stream):
                x = torch.from_numpy(xs[k]).cuda()
                y = torch.zeros_like(x)
                stream.synchronize()
                A = V.vbarms_compress(m.n, m.rowptr, m.colind, m.val, 0.8, stream=stream)
                P = V.vbarms_factor(A, 2, 1e-3, 20, precision="fp32")
                V.vbarms_apply(P, x, y)
                stream.synchronize()
                out[k].append(y.cpu().numpy())
            del P, A

    alone = [[] for _ in mats]
    for k in range(4):
        work(k, torch.cuda.Stream(), alone)
    together = [[] for _ in mats]
    threads = [threading.Thread(target=work, args=(k, torch.cuda.Stream(), together)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for k in range(4):
        assert len(together[k]) == 3
        for y in together[k] + alone[k]:
            assert np.array_equal(y, alone[k][0])
