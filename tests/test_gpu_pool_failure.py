"""A call that fails gives back the memory that its handle held."""
import gc

import numpy as np
import pytest

from gpu_helpers import cuda_ok, torch, vb

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]


def test_memory_is_given_back_when_no_handle_comes_of_a_call():
    V = vb()
    gc.collect()
    n, total = 20_000, torch.cuda.mem_get_info()[1]
    per_row = int(total / 128 / 12 / n)  # 12 bytes an entry: a 128th of the device
    rowptr = np.arange(n + 1, dtype=np.int64) * per_row
    colind, val = np.zeros(n * per_row, np.int32), np.zeros(n * per_row)
    with pytest.raises(V.VbarmsError):  # a small one first: the context and the kernels
        V.vbarms_compress(4, np.arange(5, dtype=np.int64) * 2, np.zeros(8, np.int32), np.zeros(8), 0.8)
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    with pytest.raises(V.VbarmsError) as e:
        V.vbarms_compress(n, rowptr, colind, val, 0.8)  # columns not ascending
    assert e.value.status == V.VB_EINVAL
    torch.cuda.synchronize()
    # a 256th of the device, and a page of what the driver maps at once
    assert free0 - torch.cuda.mem_get_info()[0] <= total // 256 + (64 << 20)
