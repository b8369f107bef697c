"""Edges of single kernels and of the layouts a run gets by default: alignment
remainders, tile edges and the smallest and largest sizes of each path."""
import ctypes as C

import numpy as np
import pytest

import oracle
from paper_2102_05613_gb300 import inputs, sk

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [0, 1, 7, 15])
@pytest.mark.parametrize("chains,N", [(1, 5), (3, 17), (64, 100), (40, 4099)])
def test_start_spin_check_finds_the_first_bad_spin(offset, chains, N):
    # spins in device memory at any alignment: the bytes before the first
    # 16-byte boundary, the body and the remainder are all checked, and the
    # smallest offending index is named
    torch = need_gpu()
    n = chains * N
    inst = sk.Instance(inputs.couplings_pm1(N, 3))
    good = torch.from_numpy(inputs.initial_spins(chains, N, 4).reshape(-1))
    buf = torch.ones(n + 16, dtype=torch.int8, device="cuda")
    run = sk.Run(inst, chains=chains, K=4, seed=2)
    view = buf[offset:offset + n]
    head = min(n, (16 - view.data_ptr() % 16) % 16)
    for at in sorted({0, max(0, head - 1), min(head, n - 1), n // 2, max(head, n - (n - head) % 16 - 1), n - 1}):
        for bad in (0, 2, -2, -128, 127):
            view.copy_(good)
            view[at] = bad
            if at + 3 < n:
                view[at + 3] = 5  # a later one must not be reported instead
            with pytest.raises(sk.SKError) as e:
                run.reset(view)
            assert e.value.status == sk.SK_ERR_INVALID_ARG and f"spin {at} " in str(e.value), (at, bad, str(e.value))
    buf.fill_(3)  # what lies around the spins is not looked at
    view.copy_(good)
    run.reset(view)
    assert np.array_equal(run.state()[0].reshape(-1), good.numpy())
    run.close(); inst.close()
