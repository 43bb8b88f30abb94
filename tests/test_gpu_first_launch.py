"""A handle's first call on its pack stream, right behind the packing kernels.

The decode and zero-filled kernels read weights before they wait for the launch
before them, so the first launch after packing must be an ordinary one: every
result here is compared with the same call made again.
"""
import numpy as np
import pytest

from paper_2609_33977_gb300 import workload as wl
from tests._gpu_util import to_bits, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("go,gi", [(1, 256), (1, 128), (32, 32), (64, 64)])
@pytest.mark.parametrize("T", [4, 64, 300])
def test_first_call_after_packing(built_lib, go, gi, T):
    import torch
    from paper_2609_33977_gb300 import groupsparse as gs
    out, inp = 5120, 4096
    Ws = [to_dev(wl.random_weight_bits(out, inp, seed=s)) for s in range(3)]
    Ms = [torch.from_numpy(wl.random_mask(out // go, inp // gi, 0.5, seed=9 + s)).cuda() for s in range(3)]
    x = to_dev(wl.random_activation_bits(T, inp, seed=T))
    torch.cuda.synchronize()
    for r in range(4):   # handles come and go, so buffers are used again with other weights
        ps, first = [], []
        for W, M in zip(Ws, Ms):
            ps.append(gs.pack_groups(W, M, go, gi))
            first.append(gs.linear(x, ps[-1]))
        for p, y in zip(ps, first):
            assert np.array_equal(to_bits(y), to_bits(gs.linear(x, p))), (go, gi, T, r)
        del ps, p
    assert gs.device_status() == gs.GS_OK
