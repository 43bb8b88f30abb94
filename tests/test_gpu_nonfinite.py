"""Infinities and NaN in x, on every route of the linear layer: they reach their own token's outputs
only; rows that keep the input's group are non-finite; rows that prune it have the value of their
kept groups alone or NaN."""
import numpy as np
import pytest

from paper_2609_33977_gb300 import workload as wl
from tests._gpu_util import to_bits, to_dev

pytestmark = pytest.mark.gpu
AUTO, DECODE, PREFILL, ZERO_FILLED = range(4)
INF, NINF, NAN = 0x7F80, 0xFF80, 0x7FC0

# (out, in, g_out, g_in, T, algo): each kernel with each of its group shapes and stage depths
ROUTES = [
    (520, 1024, 1, 256, 3, DECODE), (520, 1024, 1, 128, 16, DECODE),
    (20480, 1024, 1, 256, 4, AUTO), (5120, 5120, 1, 128, 16, AUTO),         # zero-filled, whole and in parts
    (520, 1152, 1, 128, 40, AUTO), (520, 1024, 1, 256, 100, AUTO),          # zero-filled, 256-deep stages
    (520, 1152, 1, 128, 700, ZERO_FILLED), (520, 1024, 1, 256, 300, AUTO),  # 128-deep
    (520, 1024, 1, 256, 60, PREFILL), (520, 1024, 1, 128, 300, PREFILL),    # gathering
    (512, 1024, 16, 16, 8, AUTO), (512, 1024, 64, 64, 12, AUTO),            # square, few tokens
    (512, 1024, 16, 16, 200, AUTO), (512, 1024, 32, 32, 64, AUTO), (512, 1024, 64, 64, 300, AUTO),
    (512, 1024, 128, 128, 8, AUTO), (512, 1024, 128, 128, 200, AUTO),
]


def f32(bits):
    return (bits.astype(np.uint32) << 16).view(np.float32)


@pytest.mark.parametrize("out,inp,go,gi,T,algo", ROUTES)
def test_nonfinite_inputs(built_lib, out, inp, go, gi, T, algo):
    import torch
    from paper_2609_33977_gb300 import groupsparse as gs
    Wb = wl.random_weight_bits(out, inp, seed=out + T)
    B = wl.random_mask(out // go, inp // gi, 0.5, seed=gi + T).astype(np.uint8)
    B[: max(1, 256 // go), inp // gi // 2] = 0         # a window that keeps nothing of one column of groups
    p = gs.pack_groups(to_dev(Wb), torch.from_numpy(B).cuda(), go, gi)
    xb = wl.random_activation_bits(T, inp, seed=T)
    clean = to_bits(gs.linear(to_dev(xb), p, algo=algo))
    bad = [(0, 5, INF), (T // 2, inp // 2 + 3, NAN), (T - 1, inp - 1, NINF)]
    xs = xb.copy()
    for t, k, v in bad:
        xs[t, k] = v
    y = to_bits(gs.linear(to_dev(xs), p, algo=algo))
    hit = {t for t, _, _ in bad}
    others = [t for t in range(T) if t not in hit]
    assert np.array_equal(y[others], clean[others])    # the other tokens
    keep = np.repeat(B, go, axis=0)
    for t in hit:
        kept = np.any([keep[:, k // gi] for tt, k, _ in bad if tt == t], axis=0)
        assert not np.isfinite(f32(y[t])[kept]).any(), t
        pruned = ~kept
        assert np.all((y[t][pruned] == clean[t][pruned]) | np.isnan(f32(y[t])[pruned])), t
    assert gs.device_status() == gs.GS_OK
