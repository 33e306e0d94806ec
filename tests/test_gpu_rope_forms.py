"""RoPE with few heads and with many (two forms of the kernel), at the sizes where a group of tokens, a CTA's share or the form
changes: bit for bit against the oracle, V copied along."""
import numpy as np
import pytest

from oracle import api as oracle
from helpers import to_bits, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Hq,Hkv,d", [(1, 1, 128), (16, 2, 128), (17, 1, 128), (18, 1, 128), (19, 1, 128), (18, 1, 64), (19, 1, 64), (2, 1, 64)])
@pytest.mark.parametrize("n", [1, 887, 889, 1775, 5329, 12000])
def test_bits(Hq, Hkv, d, n):
    import torch
    from paper_2506_19651_b200 import binding as pb
    rng = np.random.default_rng(n + Hq)
    draw = lambda h: (rng.standard_normal((n, h, d)).astype(np.float32).view(np.uint32) >> 16).astype(np.uint16)
    q, k, v = draw(Hq), draw(Hkv), draw(Hkv)
    dev = [to_dev(t) for t in (q, k, v)]
    outs = [torch.zeros_like(t) for t in dev]
    pb.pevlm_rope_qkv(pb.make_shape(n, 1, 0, 0, Hq, Hkv, d, theta=1e6), *dev, *outs, 77, n)
    wrong = [int((to_bits(o) != oracle.rope(t, 1e6, first_pos=77)).sum()) for o, t in zip(outs[:2], (q, k))]
    # the device's and the C library's sine may differ in the last place and the value then sits on a rounding boundary
    # (about 2^-27 an element): none expected, one allowed where a million elements and more are looked at
    assert wrong[0] <= (q.size > 1 << 20) and wrong[1] == 0
    np.testing.assert_array_equal(to_bits(outs[2]), v)
