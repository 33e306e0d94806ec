"""RoPE in groups of every size that the launch picks (1 to 4 tokens, with few heads up to 8): bit for bit against the oracle, V
copied along, with groups that lie across the end of a sequence and a last one that is not full."""
import numpy as np
import pytest

from oracle import api as oracle
from helpers import to_bits, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Hq,Hkv,d,batch,n", [
    (28, 4, 128, 1, 444), (28, 4, 128, 1, 620), (28, 4, 128, 2, 650), (28, 4, 128, 1, 2501), (28, 4, 128, 5, 701), (28, 4, 128, 1, 7105),  # 1, 2, 3, 3, 4, 4
    (32, 8, 64, 3, 433), (14, 2, 128, 1, 888), (14, 2, 128, 2, 651), (14, 2, 128, 1, 2501), (14, 2, 128, 7, 715), (14, 2, 128, 1, 7001),  # 3; 1, 2, 4, 6, 8
    (4, 2, 64, 1, 1), (4, 2, 64, 3, 33), (4, 2, 64, 1, 5001)])  # 4, 4, 8
def test_bits(Hq, Hkv, d, batch, n):
    import torch
    from paper_2506_19651_b200 import binding as pb
    rng = np.random.default_rng(n + Hq)
    draw = lambda h: (rng.standard_normal((batch * n, h, d)).astype(np.float32).view(np.uint32) >> 16).astype(np.uint16)
    q, k, v = draw(Hq), draw(Hkv), draw(Hkv)
    dev = [to_dev(t) for t in (q, k, v)]
    outs = [torch.zeros_like(t) for t in dev]
    pb.pevlm_rope_qkv(pb.make_shape(n, 1, 0, 0, Hq, Hkv, d, theta=1e6, batch=batch), *dev, *outs, 77, n)
    for x, o in ((q, outs[0]), (k, outs[1])):
        want = np.concatenate([oracle.rope(x[b * n:(b + 1) * n], 1e6, first_pos=77) for b in range(batch)])
        # the device's and the C library's sine may differ in the last place and the value then sits on a rounding boundary
        # (about 2^-27 an element): none expected, one allowed where a million elements and more are looked at
        assert int((to_bits(o) != want).sum()) <= (x.size > 1 << 20)
    np.testing.assert_array_equal(to_bits(outs[2]), v)
