"""The number of kernels that bench.py states for a pass: two, and a merge where the question's keys are split."""
import pytest


@pytest.mark.gpu
@pytest.mark.parametrize("shape,kernels", [((784, 784, 3, 64, 28, 4, 128), 2), ((0, 64, 100, 64, 28, 4, 128), 3), ((64, 128, 2, 0, 4, 2, 64), 2)])
def test_kernels_per_pass(shape, kernels):
    import torch
    import bench
    from paper_2506_19651_b200 import binding as pb
    from paper_2506_19651_b200.layer import LayerBuffers, layer_forward
    s = pb.make_shape(*shape)
    buf = LayerBuffers(s)
    q, k, v = (torch.zeros(s.L, h, s.head_dim, dtype=torch.bfloat16, device="cuda") for h in (s.num_q_heads, s.num_kv_heads, s.num_kv_heads))
    layer_forward(buf, q, k, v)
    assert bench.kernels_per_pass(lambda: layer_forward(buf, q, k, v)) == kernels
