"""pevlm_layer_forward and pevlm_rope_qkv against the separate calls: bit for bit where the arithmetic is the same (RoPE,
caches, video rows), within the question's summation order elsewhere; and a batch in one launch against its sequences."""
import numpy as np
import pytest

from paper_2506_19651_b200 import inputs
from helpers import gpu_shape, to_bits, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,B,N,Q,Hq,Hkv,d,causal", [
    (64, 128, 4, 32, 4, 2, 64, False), (300, 200, 9, 0, 7, 1, 128, False), (0, 0, 0, 45, 8, 2, 128, False),
    (784, 784, 15, 64, 28, 4, 128, False), (100, 300, 3, 1, 4, 4, 128, True), (1, 4000, 1, 130, 14, 2, 64, False)])
def test_one_call_equals_the_separate_calls(S, B, N, Q, Hq, Hkv, d, causal):
    import torch
    from paper_2506_19651_b200.layer import LayerBuffers, layer_forward
    w = inputs.Workload("t", S, B, N, Q, Hq, Hkv, d, 1e6, False, 99)
    q, k, v = (to_dev(t) for t in inputs.make_qkv(w))
    s = gpu_shape(w, causal)
    one = layer_forward(LayerBuffers(s), q, k, v)
    many = layer_forward(LayerBuffers(s), q, k, v, mark=lambda name: None)
    torch.cuda.synchronize()
    nv = w.n_video
    for name, rows in (("q_video", nv), ("q_question", Q), ("k_cache", w.L), ("v_cache", w.L), ("o_video", nv)):
        np.testing.assert_array_equal(to_bits(getattr(one, name)[:rows]), to_bits(getattr(many, name)[:rows]), err_msg=name)
    assert torch.equal(one.lse_video[:, :nv], many.lse_video[:, :nv])
    if Q:
        # other key splits: fp32 sums in another order (LSE about 1e-6), a result on the edge may round to its bf16 neighbour
        assert (one.lse_question - many.lse_question).abs().max() <= 1e-5
        a, b = one.o_question.float(), many.o_question.float()
        assert ((a - b).abs() <= 2.0 ** -7 * b.abs() + 2e-3).all()


@pytest.mark.parametrize("n,Hq,Hkv,d,batch", [(1, 28, 4, 128, 1), (77, 4, 2, 64, 3), (3700, 14, 2, 128, 2)])
def test_rope_qkv_equals_rope_and_copy(n, Hq, Hkv, d, batch):
    import torch
    from paper_2506_19651_b200 import binding as pb
    g = torch.Generator(device="cuda").manual_seed(5)
    rnd = lambda h: torch.randn(batch * n, h, d, generator=g, device="cuda").bfloat16()
    q, k, v = rnd(Hq), rnd(Hkv), rnd(Hkv)
    s = pb.make_shape(n, 1, 0, 0, Hq, Hkv, d, theta=1e6, batch=batch)
    outs = [torch.zeros_like(t) for t in (q, k, v)]
    pb.pevlm_rope_qkv(s, q, k, v, *outs, 31, n)
    s.batch = 1
    for b in range(batch):  # positions start again with every sequence
        i = slice(b * n, (b + 1) * n)
        qo, ko = torch.empty_like(q[i]), torch.empty_like(k[i])
        pb.pevlm_rope_qk(s, q[i], k[i], qo, ko, 31, n)
        for got, want in ((outs[0][i], qo), (outs[1][i], ko), (outs[2][i], v[i])):
            np.testing.assert_array_equal(to_bits(got), to_bits(want))


def test_batch_in_one_launch_equals_its_sequences():
    import torch
    from paper_2506_19651_b200 import binding as pb
    S, B, N, Q, Hq, Hkv, d, batch = 200, 300, 3, 21, 7, 1, 128, 5
    g = torch.Generator(device="cuda").manual_seed(6)
    nv, L = S + N * B, S + N * B + Q
    q = torch.randn(batch, nv, Hq, d, generator=g, device="cuda").bfloat16()
    qq = torch.randn(batch, Q, Hq, d, generator=g, device="cuda").bfloat16()
    k, v = (torch.randn(batch, L, Hkv, d, generator=g, device="cuda").bfloat16() for _ in range(2))
    kv, vv = k[:, :nv].contiguous(), v[:, :nv].contiguous()

    def run(shape, q, kv, vv, qq, k, v):
        n = shape.batch
        o, lse = torch.empty_like(q), torch.empty(n, Hq, nv, device="cuda")
        oq, lq = torch.empty_like(qq), torch.empty(n, Hq, Q, device="cuda")
        ws = [torch.zeros(pb.pevlm_workspace_bytes(shape, i), dtype=torch.uint8, device="cuda") for i in (0, 1)]
        pb.pevlm_parallel_prefill_attn(shape, q, kv, vv, o, lse, ws[0])
        pb.pevlm_query_attn(shape, qq, k, v, oq, lq, ws[1])
        torch.cuda.synchronize()
        assert pb.pevlm_read_status(ws[0])[0] == 0 and pb.pevlm_read_status(ws[1])[0] == 0
        return o, lse, oq, lq
    make = lambda n: pb.make_shape(S, B, N, Q, Hq, Hkv, d, batch=n)
    together = run(make(batch), q, kv, vv, qq, k, v)
    for b in range(batch):
        for x, y in zip(together, run(make(1), *(t[b:b + 1].contiguous() for t in (q, kv, vv, qq, k, v)))):
            assert torch.equal(x[b:b + 1], y)
