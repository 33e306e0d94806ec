"""A question as long as a prefill needs no more partials than fill the GPU a few times over, on top of one row for each of its
own; and what pevlm_workspace_bytes says is what pevlm_layer_forward takes."""
import ctypes as C

import pytest

from paper_2506_19651_b200 import binding as pb

CASES = [(28, 4, 128, 0, 0, 16384, 65536), (28, 4, 128, 1024, 1024, 262144, 1 << 20), (4, 4, 64, 100, 300, 100000, 300000),
         (32, 8, 128, 1152, 1152, 2000, 74000), (128, 1, 64, 64, 64, 5000, 200000), (1, 1, 128, 0, 4096, 1024, 1 << 21)]


@pytest.mark.parametrize("Hq,Hkv,d,S,B,Q,L", CASES)
def test_bounded_and_enough(Hq, Hkv, d, S, B, Q, L):
    n_blocks = (L - Q - S) // B if B else 0
    s = pb.make_shape(S if B else L - Q, max(B, 1), n_blocks, Q, Hq, Hkv, d)
    n = pb.pevlm_workspace_bytes(s, pb.WS_QUERY)
    row = (d + 1) * 4
    # 16 work items of 256 rows for each of 74 pairs of CTAs
    assert n <= 256 + 256 + (Q * Hq + 16 * 74 * 256) * row, n / (Q * Hq * row)
    p, ws = C.c_void_p(4096), C.c_void_p(4096 + 16)  # the size is checked before the alignment, which is refused: no launch
    last = B // 2
    for last_len in (0, last) if n_blocks else (0,):
        assert pb.lib().pevlm_layer_forward(C.byref(s), last_len, p, p, p, p, p, p, p, p, None, p, None, ws, 256, ws, n, None) == pb.PEVLM_EALIGN
    assert pb.lib().pevlm_query_attn(C.byref(s), p, p, p, p, None, ws, n, None) == pb.PEVLM_EALIGN


@pytest.mark.gpu
@pytest.mark.parametrize("S,B,N,Q,Hq,Hkv,d", [
    (1024, 1024, 31, 8192, 8, 8, 64), (300, 1000, 33, 3001, 12, 6, 128),
    (0, 128, 10240, 1024, 1, 1, 64)])  # 161 splits, more than the merge of few rows has room for
def test_splits_of_a_long_question(S, B, N, Q, Hq, Hkv, d):
    import torch
    from paper_2506_19651_b200.layer import LayerBuffers, layer_forward
    s = pb.make_shape(S, B, N, Q, Hq, Hkv, d, theta=1e6)
    g = torch.Generator(device="cuda").manual_seed(2)
    q, k, v = (torch.randn(s.L, h, d, generator=g, device="cuda").bfloat16() for h in (Hq, Hkv, Hkv))
    one = layer_forward(LayerBuffers(s), q, k, v)
    many = layer_forward(LayerBuffers(s), q, k, v, mark=lambda name: None)  # one piece, or 18
    torch.cuda.synchronize()
    assert pb.pevlm_read_status(one.ws_query)[0] == 0
    assert (one.lse_question - many.lse_question).abs().max() <= 1e-5  # fp32 sums in another order
    a, b = one.o_question.float(), many.o_question.float()
    assert ((a - b).abs() <= 2.0 ** -7 * b.abs() + 2e-3).all()


@pytest.mark.parametrize("Hq,Hkv,d,Q,L,batch", [(56, 8, 128, 2148, 62932, 40), (16, 2, 128, 2683, 105810, 3), (256, 16, 128, 105, 49171, 5)])
def test_a_batch_needs_no_room_for_the_one_call_pass(Hq, Hkv, d, Q, L, batch):
    # pevlm_layer_forward takes one sequence; the question attention of a batch alone has at most 74 items of 256 rows a sequence
    s = pb.make_shape(L - Q, 1, 0, Q, Hq, Hkv, d, batch=batch)
    n = pb.pevlm_workspace_bytes(s, pb.WS_QUERY)
    assert n <= 256 + batch * (256 + (Q * Hq + 74 * 256) * (d + 1) * 4)
    p, ws = C.c_void_p(4096), C.c_void_p(4096 + 16)
    assert pb.lib().pevlm_query_attn(C.byref(s), p, p, p, p, None, ws, n, None) == pb.PEVLM_EALIGN


@pytest.mark.gpu
@pytest.mark.parametrize("n,Q,Hq,Hkv,d,batch", [(9000, 356, 28, 4, 128, 1), (8000, 300, 32, 8, 64, 1), (6100, 130, 14, 2, 64, 3)])
def test_two_waves_of_shorter_items(n, Q, Hq, Hkv, d, batch):
    import torch
    s = pb.make_shape(n, 1, 0, Q, Hq, Hkv, d, batch=batch)
    g = torch.Generator(device="cuda").manual_seed(3)
    q, k, v = (torch.randn(batch, r, h, d, generator=g, device="cuda").bfloat16() for r, h in ((Q, Hq), (n + Q, Hkv), (n + Q, Hkv)))
    o, lse = torch.empty_like(q), torch.empty(batch, Hq, Q, device="cuda")
    size = pb.pevlm_workspace_bytes(s, pb.WS_QUERY)
    ws = torch.full((size + 256,), 165, dtype=torch.uint8, device="cuda")
    pb.pevlm_query_attn(s, q, k, v, o, lse, ws[:size])
    assert pb.pevlm_read_status(ws)[0] == 0 and bool((ws[size:] == 165).all())
    hidden = torch.arange(n + Q, device="cuda")[None, :] > n + torch.arange(Q, device="cuda")[:, None]
    for b in range(batch):
        for h in range(Hq):
            x = (q[b, :, h].double() @ k[b, :, h * Hkv // Hq].double().T * d ** -0.5).masked_fill(hidden, float("-inf"))
            assert (lse[b, h] - torch.logsumexp(x, -1)).abs().max() <= 1e-5  # fp32 sums of some thousand terms
            assert (o[b, :, h].double() - torch.softmax(x, -1) @ v[b, :, h * Hkv // Hq].double()).abs().max() <= 2e-2
