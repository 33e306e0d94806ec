"""Question rows whose keys are not split (the attention kernel writes the result, no merge), on both sides of the length at
which the splits begin, against float64 arithmetic on the same inputs."""
import pytest

from helpers import LSE_TOL, O_TOL

pytestmark = pytest.mark.gpu


def _expected(q, k, v, scale):
    """Rows of q are the last ones of the causal mask over k, v: (o [Q,Hq,d], lse [Hq,Q])."""
    import torch
    Q, Hq, _ = q.shape
    L, Hkv, _ = k.shape
    kk, vv = (t.double().repeat_interleave(Hq // Hkv, dim=1) for t in (k, v))
    s = torch.einsum("qhd,khd->hqk", q.double(), kk) * scale
    i = torch.arange(L, device=q.device)
    s = s.masked_fill(i[None, None, :] > (L - Q + torch.arange(Q, device=q.device))[None, :, None], float("-inf"))
    return torch.einsum("hqk,khd->qhd", torch.softmax(s, -1), vv), torch.logsumexp(s, -1)


@pytest.mark.parametrize("nv,Q,Hq,Hkv,d,batch", [
    (448, 64, 8, 2, 128, 1), (449, 64, 8, 2, 128, 3), (30, 97, 4, 4, 64, 2), (0, 45, 7, 1, 128, 1), (300, 130, 28, 4, 64, 2)])
def test_query_attn(nv, Q, Hq, Hkv, d, batch):
    import torch
    from paper_2506_19651_b200 import binding as pb
    g = torch.Generator(device="cuda").manual_seed(7)
    L = nv + Q
    q = torch.randn(batch * Q, Hq, d, generator=g, device="cuda").bfloat16()
    k, v = (torch.randn(batch * L, Hkv, d, generator=g, device="cuda").bfloat16() for _ in range(2))
    s = pb.make_shape(nv, 1, 0, Q, Hq, Hkv, d, theta=1e6, batch=batch)
    ws = torch.zeros(pb.pevlm_workspace_bytes(s, pb.WS_QUERY), dtype=torch.uint8, device="cuda")
    o = torch.full((batch * Q + 1, Hq, d), 7.0, dtype=torch.bfloat16, device="cuda")
    lse = torch.full((batch * Hq * Q + 1,), 7.0, dtype=torch.float32, device="cuda")
    pb.pevlm_query_attn(s, q, k, v, o, lse, ws)
    again = torch.empty_like(o)
    pb.pevlm_query_attn(s, q, k, v, again, None, ws)
    assert pb.pevlm_read_status(ws)[0] == 0
    assert (o[batch * Q] == 7).all() and lse[-1] == 7  # nothing past the last row
    assert torch.equal(o[:batch * Q], again[:batch * Q])
    for b in range(batch):
        want_o, want_lse = _expected(q[b * Q:(b + 1) * Q], k[b * L:(b + 1) * L], v[b * L:(b + 1) * L], d ** -0.5)
        assert (o[b * Q:(b + 1) * Q].double() - want_o).abs().max() <= O_TOL
        assert (lse[b * Hq * Q:(b + 1) * Hq * Q].view(Hq, Q).double() - want_lse).abs().max() <= LSE_TOL


# key tiles of the question against those of the longest prefill item, which decide whether the keys are split
@pytest.mark.parametrize("S,B,N,Q,Hq,Hkv,d", [
    (128, 128, 4, 128, 8, 2, 128), (128, 128, 5, 1, 8, 2, 128), (256, 0, 0, 300, 4, 2, 64), (0, 1500, 1, 20, 7, 1, 128),
    (700, 100, 1, 256, 28, 4, 128)])
def test_layer(S, B, N, Q, Hq, Hkv, d):
    import torch
    from paper_2506_19651_b200 import binding as pb
    from paper_2506_19651_b200.layer import LayerBuffers, layer_forward
    g = torch.Generator(device="cuda").manual_seed(8)
    s = pb.make_shape(S, max(B, 1), N, Q, Hq, Hkv, d, theta=1e6)
    L = s.n_video + Q
    q = torch.randn(L, Hq, d, generator=g, device="cuda").bfloat16()
    k, v = (torch.randn(L, Hkv, d, generator=g, device="cuda").bfloat16() for _ in range(2))
    buf = layer_forward(LayerBuffers(s), q, k, v)
    assert pb.pevlm_read_status(buf.ws_query)[0] == 0
    want_o, want_lse = _expected(buf.q_question[:Q], buf.k_cache, buf.v_cache, d ** -0.5)
    assert (buf.o_question[:Q].double() - want_o).abs().max() <= O_TOL
    assert (buf.lse_question[:, :Q].double() - want_lse).abs().max() <= LSE_TOL
