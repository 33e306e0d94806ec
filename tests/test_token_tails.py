"""Ragged last query tiles packed by tokens (all heads of a kv group, some tokens each) instead of by heads: the count of
tiles, and the rows against float64 arithmetic at the sizes where the form of the packing changes."""
import pytest

from helpers import LSE_TOL, O_TOL


def test_tile_count():
    from paper_2506_19651_b200 import binding as pb
    # 80 = 4 * 18 + 8 rows of 7 heads: 5 tiles, and 2 key tiles each under a sink of one block
    s = pb.make_shape(80, 80, 3, 0, 28, 4, 128)
    assert pb.pevlm_tile_stats(s, pb.WS_PREFILL).tiles == 4 * (5 + 3 * 5 * 2)
    # 176 = 128 + 48: by tokens 3 tiles at the second position, by heads it would be 4 (5 pairs of tiles instead of 6)
    s = pb.make_shape(0, 176, 1, 0, 7, 1, 64)
    assert pb.pevlm_tile_stats(s, pb.WS_PREFILL).tiles == 7 + 3 * 2


@pytest.mark.gpu
@pytest.mark.parametrize("S,B,N,last,Hq,Hkv,d", [
    (80, 80, 3, 0, 28, 4, 128), (176, 208, 2, 0, 14, 2, 64), (300, 127, 5, 65, 7, 1, 128), (65, 1000, 2, 431, 8, 2, 128),
    (48, 239, 3, 100, 3, 1, 64), (90, 72, 4, 49, 128, 1, 64), (0, 255, 2, 0, 12, 1, 128)])
def test_rows(S, B, N, last, Hq, Hkv, d):
    import torch
    from paper_2506_19651_b200 import binding as pb
    from paper_2506_19651_b200.layer import LayerBuffers
    lens = [B] * (N - 1 if last else N) + ([last] if last else [])
    nv = S + sum(lens)
    g = torch.Generator(device="cuda").manual_seed(9)
    q = torch.randn(nv, Hq, d, generator=g, device="cuda").bfloat16()
    k, v = (torch.randn(nv, Hkv, d, generator=g, device="cuda").bfloat16() for _ in range(2))
    s = pb.make_shape(S, B, N, 0, Hq, Hkv, d, theta=1e6)
    buf = LayerBuffers(s)
    o = torch.full((nv + 1, Hq, d), 7.0, dtype=torch.bfloat16, device="cuda")
    lse = torch.full((Hq * nv + 1,), 7.0, dtype=torch.float32, device="cuda")
    pb.pevlm_layer_forward(s, q, k, v, buf.q_video, None, buf.k_cache, buf.v_cache, o, lse, None, None, buf.ws_prefill, buf.ws_query,
                           last_len=last)
    assert pb.pevlm_read_status(buf.ws_prefill)[0] == 0
    assert (o[nv] == 7).all() and lse[-1] == 7  # nothing past the last row
    # visible: the sink, and one's own segment up to oneself
    segment = torch.tensor([0] * S + [i + 1 for i, n in enumerate(lens) for _ in range(n)], device="cuda")
    i = torch.arange(nv, device="cuda")
    seen = (i[None, :] <= i[:, None]) & ((segment[None, :] == 0) | (segment[None, :] == segment[:, None]))
    kk, vv = (t[:nv].double().repeat_interleave(Hq // Hkv, dim=1) for t in (buf.k_cache, buf.v_cache))
    x = torch.einsum("qhd,khd->hqk", buf.q_video[:nv].double(), kk) * d ** -0.5
    x = x.masked_fill(~seen[None], float("-inf"))
    assert (o[:nv].double() - torch.einsum("hqk,khd->qhd", torch.softmax(x, -1), vv)).abs().max() <= O_TOL
    assert (lse[:-1].view(Hq, nv).double() - torch.logsumexp(x, -1)).abs().max() <= LSE_TOL
