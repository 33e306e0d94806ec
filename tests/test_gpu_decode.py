"""pevlm_query_attn with at most 32 rows per kv head (the streaming decode kernel) and one row more (the tile kernel), against
fp64 on the same bf16 inputs: key counts around the 16-key pieces and the 128-key rounds of a CTA, every row count's edge,
both head sizes, batches, more (kv head, sequence) pairs than SMs, outliers that move the reference maximum late."""
import math

import pytest

from helpers import LSE_TOL, O_TOL

pytestmark = pytest.mark.gpu


def reference(q, k, v, nv):
    """q [Q, Hq, d], k, v [L, Hkv, d] on the GPU; fp64."""
    import torch
    Q, Hq, d = q.shape
    G = Hq // k.shape[1]
    kk, vv = (t.double().repeat_interleave(G, dim=1).transpose(0, 1) for t in (k, v))     # [Hq, L, d]
    s = q.double().transpose(0, 1) @ kk.transpose(1, 2) / math.sqrt(d)                    # [Hq, Q, L]
    hidden = torch.arange(k.shape[0], device=q.device)[None] > nv + torch.arange(Q, device=q.device)[:, None]
    s = s.masked_fill(hidden, -math.inf)
    lse = torch.logsumexp(s, -1)
    return (torch.exp(s - lse[..., None]) @ vv).transpose(0, 1), lse


@pytest.mark.parametrize("nv,Q,Hq,Hkv,d,batch,outlier", [
    (0, 1, 1, 1, 128, 1, False), (0, 16, 1, 1, 64, 1, False), (14, 2, 7, 1, 128, 1, False), (15, 1, 16, 1, 64, 1, False),
    (127, 1, 28, 4, 128, 1, False), (128, 2, 28, 4, 128, 2, True), (1000, 3, 28, 4, 128, 1, False),
    (4095, 4, 8, 2, 128, 1, True), (4096, 17, 2, 2, 64, 1, True), (5000, 8, 4, 2, 64, 3, True), (50176, 1, 28, 4, 128, 1, True),
    (300, 1, 160, 160, 64, 1, False), (700, 16, 3, 3, 128, 60, False),
    (900, 4, 28, 4, 128, 2, True), (1500, 32, 2, 2, 64, 1, True), (2000, 33, 1, 1, 128, 1, False)])
def test_few_rows_match_fp64(nv, Q, Hq, Hkv, d, batch, outlier):
    import torch
    from paper_2506_19651_b200 import binding as pb
    g = torch.Generator(device="cuda").manual_seed(nv + Q)
    rnd = lambda n, h: torch.randn(batch, n, h, d, generator=g, device="cuda")
    L = nv + Q
    q, k, v = rnd(Q, Hq), rnd(L, Hkv), rnd(L, Hkv)
    if outlier:  # the largest score of a row jumps several times, late in the cache too
        for row, f in ((0, 8.0), (L // 3, 16.0), (L - 20, 24.0), (L - 1, 32.0)):
            k[:, row] *= f
    q, k, v = (t.bfloat16() for t in (q, k, v))
    s = pb.make_shape(nv, 1, 0, Q, Hq, Hkv, d, batch=batch)
    o, lse = torch.full_like(q, float("nan")), torch.full((batch, Hq, Q), float("nan"), device="cuda")
    ws = torch.full((pb.pevlm_workspace_bytes(s, pb.WS_QUERY) + 512,), 0xA5, dtype=torch.uint8, device="cuda")  # any contents
    pb.pevlm_query_attn(s, q, k, v, o, lse, ws[:-512])
    torch.cuda.synchronize()
    assert pb.pevlm_read_status(ws)[0] == 0
    assert bool((ws[-512:] == 0xA5).all())
    for b in range(batch):
        ro, rl = reference(q[b], k[b], v[b], nv)
        assert (o[b].double() - ro).abs().max() <= O_TOL
        assert (lse[b].double() - rl).abs().max() <= LSE_TOL
