"""The sequences of a batch do not see one another: what one of them holds, NaN included, changes no bit of the others, and what
the blocks hold changes no bit of the sink's rows."""
import pytest

pytestmark = pytest.mark.gpu
NAN = float("nan")


@pytest.mark.parametrize("S,B,N,Q,Hq,Hkv,d,causal", [
    (200, 300, 3, 21, 7, 1, 128, False), (65, 129, 2, 40, 8, 2, 64, False), (0, 1000, 1, 3, 4, 2, 128, False),
    (777, 100, 1, 90, 4, 4, 64, False), (100, 211, 3, 1, 8, 2, 128, True)])
def test_a_bad_sequence_stays_alone(S, B, N, Q, Hq, Hkv, d, causal):
    import torch
    from paper_2506_19651_b200 import binding as pb
    batch, nv = 3, S + N * B
    g = torch.Generator(device="cuda").manual_seed(4)
    rnd = lambda n, h: torch.randn(batch, n, h, d, generator=g, device="cuda").bfloat16()
    q, k, v = rnd(nv, Hq), rnd(nv, Hkv), rnd(nv, Hkv)
    qq, kc, vc = rnd(Q, Hq), rnd(nv + Q, Hkv), rnd(nv + Q, Hkv)
    s = pb.make_shape(S, B, N, Q, Hq, Hkv, d, batch=batch, mask_mode=pb.MASK_FULL_CAUSAL if causal else pb.MASK_PEVLM)

    def run():
        o, lse = torch.empty_like(q), torch.empty(batch, Hq, nv, device="cuda")
        oq, lq = torch.empty_like(qq), torch.empty(batch, Hq, Q, device="cuda")
        ws = [torch.zeros(pb.pevlm_workspace_bytes(s, i), dtype=torch.uint8, device="cuda") for i in (0, 1)]
        pb.pevlm_parallel_prefill_attn(s, q, k, v, o, lse, ws[0])
        pb.pevlm_query_attn(s, qq, kc, vc, oq, lq, ws[1])
        torch.cuda.synchronize()
        assert pb.pevlm_read_status(ws[0])[0] == 0 and pb.pevlm_read_status(ws[1])[0] == 0
        return o, lse, oq, lq
    want = run()
    for t in (q, k, v, qq, kc, vc):
        t[1] = NAN
    got = run()
    for b in (0, 2):
        assert all(torch.equal(x[b], y[b]) for x, y in zip(got, want)), b
    if S and not causal:
        for t in (k, v):
            t[0, S:] = NAN  # the blocks of the first sequence
        o, lse = run()[:2]
        assert torch.equal(o[0, :S], want[0][0, :S]) and torch.equal(lse[0, :, :S], want[1][0, :, :S])
