"""Steps that read what the step before them has just written, back to back over reused buffers with other inputs each time:
the kernels overlap at their ends, and none may read what a buffer held before."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,Hkv,d,batch", [(1, 4, 128, 1), (40, 2, 64, 3), (300, 4, 128, 2), (5000, 4, 128, 1)])
def test_copy_of_what_rope_has_just_written(n, Hkv, d, batch):
    import torch
    from paper_2506_19651_b200 import binding as pb
    rounds = 24
    g = torch.Generator(device="cuda").manual_seed(8)
    rows = batch * n
    k, v = (torch.randn(rounds, rows, Hkv, d, generator=g, device="cuda").bfloat16() for _ in range(2))
    s = pb.make_shape(n, 1, 0, 0, Hkv, Hkv, d, theta=1e6, batch=batch)
    roped = torch.zeros(rows, Hkv, d, dtype=torch.bfloat16, device="cuda")
    caches = torch.zeros(2, rounds, rows, Hkv, d, dtype=torch.bfloat16, device="cuda")
    want = torch.empty_like(k)
    for i in range(rounds):
        pb.pevlm_rope_qk(s, None, k[i], None, want[i], 0, n)
    torch.cuda.synchronize()
    for again in range(8):
        caches.zero_()
        for i in range(rounds):
            pb.pevlm_rope_qk(s, None, k[i], None, roped, 0, n)
            pb.pevlm_assemble_kv(s, roped, v[i], None, None, caches[0, i], caches[1, i])
        assert torch.equal(caches[0], want) and torch.equal(caches[1], v)
