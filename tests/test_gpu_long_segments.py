"""Sinks and shorter last blocks whose pairs are handed out one by one (more than four query tiles, few items) and as whole lists
(four tiles, or 16 items and more for every SM): lengths on both sides of the lines, odd numbers of query tiles.  Against the
fp64 oracle, with guard bytes around every buffer; tolerances as in helpers.py."""
import numpy as np
import pytest

from oracle import api as oracle
from paper_2506_19651_b200 import inputs
from helpers import LSE_TOL, O_TOL, GuardedAllocator, bits_to_f64, to_bits, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,B,N,B_last,Q,Hq,Hkv,d", [
    (512, 600, 2, 512, 3, 7, 1, 128),    # four tiles: whole lists
    (513, 600, 2, 513, 3, 7, 1, 128),    # five tiles, the last of one row
    (641, 700, 2, 650, 5, 5, 1, 128),    # six tiles of five heads: the last pair has one tile
    (1000, 900, 2, 777, 2, 3, 3, 64),    # groups of one head: two tiles of different lengths in a pair
    (9216, 64, 1, 33, 1, 64, 64, 64),    # 72 tiles of 64 kv heads: 2,304 items, under 16 for each of 148 SMs
    (9217, 64, 1, 33, 1, 64, 64, 64),    # 73 tiles: 2,368 items, whole lists again
])
def test_rows(S, B, N, B_last, Q, Hq, Hkv, d):
    import torch
    from paper_2506_19651_b200 import binding as pb
    from paper_2506_19651_b200.layer import ragged_layer_forward
    w = inputs.Workload("t", S, B, N, Q, Hq, Hkv, d, 1e6, True, S + B_last, B_last=B_last)
    q, k, v = inputs.make_qkv(w)
    guard = GuardedAllocator()
    o_v, lse_v, o_q, lse_q, ws = ragged_layer_forward(to_dev(q), to_dev(k), to_dev(v), S, B, N, B_last, Q, w.theta, alloc=guard)
    torch.cuda.synchronize()
    for one in ws:
        assert pb.pevlm_read_status(one)[0] == 0
    guard.check()
    sh = oracle.make_shape(S, B, N, Q, Hq, Hkv, d, B_last=B_last)
    rows = np.arange(w.L) if w.L <= 3000 else np.unique(np.concatenate([np.random.default_rng(9).integers(0, w.L, size=150), [S - 1, S, w.L - 1]]))
    o, lse = oracle.attn_rows(sh, oracle.rope(q, w.theta), oracle.rope(k, w.theta), v, rows)
    o_gpu = np.concatenate([bits_to_f64(to_bits(o_v)), bits_to_f64(to_bits(o_q))])[rows]
    lse_gpu = np.concatenate([lse_v.double().cpu().numpy().T, lse_q.double().cpu().numpy().T])[rows]
    assert np.abs(o_gpu - o).max() <= O_TOL
    assert np.abs(lse_gpu - lse).max() <= LSE_TOL
    assert np.isfinite(lse_v.cpu().numpy()).all()   # every row of every head was written
