"""The CTA-pair attention kernel at the sizes where its hand-overs can go wrong, against the fp64 oracle: work items of one
to a handful of key tiles (shorter than the look-ahead of QK over PV and than the ring), pairs whose second query tile does
not exist, launches with fewer and with more items than CTA pairs, and a reference maximum that has to move in every key
tile, so that each warpgroup takes it over from the other and rescales.  Tolerances as in helpers.py."""
import numpy as np
import pytest

from paper_2506_19651_b200 import inputs
from helpers import LSE_TOL, O_TOL, check_against_oracle, run_gpu_layer

pytestmark = pytest.mark.gpu


def _check(w, q, k, v):
    res = run_gpu_layer(w, q, k, v)
    errs, _, _ = check_against_oracle(w, q, k, v, res, np.arange(w.L))
    for name, e in errs.items():
        assert e <= (LSE_TOL if "lse" in name else O_TOL), (name, e)


@pytest.mark.parametrize("S,B,N,Q,Hq,Hkv,d", [
    (0, 1, 3, 1, 1, 1, 128),        # one key, one row, one query tile: the pair's second slot is empty
    (0, 16, 200, 3, 1, 1, 64),      # more one-tile items than CTA pairs
    (0, 128, 90, 2, 3, 1, 128),     # odd number of query tiles per block
    (128, 129, 3, 19, 2, 2, 128),   # two heads of their own kv head: tiles of different lengths in one pair
    (383, 257, 2, 130, 7, 1, 64),   # odd tile counts, both warpgroups end items
    (17, 640, 1, 37, 5, 1, 128),
])
def test_short_items_and_lone_tiles(S, B, N, Q, Hq, Hkv, d):
    w = inputs.Workload("t", S, B, N, Q, Hq, Hkv, d, 1e6, False, 77)
    _check(w, *inputs.make_qkv(w))


@pytest.mark.parametrize("d", [64, 128])
def test_reference_maximum_moves_in_every_key_tile(d):
    # key rows growing by a factor of 2 from tile to tile: the largest score of a row grows by far more than 2^8 in each
    w = inputs.Workload("t", 300, 900, 1, 40, 4, 2, d, 1e6, False, 78)
    q, k, v = inputs.make_qkv(w)
    kf = inputs.bf16_bits_to_f32(k)
    kf *= np.float32(2.0) ** (np.arange(w.L) // 128)[:, None, None].astype(np.float32)   # exact in bf16
    _check(w, q, inputs.f32_to_bf16_bits(kf), v)
