"""What layer.py refuses on the host, before anything is launched, and what it returns (no device is needed to see it)."""
import pytest

from paper_2506_19651_b200 import binding as pb
from paper_2506_19651_b200 import layer


@pytest.fixture
def no_calls(monkeypatch):
    """The library's launching calls, recorded instead of made."""
    made = []
    monkeypatch.setattr(pb, "_native", lambda: pytest.fail("a call was made"))
    for name in ("pevlm_layer_forward", "pevlm_rope_qk", "pevlm_rope_qkv", "pevlm_assemble_kv", "pevlm_parallel_prefill_attn",
                 "pevlm_block_attn", "pevlm_query_attn"):
        monkeypatch.setattr(pb, name, lambda *a, _n=name, **k: made.append(_n))
    return made


@pytest.mark.parametrize("mark", [None, lambda name: None])
def test_layer_pass_is_one_sequence(no_calls, mark):
    import torch
    one, two = (pb.make_shape(16, 32, 2, 8, 4, 2, 64, batch=b) for b in (1, 2))
    t = torch.zeros(2 * one.L, 4, 64, dtype=torch.bfloat16)
    buf = layer.LayerBuffers(one, device="cpu")
    layer.layer_forward(buf, t, t, t, mark=mark)
    assert no_calls
    with pytest.raises(ValueError, match="one sequence"):
        layer.LayerBuffers(two, device="cpu")
    no_calls.clear()
    buf.shape = two  # buffers of one sequence, a shape of two
    with pytest.raises(ValueError, match="one sequence"):
        layer.layer_forward(buf, t, t, t, mark=mark)
    assert not no_calls


def test_streaming_window_takes_only_rows_that_fit(no_calls):
    import torch
    S, B, W, Q_max = 8, 16, 2, 4
    win = layer.StreamingWindow(S, B, W, Q_max, 4, 2, 64, 1e4, device="cpu")
    rows = lambda n: [torch.zeros(n, h, 64, dtype=torch.bfloat16) for h in (4, 2, 2)]
    short = lambda n, i: [t[:-1] if j == i else t for j, t in enumerate(rows(n))]
    for i in range(3):
        with pytest.raises(ValueError, match="rows"):
            win.set_sink(*short(S, i))
        with pytest.raises(ValueError, match="rows"):
            win.append_block(*short(B, i))
        if i:
            with pytest.raises(ValueError, match="rows"):
                win.ask(*short(3, i))
    assert not no_calls and win.blocks_seen == 0
    win.set_sink(*rows(S))
    win.append_block(*rows(B))
    win.ask(*rows(B))  # one block of two: the question has the other's room too
    win.append_block(*rows(B))
    win.ask(*rows(Q_max))
    no_calls.clear()
    for n in (Q_max + 1, B + 1):  # past the end of the caches; of the roped question too
        with pytest.raises(ValueError, match="rows"):
            win.ask(*rows(n))
    assert not no_calls
    win.append_block(*rows(B + 5))  # rows past the block's are not looked at
    assert no_calls and win.blocks_seen == 3


@pytest.mark.parametrize("Q", [0, 5])
def test_ragged_pass_names_a_workspace_for_each_part(no_calls, Q):
    import torch
    L = 8 + 16 + 7 + Q
    t = [torch.zeros(L, h, 64, dtype=torch.bfloat16) for h in (4, 2, 2)]
    full, last, question = layer.ragged_layer_forward(*t, 8, 16, 2, 7, Q, 1e4)[4]  # of the full blocks, the last one, the question
    shape = pb.make_shape(8, 16, 2, Q, 4, 2, 64)
    assert full.numel() == last.numel() == pb.pevlm_workspace_bytes(shape, pb.WS_PREFILL)
    assert question.numel() == pb.pevlm_workspace_bytes(shape, pb.WS_QUERY)


def test_nothing_to_do_is_no_error(no_calls):
    import torch
    empty = pb.make_shape(0, 16, 0, 0, 4, 2, 64)
    buf = layer.LayerBuffers(empty, device="cpu")
    t = torch.zeros(0, 4, 64, dtype=torch.bfloat16)
    for mark in (None, lambda name: None):
        assert layer.layer_forward(buf, t, t, t, mark=mark) is buf
    assert not no_calls
