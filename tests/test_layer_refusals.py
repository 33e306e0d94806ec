"""What layer.py refuses on the host, before anything is launched (no device is needed to see it)."""
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
