"""Arguments of a wrong type: every call raises what the conversion of the first bad argument raised, before it launches
anything (no device is needed to see it)."""
import ctypes as C

import pytest

from paper_2506_19651_b200 import binding as pb


class Tensor:
    """Something with an address, as the calls look at it."""
    nbytes = 1 << 20

    def __init__(self, at=4096):
        self.at = at

    def data_ptr(self):
        return self.at


@pytest.fixture
def s(monkeypatch):
    monkeypatch.setattr(pb, "_stream", lambda: 0)
    return pb.make_shape(64, 128, 4, 32, 4, 2, 64)


def calls(s):
    """Every launching call as (function, arguments behind the shape); a bad alignment keeps each from launching."""
    t, odd = Tensor(), Tensor(4098)
    return [(pb.pevlm_rope_qk, [odd, t, t, t, 0, 4]), (pb.pevlm_rope_qkv, [odd, t, t, t, t, t, 0, 4]),
            (pb.pevlm_rope_qk_mrope, [odd, t, t, t, 4, t, (8, 12, 12)]), (pb.pevlm_parallel_prefill_attn, [odd, t, t, t, t, t]),
            (pb.pevlm_block_attn, [odd, t, t, 64, 576, t, t, t]), (pb.pevlm_assemble_kv, [odd, t, t, t, t, t]),
            (pb.pevlm_query_attn, [odd, t, t, t, t, t]), (pb.pevlm_query_attn_noalloc, [odd, t, t, t, t]),
            (pb.pevlm_layer_forward, [odd] + [t] * 12)]


def test_all_calls_reach_the_checks(s):
    for f, args in calls(s):
        with pytest.raises(pb.PevlmError) as e:
            f(s, *args)
        assert e.value.code == pb.PEVLM_EALIGN, f.__name__


def test_a_wrong_type_in_any_place(s):
    for f, args in calls(s):
        for i, a in enumerate(args):
            if isinstance(a, tuple):
                continue
            wrong = args[:i] + ["x"] + args[i + 1:]
            with pytest.raises(TypeError if isinstance(a, int) else AttributeError, match="'str' object"):
                f(s, *wrong)


def test_an_exception_of_a_tensor_comes_through(s):
    class Gone(Tensor):
        def data_ptr(self):
            raise RuntimeError("storage is gone")
    t = Tensor()
    with pytest.raises(RuntimeError, match="storage is gone"):
        pb.pevlm_rope_qk(s, Gone(), t, t, t, 0, 4)


def test_fewer_than_three_sections(s):
    # those that are not given are empty, as in a C array; the alignment of q_in is looked at before their sum
    t = Tensor()
    for sections, code in (((32,), pb.PEVLM_EALIGN), ([8, 24], pb.PEVLM_EALIGN), ((), pb.PEVLM_EALIGN)):
        with pytest.raises(pb.PevlmError) as e:
            pb.pevlm_rope_qk_mrope(s, Tensor(4098), t, t, t, 4, t, sections)
        assert e.value.code == code
    with pytest.raises(pb.PevlmError) as e:
        pb.pevlm_rope_qk_mrope(s, t, t, t, t, 4, t, (8, 23))
    assert e.value.code == pb.PEVLM_EINVAL
    with pytest.raises((TypeError, IndexError)):
        pb.pevlm_rope_qk_mrope(s, t, t, t, t, 4, t, (8, 12, 12, 0))


def test_a_shape_is_a_shape(s):
    class Other(C.Structure):
        _fields_ = [("batch", C.c_int32)]

    class Mine(pb.Shape):
        pass
    for f, args in calls(s):
        for bad in (Other(1), C.c_int32(1), C.pointer(s), None, 4096):  # what ctypes refuses for a pevlm_shape_t*
            with pytest.raises((C.ArgumentError, TypeError)):
                f(bad, *args)
        with pytest.raises(pb.PevlmError) as e:
            f(Mine(*(getattr(s, n) for n, _ in pb.Shape._fields_)), *args)
        assert e.value.code == pb.PEVLM_EALIGN
