"""The workspace of a question is enough for shorter questions and caches too (a window that is still filling)."""
import ctypes as C

import pytest

from paper_2506_19651_b200 import binding as pb


@pytest.mark.parametrize("Hq,Hkv,d,keys,Q_max,batch", [
    (28, 4, 128, 6081, 1, 1), (28, 4, 128, 9000, 40, 1), (8, 2, 64, 5000, 70, 3), (4, 4, 64, 3000, 129, 1), (14, 2, 128, 700, 300, 2)])
def test_enough_for_shorter_ones(Hq, Hkv, d, keys, Q_max, batch):
    f = pb.lib().pevlm_query_attn
    most = pb.pevlm_workspace_bytes(pb.make_shape(keys, 1, 0, Q_max, Hq, Hkv, d, batch=batch), pb.WS_QUERY)
    p, ws = C.c_void_p(4096), C.c_void_p(4096 + 16)  # the size is checked before the alignment, which is refused: no launch
    for Q in range(1, Q_max + 1, 1 + Q_max // 40):
        for n in list(range(0, keys + 1, 97)) + [keys]:
            s = pb.make_shape(n, 1, 0, Q, Hq, Hkv, d, batch=batch)
            assert f(C.byref(s), p, p, p, p, None, ws, most, None) == pb.PEVLM_EALIGN, (Q, n)
            # with a prefill part beside it
            if batch == 1 and n > 200:
                s = pb.make_shape(100, (n - 100) // 2, 2, Q, Hq, Hkv, d)
                assert s.L <= keys + Q_max
                assert pb.lib().pevlm_layer_forward(C.byref(s), 0, p, p, p, p, p, p, p, p, None, p, None, ws, 256, ws, most, None) == pb.PEVLM_EALIGN
