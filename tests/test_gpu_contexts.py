"""The library in a second context on the same device, in a process of its own: kernel attributes and the addresses of device
arrays belong to a context."""
import subprocess
import sys
import os

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import ctypes as C
from paper_2506_19651_b200 import binding as pb
cu, lib = C.CDLL("libcuda.so.1"), pb.lib()
def ok(rc): assert rc == 0, (rc, lib.pevlm_last_cuda_error())
def filled(n, bits):
    p = C.c_uint64()
    ok(cu.cuMemAlloc_v2(C.byref(p), C.c_size_t(2 * n)))
    ok(cu.cuMemsetD16_v2(p, C.c_ushort(bits), C.c_size_t(n)))
    return C.c_void_p(p.value)
def run():
    one, n = 0x3F80, 740
    s = pb.make_shape(300, 200, 2, 40, 8, 2, 128)
    q, k, v, o, oq = filled(8 * 128 * n, one), filled(2 * 128 * n, one), filled(2 * 128 * n, one), filled(8 * 128 * n, 0), filled(8 * 128 * 40, 0)
    ws, b = filled(1 << 22, 0), C.byref(s)
    ok(lib.pevlm_rope_qk(b, q, k, q, k, 0, n, None, None))
    ok(lib.pevlm_parallel_prefill_attn(b, q, k, v, o, None, ws, 1 << 23, None))
    for Q in (40, 1):  # the tile kernel, the decode kernel; both with a merge
        s.sink_len = n - 400 - Q
        s.query_len = Q
        ok(lib.pevlm_query_attn(b, q, k, v, oq, None, ws, 1 << 23, None))
    ok(lib.pevlm_query_attn_noalloc(b, q, k, v, oq, None, None))  # partials in the context's own copy of the built-in array
    ok(cu.cuCtxSynchronize())
    status = C.c_int32(1)
    ok(lib.pevlm_read_status(None, None, C.byref(status), None))
    assert status.value == 0
    got = (C.c_uint16 * (8 * 128 * 700))()
    ok(cu.cuMemcpyDtoH_v2(got, o, C.c_size_t(2 * len(got))))
    assert set(got) == {one}  # averages of ones
dev, first, second = C.c_int(), C.c_void_p(), C.c_void_p()
ok(cu.cuInit(0)); ok(cu.cuDeviceGet(C.byref(dev), 0))
ok(cu.cuDevicePrimaryCtxRetain(C.byref(first), dev)); ok(cu.cuCtxSetCurrent(first))
run()
ok(cu.cuCtxCreate_v2(C.byref(second), 0, dev))
run()
ok(cu.cuCtxSetCurrent(first))
run()
print("both contexts")
"""


@pytest.mark.gpu
def test_second_context():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "both contexts" in r.stdout, r.stdout + r.stderr
