"""The fp32 rotation of the RoPE kernel is taken only where it rounds like the fp64 definition: the argument at the kernel
(rope_kernel.cu, rotate2) on values steered at its corners, and subnormal pairs bit for bit on the GPU."""
import numpy as np
import pytest

from oracle import api as oracle

F = np.float32


def _fma(a, b, c):  # the product is exact in 32 bits, the sum rounds to 64 before it rounds to 24
    return (a.astype(np.longdouble) * b.astype(np.longdouble) + c.astype(np.longdouble)).astype(F)


def _bf16(x):
    u = x.view(np.uint32)
    return ((u + 0x7FFF + ((u >> 16) & 1)) >> 16).astype(np.uint16)


def _rotate(a, b, c, s):
    """(r, E, taken, bf16 result, fp64 value) of a c - b s as the kernel forms it; a, b are bf16 values as float32."""
    r = _fma(a, c.astype(F), b * -s.astype(F))
    m = np.abs(a) + np.abs(b)
    e = np.full_like(m, 2.0 ** -23)
    hi, lo = _fma(m, e, r), _fma(m, -e, r)
    taken = (_bf16(hi) == _bf16(lo)) & ~((m > 0) & (m < F(2.0 ** -126)))
    x = a.astype(np.float64) * c - b.astype(np.float64) * s
    return r, m.astype(np.float64) * 2.0 ** -23, taken, _bf16(hi), x


def _angles(rng, n, near_quarter):
    ang = rng.integers(0, 80000, n) * 1e6 ** (-2.0 * rng.integers(0, 64, n) / 128)
    if near_quarter:
        ang = rng.integers(0, 20000, n) * np.pi + np.pi / 2 + rng.uniform(-0.3, 0.3, n)
    return np.cos(ang), np.sin(ang)


def _values(rng, n, emin, emax):
    return ((rng.integers(0, 2, n) << 15 | rng.integers(emin, emax, n) << 7 | rng.integers(0, 128, n)).astype(np.uint32) << 16).view(F)


@pytest.mark.parametrize("kind", ["usual", "sine near one, b just over a power of two, small a", "smallest normal", "subnormal"])
def test_taken_results_are_the_fp64_ones(kind):
    rng = np.random.default_rng(11)
    n = 4_000_000
    if kind == "usual":
        (c, s), a, b = _angles(rng, n, False), _values(rng, n, 120, 130), _values(rng, n, 120, 130)
    elif kind == "smallest normal":
        (c, s), a, b = _angles(rng, n, False), _values(rng, n, 0, 3), _values(rng, n, 0, 3)
    elif kind == "subnormal":
        (c, s), a, b = _angles(rng, n, False), _values(rng, n, 0, 1), _values(rng, n, 0, 1)
    else:
        c, s = _angles(rng, n, True)
        b = ((rng.integers(0, 2, n) << 15 | 127 << 7 | rng.integers(0, 24, n)).astype(np.uint32) << 16).view(F)
        a = _values(rng, n, 110, 126)
    r, E, taken, got, x = _rotate(a, b, c, s)
    want = _bf16(x.astype(F))
    assert np.array_equal(got[taken], want[taken])
    if kind != "subnormal":
        assert taken.mean() > 0.9
    if "normal" not in kind:
        # the error may exceed E, by up to a third, only with |a| + |b| in [1, 1.34) * 2^k; r is then on the grid of 2^(k - 23)
        m = np.abs(a).astype(np.float64) + np.abs(b)
        k, off = np.floor(np.log2(m)), np.abs(x - r)
        over = off > E
        assert (m[over] < 1.34 * 2.0 ** k[over]).all() and (off[over] < 1.34 * 2.0 ** (k[over] - 23)).all()
        assert (np.abs(r[over]) >= 2.0 ** k[over]).all()
        assert over.any() or kind == "usual"


# (a, b as bf16 bits, position, rotary pair) at theta 1e6, d 128: pairs for which an unchecked fp32 rotation rounds the other way
SUBNORMAL = [(0x8001, 0x003a, 75362, 51), (0x0017, 0x800d, 20868, 61), (0x8001, 0x803f, 13767, 54), (0x0033, 0x8005, 26803, 48),
             (0x8002, 0x002f, 46172, 60), (0x8004, 0x800f, 6513, 27), (0x001d, 0x0019, 39103, 33), (0x8012, 0x0023, 63544, 50),
             (0x8002, 0x8013, 75744, 53), (0x8031, 0x000b, 43390, 38), (0x0030, 0x0003, 61605, 62), (0x001a, 0x800c, 5443, 29)]


@pytest.mark.gpu
def test_subnormal_pairs_bit_for_bit():
    import torch
    from helpers import to_bits, to_dev
    from paper_2506_19651_b200 import binding as pb
    n = 4096
    rng = np.random.default_rng(3)
    x = (rng.integers(0, 2, (n, 3, 128)) << 15 | rng.integers(0, 128, (n, 3, 128))).astype(np.uint16)  # subnormals and zeros
    x[2048:3072, :, 40:64] = x[2048:3072, :, 104:128] = 0  # pairs of zeros among them
    pos = rng.integers(0, 80000, n).astype(np.int32)
    for t, (a, b, p, i) in enumerate(SUBNORMAL):
        pos[t] = p
        x[t, :, i], x[t, :, i + 64] = a, b
    q, k = np.ascontiguousarray(x[:, :2]), np.ascontiguousarray(x[:, 2:])
    qd, kd = to_dev(q), to_dev(k)
    pb.pevlm_rope_qk(pb.make_shape(n, 1, 0, 0, 2, 1, 128, theta=1e6), qd, kd, qd, kd, 0, n, torch.from_numpy(pos).cuda())
    np.testing.assert_array_equal(to_bits(qd), oracle.rope(q, 1e6, pos=pos.astype(np.int64)))
    np.testing.assert_array_equal(to_bits(kd), oracle.rope(k, 1e6, pos=pos.astype(np.int64)))
