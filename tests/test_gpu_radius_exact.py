"""The Box-Muller radius of the smart Monte Carlo draw against IEEE FP32
arithmetic without exception: test_gpu_radius.py evaluates its reference's fused
multiply-adds in FP64, which may round twice, and accepts a few differing
uniforms.  Here every uniform whose value differs from that reference is evaluated
once more in rational arithmetic, one rounding per operation, and has to agree."""
from fractions import Fraction
from math import isqrt

import numpy as np
import pytest

from paper_1711_03828_gb300 import _abi
from tests.test_gpu_radius import _radius

f32 = np.float32


def _round(x: Fraction) -> Fraction:
    """x rounded to FP32, to nearest, ties to even (normal range)."""
    if x == 0:
        return x
    a = abs(x)
    e = a.numerator.bit_length() - a.denominator.bit_length()
    if Fraction(2) ** e > a:
        e -= 1                               # 2^e <= a < 2^(e + 1)
    unit = Fraction(2) ** (e - 23)
    n = a / unit
    k = n.numerator // n.denominator
    r = n - k
    k += r > Fraction(1, 2) or (r == Fraction(1, 2) and k % 2)
    return (k * unit) if x > 0 else -(k * unit)


def _c(v) -> Fraction:
    return Fraction(float(f32(v)))


def _sqrt(x: Fraction) -> Fraction:
    """FP32 root: x is an FP32 number; 80 bits of its root decide the rounding (a tie or
    a longer run is impossible: the root of an FP32 number that is no FP32 number is not
    within 2^-50 of a midpoint)."""
    s = 2 ** 160
    n = isqrt(x.numerator * s // x.denominator)
    return _round(Fraction(n, 2 ** 80))


def _radius_exact(k: int) -> float:
    u = _round(Fraction(2 * k + 1, 2 ** 25))
    v = _round(Fraction(2 ** 25 - 2 * k - 1, 2 ** 25))
    assert k >= 1 << 23 or u == Fraction(2 * k + 1, 2 ** 25)
    if k >= 1 << 23:
        e0 = v <= _c(0.29289321881345248)
        e, f = (0, -v) if e0 else (-1, _round(1 - 2 * v))
    else:
        e, m = 0, u
        while m < 1:
            e, m = e - 1, 2 * m
        if m >= _c(1.41421356237309505):
            e, m = e + 1, m / 2
        f = m - 1
    s = _round(f / _round(2 + f))
    z = _round(s * s)
    t = _round(z * _c(1 / 9) + _c(1 / 7))
    t = _round(z * t + _c(0.2))
    t = _round(z * t + _c(1 / 3))
    ss = s + s
    ln = _round(_round(ss * z) * t + ss)
    ln = _round(e * _c(0.693145751953125) + _round(e * _c(1.428606820309417232e-6) + ln))
    return float(_sqrt(-2 * ln))


def test_rounding_and_root_on_known_values():
    rng = np.random.default_rng(0)
    for x in rng.uniform(0.01, 20.0, 300):
        assert float(_round(Fraction(x))) == float(f32(x))
        y = f32(x)
        assert float(_sqrt(Fraction(float(y)))) == float(np.sqrt(y))


@pytest.mark.gpu
def test_every_uniform_without_exception(cuda_device):
    import torch
    n = 1 << 24
    k = np.arange(n, dtype=np.uint32)
    w = np.zeros((n, 4), np.uint32)
    w[:, 0] = k << np.uint32(8)
    w[:, 2] = (np.uint32(n - 1) - k) << np.uint32(8)
    w[:, 1] = w[:, 3] = np.uint32((1 << 23) << 8)   # the cosine rounds to -1: the normals are -radius
    src = torch.from_numpy(w.reshape(-1).view(np.int32)).to(cuda_device)
    out = torch.empty(4 * n, dtype=torch.float32, device=cuda_device)
    _abi.soma_smc_draws(src.data_ptr(), out.data_ptr(), n, None)
    torch.cuda.synchronize()
    o = out.cpu().numpy().reshape(n, 4)
    want = _radius(k)
    for got in (-o[:, 0], -o[::-1, 2]):
        differ = np.nonzero(got != want)[0]
        assert len(differ) <= 100            # else the reference itself is wrong
        for i in differ.tolist():
            assert float(got[i]) == _radius_exact(i), i
        for i in np.random.default_rng(1).integers(0, n, 500).tolist():   # and the two references agree
            assert float(got[i]) == _radius_exact(i), i
