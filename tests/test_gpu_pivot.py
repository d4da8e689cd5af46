"""The pivot of an FP64 reflector (csrc/pivot_fp64.cuh): s = sqrt(S), up = x0 - cl and
rb = -1 / (S + |x0| s) against exact integer square roots and rational arithmetic.

Bounds (u = 2^-53, from the header's error analysis with seeds good to 2^-19): the
quick form's s is off by its last rounding, half a unit in the last place, and at most
2^-56 s before that, less than 0.55 units together with the correction's own rounding;
rb by the rounding of S + |x0| s, by s's error in it and by its own rounding, 3 u with
higher-order terms far below the 2^-8 allowed for.  The general form (S out of [2^-900, 2^900) or a column of
extreme scale) uses sqrt and a division: s within one unit of the square root of the
rounded S, rb within 5 u.
"""
import ctypes
import math
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_2506_09463_gb300 import build
    so = str(tmp_path_factory.mktemp("pivot") / "pivot_probe.so")
    subprocess.run([build._nvcc(), *build.NVCC_FLAGS, f"-I{build.CSRC}", "-shared",
                    os.path.join(HERE, "pivot_probe.cu"), "-o", so], check=True)
    fn = ctypes.CDLL(so).pivot_probe
    fn.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int, ctypes.c_void_p, ctypes.c_int]

    def run(x0, tail, E=None, from_S=False):
        n = len(x0)
        d = [torch.from_numpy(np.ascontiguousarray(v, dtype=np.float64)).cuda() for v in (x0, tail)]
        e = torch.from_numpy(np.asarray(E if E is not None else np.zeros(n), dtype=np.int32)).cuda()
        out = torch.empty(n, 4, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert fn(d[0].data_ptr(), d[1].data_ptr(), e.data_ptr(), n, out.data_ptr(),
                  int(from_S)) == 0
        return out.cpu().numpy()
    return run


def exact_sqrt(S):
    """sqrt of a positive Fraction to 2^-90 of itself."""
    p, q = S.numerator, S.denominator
    k = max(0, 100 - (p.bit_length() - q.bit_length()) // 2)
    return Fraction(math.isqrt((p << (2 * k)) // q), 1 << k)


def errors(S, x0, row):
    """Error of s in units of its last place, of up and rb relative to their values."""
    cl, up, rb, defined = (float(v) for v in row)
    assert defined == 1.0
    s = exact_sqrt(Fraction(S))
    ulp = Fraction(math.ulp(abs(cl)))
    es = abs(Fraction(abs(cl)) - s) / ulp
    assert (cl < 0) == (x0 > 0)
    assert up == x0 - cl
    b = -(Fraction(S) + abs(Fraction(x0)) * s)
    return float(es), float(abs(Fraction(rb) * b - 1))


def samples(seed, lo, hi, n):
    """S over all exponents lo .. hi, x0 from 0 to sqrt(S)."""
    rng = np.random.default_rng(seed)
    S = np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(lo, hi, n))
    x0 = np.sqrt(S) * rng.choice([0.0, 1e-18, 1e-9, 0.03, 0.5, 0.999, 1.0], n) * rng.choice([-1, 1], n)
    return S, x0


@pytest.mark.parametrize("lo,hi", [(-900, 900), (-8, 8), (-900, -898), (898, 900)])
def test_quick_form(probe, lo, hi):
    S, x0 = samples(lo + 2000, lo, hi, 4000)
    out = probe(x0, S, from_S=True)
    es, eb = zip(*(errors(S[i], float(x0[i]), out[i]) for i in range(len(S))))
    assert max(es) <= 0.55
    assert max(eb) <= (3 + 2.0 ** -8) * U


@pytest.mark.parametrize("k", [-1000, -901, -900, -899, 0, 899, 900, 1000])
def test_both_sides_of_the_range(probe, k):
    """x0^2 + tail around 2^k: the quick form inside [2^-900, 2^900), the general outside."""
    rng = np.random.default_rng(k + 5000)
    S = np.ldexp(rng.uniform(0.5, 2.0, 400), k)
    x0 = np.where(rng.random(400) < 0.2, 0.0, np.sqrt(S * rng.random(400)))
    tail = np.where(rng.random(400) < 0.1, 0.0, S)
    x0 = np.where((x0 == 0) & (tail == 0), np.sqrt(S), x0)
    out = probe(x0, tail)
    for i in range(len(S)):
        T = Fraction(float(x0[i])) ** 2 + Fraction(float(tail[i]))
        r = float(T)                              # (rounded once, as the FMA does)
        if math.isinf(r):
            continue
        es, eb = errors(r, float(x0[i]), out[i])
        assert es <= 1.0 and eb <= 5.0 * U + 2.0 ** -60


@pytest.mark.parametrize("E", [-1000, -401, 401, 1000])
def test_extreme_scale(probe, E):
    """tail holds the scaled squares, x0 is as stored: s = sqrt((2^-E x0)^2 + tail) 2^E."""
    rng = np.random.default_rng(E + 3000)
    t0, tail = rng.uniform(0.1, 1.0, 300), rng.uniform(0.0, 8.0, 300)
    out = probe(np.ldexp(t0, E), tail, E=np.full(300, E))
    for i in range(300):
        S = float(Fraction(float(t0[i])) ** 2 + Fraction(float(tail[i])))
        s = exact_sqrt(Fraction(S))
        cl = math.ldexp(-float(out[i, 0]), -E)
        assert abs(Fraction(cl) - s) <= Fraction(math.ulp(cl))


def test_no_reflector(probe):
    out = probe(np.zeros(4), np.zeros(4))
    assert (out == 0.0).all()
