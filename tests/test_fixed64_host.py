"""The FP64 form's fixed-point arithmetic, compiled for the host from the kernels' own headers,
against exact rational arithmetic."""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1303_4624_gb300", "csrc")


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    so = str(tmp_path_factory.mktemp("host") / "fixed64_host.so")
    subprocess.check_call([gxx, "-O1", "-std=c++17", "-ffp-contract=off", "-Wno-attributes", "-shared", "-fPIC",
                           "-I", CSRC, "-o", so, os.path.join(HERE, "fixed64_host.cpp")])
    lib = ctypes.CDLL(so)
    d, ll, i = ctypes.c_double, ctypes.c_longlong, ctypes.c_int
    lib.host_fx_to.restype, lib.host_fx_to.argtypes = d, [ll, i]
    lib.host_fx_from.restype, lib.host_fx_from.argtypes = ll, [d, i]
    lib.host_fx_mul.restype, lib.host_fx_mul.argtypes = ll, [ll, d]
    lib.host_relax.argtypes = [d, d, ctypes.POINTER(d), ctypes.POINTER(d), d]
    return lib


def integers(rng, n):
    """Signed 63-bit integers of every length, many of them ties or next to one."""
    out = []
    for _ in range(n):
        v = int(rng.integers(1, 1 << 62)) >> int(rng.integers(0, 62))
        drop = max(0, v.bit_length() - 53)
        if drop and rng.random() < 0.5:
            v = (v >> drop << drop) + (1 << (drop - 1)) + int(rng.integers(-1, 2))
        out.append(v if rng.random() < 0.5 else -v)
    return out + [0, 1, -1, (1 << 62) - 1, (1 << 63) - 1, -(1 << 63) + 1]


def test_conversion_back_rounds_to_nearest_even(host):
    rng = np.random.default_rng(1)
    for v in integers(rng, 4000):
        for e in (1023, 700, 64):
            assert host.host_fx_to(v, e) == float(Fraction(v) * Fraction(2) ** (e - 1022 - 60)), (v, e)


def test_conversion_keeps_60_bits(host):
    rng = np.random.default_rng(2)
    for e in (1023, 500, 64):
        unit = Fraction(2) ** (e - 1022 - 60)
        for v in np.concatenate([rng.uniform(-1, 1, 500) * 2.0 ** rng.integers(-70, 0, 500), [0.0, -0.0]]):
            v = float(v) * float(Fraction(2) ** (e - 1022))
            if abs(v) < 2.0 ** -1022:           # subnormal values are held as 0
                continue
            exact = Fraction(v) / unit
            want = abs(exact) // 1
            assert host.host_fx_from(v, e) == (want if v >= 0 else -want)


@pytest.mark.parametrize("omega", [2.0 ** -6, 0.3, 1.0, 1.2, 1.5, 1.8, 1.999])
def test_product_by_omega_has_no_preferred_sign(host, omega):
    """Error within four units; its mean over n products within 6 standard deviations of 0 for
    errors of at most 4 units each (4 / sqrt(n) is one)."""
    rng = np.random.default_rng(3)
    n, err = 20000, []
    for _ in range(n):
        a = int(rng.integers(-3 << 60, 3 << 60))
        err.append(float(host.host_fx_mul(a, omega) - Fraction(a) * Fraction(omega)))
    assert np.max(np.abs(err)) <= 4.0
    assert abs(np.mean(err)) <= 6 * 4 / np.sqrt(n)


@pytest.mark.parametrize("omega", [2.0 ** -6, 1.0, 1.2, 1.8, 1.999])
def test_relaxation_of_a_pair(host, omega):
    """h + omega (h^eq - h) within nine units of 2^-60 of the largest term's power of two and
    one FP64 rounding, terms spread over 18 decades, zeros among them."""
    rng = np.random.default_rng(4)
    for _ in range(3000):
        t = rng.standard_normal(4) * 10.0 ** rng.uniform(-18, 0, 4)
        t[rng.random(4) < 0.1] = 0.0
        ev, od, hp, hm = (float(v) for v in t)
        gp, gm = ctypes.c_double(hp), ctypes.c_double(hm)
        host.host_relax(ev, od, ctypes.byref(gp), ctypes.byref(gm), omega)
        unit = Fraction(2) ** (int(np.frexp(np.abs(t).max())[1]) - 60)
        for got, h, eq in ((gp.value, hp, Fraction(ev) + Fraction(od)), (gm.value, hm, Fraction(ev) - Fraction(od))):
            want = Fraction(h) + Fraction(omega) * (eq - Fraction(h))
            assert abs(Fraction(got) - want) <= 9 * unit + abs(want) * Fraction(2) ** -53
