"""The FP64 form's arithmetic, compiled for the host from the kernels' own headers: the
fixed-point operations against exact rational arithmetic, whole runs against the same formulas
in extended precision."""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from oracle.model import get_model

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
def test_product_by_omega_rounds_to_nearest(host, omega):
    """Error at most half a unit and 2^-28 (two truncated terms below 2^-29 each), zero of zero
    and of terms far below a unit; the mean error of n products within 6 standard deviations
    of 0 for errors of at most half a unit each (0.5 / sqrt(n) is one)."""
    rng = np.random.default_rng(3)
    n, err = 20000, []
    assert host.host_fx_mul(0, omega) == 0
    for k in range(n):
        a = int(rng.integers(-3 << 60, 3 << 60)) >> (k % 60 if k % 4 == 0 else 0)
        err.append(Fraction(host.host_fx_mul(a, omega)) - Fraction(a) * Fraction(omega))
    assert max(abs(v) for v in err) <= Fraction(1, 2) + Fraction(1, 1 << 28)
    assert abs(float(sum(err)) / n) <= 6 * 0.5 / np.sqrt(n)


@pytest.mark.parametrize("omega", [0.3, 1.0, 1.2, 1.5, 1.8, 1.999])
def test_equilibrium_is_a_fixed_point(host, omega):
    """A pair at its equilibrium stays there bit for bit, the rest state's zeros among them."""
    rng = np.random.default_rng(5)
    for k in range(500):
        ev = 0.0 if k % 5 == 0 else float(rng.standard_normal() * 10.0 ** rng.uniform(-12, 0))
        od = 0.0 if k % 3 == 0 else ev * float(rng.integers(-64, 65)) / 64.0
        if Fraction(ev + od) != Fraction(ev) + Fraction(od) or Fraction(ev - od) != Fraction(ev) - Fraction(od):
            continue
        hp, hm = ctypes.c_double(ev + od), ctypes.c_double(ev - od)
        host.host_relax(ev, od, ctypes.byref(hp), ctypes.byref(hm), omega)
        assert (hp.value, hm.value) == (ev + od, ev - od)


@pytest.mark.parametrize("omega", [2.0 ** -6, 1.0, 1.2, 1.8, 1.999])
def test_relaxation_of_a_pair(host, omega):
    """h + omega (h^eq - h) within six units of 2^-60 of the largest term's power of two and
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
            assert abs(Fraction(got) - want) <= 6 * unit + abs(want) * Fraction(2) ** -53


def collide(e, w, a, D, h, omega):
    """The collision of the deviations h [Q, cells], direction by direction, in h's type."""
    one = h.dtype.type
    x2 = [one(a * a * float(v @ v)) for v in e]            # the library's table: rounded once
    zero = np.zeros(h.shape[1], h.dtype)
    r, E, j = zero.copy(), zero.copy(), [zero.copy() for _ in range(D)]
    for i in range(len(e)):
        t = one(w[i]) * h[i]
        r += t
        E += x2[i] * t
        for d in range(D):
            j[d] += one(e[i, d]) * t
    rho = 1 + r
    u = [one(a) * j[d] / rho for d in range(D)]
    q = sum(v * v for v in u)
    t = ((E - D * r) / rho - q) / D
    out = np.empty_like(h)
    for i in range(len(e)):
        s = sum(one(a) * one(e[i, d]) * u[d] for d in range(D))
        x = x2[i]
        a0 = q * (q / 8 - one(0.5)) + t * (t * one(D * (D + 2) / 8) + q * one((D + 2) / 4) - one(D / 2)) \
            + x * (t * (one(0.5) - q / 4 - t * one((D + 2) / 4)) + x * t * t / 8)
        a1 = 1 - q / 2 - t * one((D + 2) / 2) + x * t / 2
        a2 = one(0.5) - q / 4 - t * one((D + 4) / 4) + x * t / 4
        eq = r + rho * (a0 + s * (a1 + s * (a2 + s * (one(1) / 6 + s / 24))))
        out[i] = h[i] + one(omega) * (eq - h[i])
    return out


def set_up(host, model):
    """Lattice vectors in the library's order, their weights, a and D; the host tables filled."""
    mdl, m = get_model(model), int(model == "D3Q95")
    a = float(np.sqrt(2.0) * mdl.c)
    order = np.zeros((mdl.Q, 3), np.int32)
    host.host_velocities(m, order.ctypes.data_as(ctypes.c_void_p))
    e = order[:, :mdl.D]
    pos = {tuple(v): i for i, v in enumerate(mdl.e.tolist())}
    w = np.ascontiguousarray([mdl.w[pos[tuple(v)]] for v in e.tolist()])
    host.host_setup(m, w.ctypes.data_as(ctypes.c_void_p), ctypes.c_double(a))
    return e, w, a, mdl.D


@pytest.mark.parametrize("model,dims,steps,omega", [("D2Q33", (64, 8, 1), 150, 1.5), ("D2Q33", (25, 13, 1), 60, 1.2),
                                                    ("D3Q95", (16, 7, 6), 40, 1.8), ("D3Q95", (9, 8, 5), 40, 1.2)])
def test_whole_runs_stay_as_near_to_exact_as_plain_fp64(host, model, dims, steps, omega):
    """A perturbed two-state flow: the populations' rms distance from extended precision after
    all steps is at most that of the same collision evaluated direction by direction in FP64,
    with a fifth for the scatter of two rounding sequences."""
    m, (order, w, a, D) = int(model == "D3Q95"), set_up(host, model)
    order = np.pad(order, ((0, 0), (0, 3 - D)))
    Q = len(order)
    e = order.astype(np.float64)
    rng = np.random.default_rng(9)
    z, y, x = np.meshgrid(*[np.arange(n) for n in dims[::-1]], indexing="ij")
    wave = 0.02 * np.cos(2 * np.pi * x / dims[0] + 1) * np.cos(2 * np.pi * y / dims[1] + 0.3)
    h0 = (np.where(x < dims[0] // 2, 0.0, -0.4) + wave).reshape(1, -1) + 0.02 * np.sin(e[:, :1] + z.reshape(1, -1))
    h0 = h0 * (1 + 1e-3 * rng.standard_normal(h0.shape))
    cells = np.arange(h0.shape[1]).reshape(dims[::-1])
    gather = np.stack([np.roll(cells, tuple(int(v) for v in order[i][::-1]), (0, 1, 2)).ravel() for i in range(Q)])
    rows = np.arange(Q)[:, None]

    def kernels(g):
        c = np.ascontiguousarray(g.T)
        host.host_collide(m, c.ctypes.data_as(ctypes.c_void_p), ctypes.c_long(c.shape[0]), ctypes.c_double(omega))
        return c.T

    def run(h, f):
        for _ in range(steps):
            h = f(h[rows, gather])
        return h

    plain = run(h0, lambda g: collide(order[:, :D], w, a, D, g, omega))
    exact = run(h0.astype(np.longdouble), lambda g: collide(order[:, :D], w, a, D, g, omega))
    got = run(h0, kernels)
    rms = lambda v: float(np.sqrt(np.mean((v - exact) ** 2)))
    assert rms(got) <= 1.2 * rms(plain)


@pytest.mark.parametrize("model", ["D2Q33", "D3Q95"])
def test_collision_has_no_bias(host, model):
    """One collision of random near-equilibrium cells: each direction's mean error against
    extended precision is within 6 standard deviations of its own mean of zero (every constant
    that is multiplied in by a rounded value would show here)."""
    m, (e, w, a, D) = int(model == "D3Q95"), set_up(host, model)
    rng = np.random.default_rng(12)
    n = 40000
    r, t, u = rng.uniform(-0.4, 0.4, n), rng.uniform(-0.3, 0.3, n), 0.1 * rng.standard_normal((D, n))
    h = np.empty((len(e), n))
    for i in range(len(e)):
        s, x, q = a * (e[i].astype(float) @ u), a * a * float(e[i] @ e[i]), (u * u).sum(0)
        h[i] = r + (1 + r) * (-q / 2 + t * (x - D) / 2 + s * (1 + s / 2))
    h *= 1 + 0.05 * rng.standard_normal(h.shape)
    c = np.ascontiguousarray(h.T)
    host.host_collide(m, c.ctypes.data_as(ctypes.c_void_p), ctypes.c_long(n), ctypes.c_double(1.0))
    err = c.T - collide(e, w, a, D, h.astype(np.longdouble), 1.0)
    assert np.all(np.abs(err.mean(axis=1)) <= 6 * err.std(axis=1) / np.sqrt(n))
