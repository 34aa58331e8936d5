"""Rounding of lbm_set_populations: the FP64 form without a bias of its direction, the 16-bit
forms next to the midpoint of two stored values."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def set_and_read(lbm, model, dims, storage, f):
    import torch
    lat = lbm.Lattice(model, dims, 1.0, storage)
    lbm.lbm_set_populations(lat.ctx, torch.from_numpy(np.ascontiguousarray(f)).cuda())
    raw = lat.raw()
    lat.close()
    return raw


@pytest.mark.parametrize("model,dims", [("D3Q95", (32, 16, 8)), ("D2Q33", (64, 65, 1))])
def test_fp64_rest_populations_are_exact_zeros(lbm, model, dims):
    w = lbm.lbm_model_info(model)["w"].reshape(-1, 1, 1, 1)
    h = set_and_read(lbm, model, dims, "fp64", np.broadcast_to(w, (len(w),) + dims[::-1]))
    assert np.all(h == 0.0)


@pytest.mark.parametrize("scale", [1e-9, 1e-3, 0.3, 100.0])
@pytest.mark.parametrize("model,dims", [("D3Q95", (32, 16, 8)), ("D2Q33", (64, 65, 1))])
def test_fp64_deviations_have_no_bias(lbm, model, dims, scale):
    """h = f / w - 1 in two roundings at h's own size: within 2 x 2^-53 of h (and 2^-104, the
    reciprocal's rest), and per direction a mean error within 6 standard deviations of 0 for
    relative errors of at most 2 x 2^-53 each (that over sqrt(cells) is one)."""
    w = lbm.lbm_model_info(model)["w"].reshape(-1, 1, 1, 1)
    rng = np.random.default_rng(41)
    f = w * (1.0 + scale * rng.standard_normal((len(w),) + dims[::-1]))
    got = set_and_read(lbm, model, dims, "fp64", f)
    wl = w.astype(np.longdouble)
    want = (f.astype(np.longdouble) - wl) / wl
    err = got - want
    assert np.all(np.abs(err) <= 2 * 2.0 ** -53 * np.abs(want) * (1 + 1e-9) + 2.0 ** -104)
    part = (err / np.maximum(np.abs(want), 2.0 ** -80)).reshape(len(w), -1)
    assert np.all(np.abs(part.mean(axis=1)) <= 6 * 2 * 2.0 ** -53 / np.sqrt(part.shape[1]))


def to_bits(v, storage):
    """FP64 values rounded once (to nearest, even) to FP16 or BF16, as stored bits."""
    if storage == "fp16":
        return v.astype(np.float16).view(np.uint16)
    m, e = np.frexp(v)                                # v = m 2^e, 1/2 <= |m| < 1: 8 bits kept
    r = np.ldexp(np.rint(m * 256.0), e - 8).astype(np.float32)
    return (r.view(np.uint32) >> 16).astype(np.uint16)


@pytest.mark.parametrize("storage", ["fp16", "bf16"])
@pytest.mark.parametrize("model,dims", [("D3Q95", (64, 8, 4)), ("D2Q33", (64, 33, 1))])
def test_16_bit_values_next_to_a_midpoint(lbm, model, dims, storage):
    """f whose deviation lies within a few units of FP64 of the middle between two stored
    values: the stored one is that of f / w - 1 in FP64."""
    w = lbm.lbm_model_info(model)["w"].reshape(-1, 1, 1, 1)
    bits = 11 if storage == "fp16" else 8
    rng = np.random.default_rng(43)
    shape = (len(w),) + dims[::-1]
    m = rng.integers(1 << (bits - 1), 1 << bits, shape) + 0.5              # a midpoint's digits
    mid = np.ldexp(m, rng.integers(-4, 4, shape) - bits) * rng.choice([-1.0, 1.0], shape)
    f = w * (1.0 + mid)
    f = f * (1.0 + 2.0 ** -53 * rng.integers(-3, 4, shape))                # some ulps off
    got = set_and_read(lbm, model, dims, storage, f).view(np.uint16)
    assert np.array_equal(got.reshape(-1), to_bits(f / w - 1.0, storage).reshape(-1))
