"""lbm_set_populations / lbm_get_populations against numpy in 64 bits: odd and tiny grids
(elements of several directions in one thread's pair), buffers aligned to 8 bytes only, and
values that the integer conversions leave to the conversion instruction.

Bounds.  set: h = f / w - 1 rounded once to the storage type, half an ulp of h, and 2^-50
relative (the double-float product) before that rounding; f itself is known to the library
to 2^-53 and its weights agree with the oracle's to 1e-13 relative, which moves h by
(1 + h) 1e-13.  get: f = w (1 + h) in one FP64 rounding, and the same weight difference."""
import numpy as np
import pytest

from oracle.model import get_model

pytestmark = pytest.mark.gpu

HALF_ULP = {"fp64": 2.0 ** -53, "fp32": 2.0 ** -24, "fp16": 2.0 ** -11, "bf16": 2.0 ** -8}
TINY = {"fp64": 0.0, "fp32": 2.0 ** -150, "fp16": 2.0 ** -25, "bf16": 2.0 ** -134}
W_TOL = 2e-13


def stored(lat, storage):
    h = lat.raw()
    if storage == "bf16":
        h = (h.astype(np.uint32) << 16).view(np.float32)
    return h.astype(np.float64)


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp16", "bf16"])
@pytest.mark.parametrize("model,dims", [("D3Q95", (1, 1, 1)), ("D3Q95", (3, 5, 7)),
                                        ("D3Q95", (37, 6, 7)), ("D2Q33", (131, 5, 1)),
                                        ("D2Q33", (1, 1, 1))])
def test_populations_round_trip(lbm, model, dims, storage, offset):
    import torch
    lat = lbm.Lattice(model, dims, 1.0, storage)
    mdl = get_model(model)
    pos = {tuple(v): j for j, v in enumerate(mdl.e.tolist())}
    w = mdl.w[[pos[tuple(v)] for v in lat.info["e"].tolist()]].reshape(-1, 1, 1, 1)
    rng = np.random.default_rng(31)
    shape = (lat.info["Q"],) + dims[::-1]
    h = 0.3 * rng.standard_normal(shape)
    flat = h.reshape(-1)
    flat[::5] *= 1e-7                                   # f next to w
    flat[::7] = 0.0
    flat[3::11] *= 1e3
    f = w * (1.0 + h)
    dev = torch.zeros(f.size + offset, dtype=torch.float64, device="cuda")[offset:]
    dev.copy_(torch.from_numpy(f.reshape(-1)))
    lbm.lbm_set_populations(lat.ctx, dev)
    got = stored(lat, storage)
    want = (f - w) / w
    bound = HALF_ULP[storage] * np.abs(want) * (1 + 2.0 ** -20) + TINY[storage] + 2.0 ** -50 * np.abs(want) \
        + W_TOL * np.abs(1 + want)
    assert np.all(np.abs(got - want) <= bound)
    out = torch.full((f.size + offset,), -1.0, dtype=torch.float64, device="cuda")[offset:]
    lbm.lbm_get_populations(lat.ctx, out)
    back = out.cpu().numpy().reshape(shape)
    assert np.all(np.abs(back - w * (1.0 + got)) <= W_TOL * w * np.abs(1.0 + got) + 2.0 ** -52 * w)
    lat.close()


@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp16", "bf16"])
def test_values_outside_the_fast_conversion(lbm, storage):
    """Subnormal, huge, infinite and NaN populations keep the meaning of the conversions:
    overflow to infinity in the narrow types, NaN stays NaN, signs are kept."""
    import torch
    lat = lbm.Lattice("D3Q95", (4, 1, 1), 1.0, storage)
    w = lbm.lbm_model_info("D3Q95")["w"].reshape(-1, 1, 1, 1)
    f = np.broadcast_to(w, (95, 1, 1, 4)).copy()
    f[1, 0, 0] = (np.inf, -np.inf, np.nan, 1e300)
    f[2, 0, 0] = (1e-310, -1e30, 1e9, 0.0)
    f[3, 0, 0] = w[3, 0, 0, 0] * (1 + np.array([2.0 ** -52, -2.0 ** -53, 2.0 ** -50, 0.0]))
    lbm.lbm_set_populations(lat.ctx, torch.from_numpy(f).cuda())
    with np.errstate(all="ignore"):
        want = (f - w) / w
        top = {"fp64": np.inf, "fp32": 3.4e38, "fp16": 65519.0, "bf16": 3.38e38}[storage]
        want = np.where(np.abs(want) > top, np.copysign(np.inf, want), want)
    got = stored(lat, storage)
    same = np.isfinite(want)
    assert np.array_equal(np.isnan(got), np.isnan(want))
    assert np.array_equal(got[np.isinf(want)], want[np.isinf(want)])
    tol = 2.01 * HALF_ULP[storage] * np.abs(want[same]) + TINY[storage] + 2.0 ** -51
    assert np.all(np.abs(got[same] - want[same]) <= tol)
    out = torch.empty(f.shape, dtype=torch.float64, device="cuda")
    lbm.lbm_get_populations(lat.ctx, out)
    back = out.cpu().numpy()
    assert np.array_equal(np.isnan(back), np.isnan(got))
    assert np.array_equal(back[np.isinf(got)], got[np.isinf(got)])
    lat.close()
