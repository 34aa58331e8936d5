"""The step's own fixed end planes against the separate kernel, and the FP64 form's fixed-point
sums at the edges of their range.

End planes: the TMA variant writes them with a second kernel, the library's choice in the
step itself; the arithmetic is the same, so the states agree bit for bit.

Fixed point: one FP64 step is compared with the oracle's collision of the same gathered
populations.  Both work in FP64 (the library's sums with at least 56 bits below a shell's
largest member).  A relative error 2^-53 in each of about 100 terms of the moments moves
every direction by at most 100 x 2^-53 times the largest |h| of the cell times the outer
shells' sensitivity (SENS of the parity tests); the bound is that, with f / w = 1 + h of the
oracle's populations adding 1 to the scale."""
import numpy as np
import pytest

from oracle import lbm as olbm
from oracle.model import get_model

pytestmark = pytest.mark.gpu

SENS = {"D2Q33": 100.0, "D3Q95": 20.0}


@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("model,dims,axis,width", [("D3Q95", (8, 6, 40), 2, 5), ("D3Q95", (48, 5, 3), 0, 7),
                                                   ("D3Q95", (8, 24, 3), 1, 5), ("D2Q33", (72, 7, 1), 0, 4),
                                                   ("D2Q33", (136, 16, 1), 1, 8)])
def test_end_planes_in_the_step_match_the_separate_kernel(lbm, model, dims, axis, width, storage):
    mdl = get_model(model)
    D, T0 = mdl.D, mdl.T0
    lo, hi = [1.2] + [0.01] * D + [T0], [0.9] + [0.0] * D + [1.1 * T0]
    rng = np.random.default_rng(3)
    shape = dims[::-1]
    rho, U = 1 + 0.1 * rng.uniform(-1, 1, shape), 0.02 * rng.uniform(-1, 1, (D,) + shape)
    T = T0 * (1 + 0.1 * rng.uniform(-1, 1, shape))
    out = []
    for variant in (lbm.VARIANT_DIRECT, lbm.VARIANT_TMA):
        lat = lbm.Lattice(model, dims, 1.6, storage)
        lbm.lbm_set_variant(lat.ctx, variant)
        lat.init(rho, U, T)
        lbm.lbm_set_fixed_ends(lat.ctx, axis, width, lo, hi)
        lat.step(5)
        lbm.lbm_synchronize(lat.ctx)
        out.append(lat.raw())
        lat.close()
    assert np.array_equal(out[0].view(np.uint8), out[1].view(np.uint8))


@pytest.mark.parametrize("omega", [0.004, 1.0, 1.93])
@pytest.mark.parametrize("scale", [1e-9, 1e-2])
@pytest.mark.parametrize("model,dims", [("D3Q95", (13, 6, 7)), ("D2Q33", (37, 9, 1)), ("D2Q33", (300, 200, 1))])
def test_fp64_step_of_populations_far_apart_in_size(lbm, model, dims, scale, omega):
    """Members of a shell spread over nine decades, exact zeros among them; relaxation below
    the fixed-point range of omega, and near 2."""
    mdl = get_model(model)
    lat = lbm.Lattice(model, dims, omega, "fp64")
    Q, e = lat.info["Q"], lat.info["e"].astype(int)
    rng = np.random.default_rng(5)
    h = scale * rng.standard_normal((Q,) + dims[::-1]) * 10.0 ** rng.uniform(-9, 0, (Q,) + dims[::-1])
    h[rng.random(h.shape) < 0.1] = 0.0
    lat.set_raw(h)
    lat.step(1)
    got = lat.raw()
    lat.close()
    g = np.stack([np.roll(h[i], (int(e[i, 2]) if mdl.D == 3 else 0, int(e[i, 1]), int(e[i, 0])), (0, 1, 2))
                  for i in range(Q)]).reshape(Q, -1)
    pos = {tuple(v): j for j, v in enumerate(e.tolist())}
    perm = [pos[tuple(v)] for v in mdl.e.tolist()]
    w = mdl.w[:, None]
    ref = olbm.collide(mdl, w * (1.0 + g[perm]), omega) / w - 1.0
    err = np.abs(got.reshape(Q, -1)[perm] - ref)
    assert np.all(err <= 100 * 2.0 ** -53 * SENS[model] * (1.0 + np.abs(g).max(axis=0)))
    if scale == 1e-9:      # nothing is lost to the 1 of f / w = 1 + h: the rest state is not reached
        assert np.abs(got).max() > 1e-12


def test_fp64_non_finite_populations_stay_in_their_cells(lbm):
    """A NaN or infinite population spoils the cell that gathers it and no other."""
    dims = (40, 12, 11)
    lat = lbm.Lattice("D3Q95", dims, 1.5, "fp64")
    e = lat.info["e"].astype(int)
    rng = np.random.default_rng(6)
    h = 0.05 * rng.standard_normal((95,) + dims[::-1])
    lat.set_raw(h)
    lat.step(1)
    clean = lat.raw()
    bad = []
    for i, v in ((3, np.nan), (50, np.inf), (94, -np.inf), (0, np.nan), (20, 1e305)):
        z, y, x = (int(rng.integers(0, n)) for n in dims[::-1])
        h[i, z, y, x] = v
        bad.append(((z + e[i, 2]) % dims[2], (y + e[i, 1]) % dims[1], (x + e[i, 0]) % dims[0]))
    lat.set_raw(h)
    lat.step(1)
    got = lat.raw()
    lat.close()
    spoiled = np.zeros(dims[::-1], bool)
    for c in bad:
        spoiled[c] = True
        assert not np.all(np.isfinite(got[(slice(None),) + c]))
    assert np.array_equal(got[:, ~spoiled], clean[:, ~spoiled])
