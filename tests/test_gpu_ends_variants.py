"""Fixed end planes written by the row-mapped and the linear kernels of every storage form, and
by the separate kernel behind the default two-cell kernel, against the split variant followed
by the separate end-plane kernel: the same arithmetic, so the states agree bit for bit.

Grids: rows that fill their blocks (the 16-bit forms keep the row mapping there), a row of one
block and a bit, rows with most lanes idle (linear mapping), an Nx that is no multiple of 8,
planes along each axis, planes that meet in the middle, and both walking directions (five
steps alternate)."""
import numpy as np
import pytest

from oracle.model import get_model

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["fp16", "bf16", "fp32"])
@pytest.mark.parametrize("model,dims,axis,width",
                         [("D3Q95", (128, 11, 10), 0, 5), ("D3Q95", (256, 10, 12), 1, 5),
                          ("D3Q95", (128, 6, 13), 2, 6), ("D3Q95", (131, 10, 10), 0, 7),
                          ("D3Q95", (61, 7, 12), 2, 6), ("D3Q95", (11, 10, 9), 0, 5),
                          ("D2Q33", (256, 17, 1), 0, 4), ("D2Q33", (257, 9, 1), 1, 4),
                          ("D2Q33", (130, 8, 1), 1, 4)])
def test_end_planes_of_the_direct_and_default_kernels(lbm, model, dims, axis, width, storage):
    mdl = get_model(model)
    D, T0 = mdl.D, mdl.T0
    lo, hi = [1.2] + [0.01] * D + [T0], [0.9] + [0.0] * D + [1.1 * T0]
    rng = np.random.default_rng(11)
    shape = dims[::-1]
    rho, U = 1 + 0.1 * rng.uniform(-1, 1, shape), 0.02 * rng.uniform(-1, 1, (D,) + shape)
    T = T0 * (1 + 0.1 * rng.uniform(-1, 1, shape))
    out = []
    for variant in (lbm.VARIANT_SPLIT, lbm.VARIANT_DIRECT, lbm.VARIANT_AUTO):
        lat = lbm.Lattice(model, dims, 1.6, storage)
        lbm.lbm_set_variant(lat.ctx, variant)
        lat.init(rho, U, T)
        lbm.lbm_set_fixed_ends(lat.ctx, axis, width, lo, hi)
        lat.step(5)
        lbm.lbm_synchronize(lat.ctx)
        out.append(lat.raw())
        lat.close()
    for got in out[1:]:
        assert np.array_equal(out[0].view(np.uint8), got.view(np.uint8))
