"""Kernels that the library picks by grid size, each at sizes that select it (152 SMs): the FP64
step and adjoint with 4, 2 and 1 warps per 32 cells, and the linear FP32 kernel with 64-bit
element indices."""
import numpy as np
import pytest

from oracle import lbm as olbm
from oracle.model import get_model

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.max(np.abs(np.asarray(a) - np.asarray(b))) / np.max(np.abs(b)))


@pytest.mark.parametrize("model,dims", [("D2Q33", (40, 13, 1)), ("D2Q33", (200, 41, 1)), ("D2Q33", (248, 101, 1)),
                                        ("D3Q95", (24, 19, 11)), ("D3Q95", (40, 21, 18)), ("D3Q95", (40, 27, 21))])
def test_fp64_step_has_the_same_bits_for_every_number_of_warps(lbm, model, dims):
    """D2Q33 with 4, 2 and 1 warps, D3Q95 with 4, 2 and again 4, against the TMA variant, whose
    one thread per cell does all parts (its Nx is a multiple of 8; the last group of 32 cells is
    ragged)."""
    mdl = get_model(model)
    rng = np.random.default_rng(21)
    shape = dims[::-1]
    rho, U = 1 + 0.1 * rng.uniform(-1, 1, shape), 0.02 * rng.uniform(-1, 1, (mdl.D,) + shape)
    T = mdl.T0 * (1 + 0.1 * rng.uniform(-1, 1, shape))
    out = []
    for variant in (lbm.VARIANT_TMA, lbm.VARIANT_DIRECT):
        lat = lbm.Lattice(model, dims, 1.7, "fp64")
        lbm.lbm_set_variant(lat.ctx, variant)
        lat.init(rho, U, T)
        lat.step(3)
        out.append(lat.raw())
        lat.close()
    assert np.array_equal(out[0].view(np.uint64), out[1].view(np.uint64))


@pytest.mark.parametrize("model,dims,n", [("D2Q33", (201, 41, 1), 4), ("D2Q33", (131, 119, 1), 4),
                                          ("D3Q95", (41, 17, 11), 3), ("D3Q95", (37, 31, 29), 2)])
def test_fp64_adjoint_with_two_warps_and_one(lbm, model, dims, n):
    """Gradients against the oracle's, 2 and 1 warps for either model; the bound is that of the
    small grids (4 warps): 1e-10 of the largest component."""
    mdl = get_model(model)
    rng = np.random.default_rng(22)
    shape = dims[::-1]
    rho0 = 1.0 + 0.05 * rng.standard_normal(shape)
    U0 = 0.03 * rng.standard_normal((mdl.D,) + shape)
    T0 = mdl.T0 * (1.0 + 0.05 * rng.standard_normal(shape))
    c = rng.standard_normal(shape)
    lat = lbm.Lattice(model, dims, 1.6, "fp64")
    lat.init(rho0, U0, T0)
    lbm.lbm_record(lat.ctx, n, 2)
    dr, dU, dT = np.zeros_like(rho0), np.zeros_like(U0), np.zeros_like(T0)
    dom = lbm.lbm_backward(lat.ctx, np.ascontiguousarray(c), dr, dU, dT)
    lat.close()
    _, odr, odU, odT, odom = olbm.rollout_gradients(mdl, rho0, U0, T0, 1.6, n, c)
    assert rel(dr, odr) < 1e-10
    assert rel(dU, odU) < 1e-10
    assert rel(dT, odT) < 1e-10
    assert abs(dom - odom) < 1e-10 * max(1.0, abs(odom))


def test_linear_fp32_kernel_beyond_32_bit_indices(lbm):
    """D3Q95 FP32 on 201 x 475 x 475 cells (95 x 45.4 M elements, more than 2^32; rows leave
    lanes idle, so the linear kernel runs) against the split variant, bit for bit."""
    import torch
    dims = (201, 475, 475)
    need = 95 * 4 * 4 * 201 * 475 * 475 + (8 << 30)
    if torch.cuda.mem_get_info()[0] < need:
        pytest.skip("not enough device memory")
    mdl = get_model("D3Q95")
    g = torch.Generator(device="cuda").manual_seed(5)
    rho = 1 + 0.1 * torch.rand(dims[::-1], dtype=torch.float64, device="cuda", generator=g)
    U = 0.02 * torch.rand((3,) + dims[::-1], dtype=torch.float64, device="cuda", generator=g)
    T = mdl.T0 * (1 + 0.1 * torch.rand(dims[::-1], dtype=torch.float64, device="cuda", generator=g))
    out = []
    for variant in (lbm.VARIANT_SPLIT, lbm.VARIANT_DIRECT):
        lat = lbm.Lattice("D3Q95", dims, 1.8, "fp32")
        lbm.lbm_set_variant(lat.ctx, variant)
        lbm.lbm_init(lat.ctx, rho, U, T)
        lat.step(2)
        raw = torch.empty((95,) + dims[::-1], dtype=torch.float32, device="cuda")
        lbm.lbm_get_raw(lat.ctx, raw)
        lbm.lbm_synchronize(lat.ctx)
        out.append(raw)
        lat.close()
    assert all(torch.equal(a.view(torch.int32), b.view(torch.int32)) for a, b in zip(*out))
    del out, raw, rho, U, T
    torch.cuda.empty_cache()
