"""The mass product on the caller's layout (wm_apply_mass with x and y apart) against the
tiled product that an in-place call takes: the same sums in the same order, so the same bits."""
import ctypes as C

import pytest
import torch

import paper_2605_24882_gb300 as wm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("surf", [("sphere", 1, 4, 4), ("sphere", 2, 8, 8), ("sphere", 4, 2, 2), ("torus", 3, 16, 8)])
@pytest.mark.parametrize("n_vec", [1, 3, 4, 31, 33, 70])
def test_rows_product_equals_the_tiled_one(surf, n_vec):
    kind, p, nu, nv = surf
    hier = wm.Hierarchy(wm.Geometry(kind, p, nu, nv), 1)
    g = torch.Generator(device="cuda").manual_seed(n_vec)
    x = torch.randn((n_vec, hier.num_dofs(0)), dtype=torch.float64, device="cuda", generator=g)
    x[0, 0] = float("inf")  # stays in the rows that hold DOF 0 of vector 0
    y = hier.apply_mass(x)
    z = x.clone()
    ptr = C.c_void_p(z.data_ptr())
    wm.check(wm.lib().wm_apply_mass(hier._h, 0, ptr, ptr, n_vec, None), "wm_apply_mass")
    torch.cuda.synchronize()
    assert torch.equal(torch.nan_to_num(y, nan=7.0), torch.nan_to_num(z, nan=7.0))
    assert bool(torch.isfinite(y[1:]).all())
