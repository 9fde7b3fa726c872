"""Streaming stencil kernels of the float V-cycle (csrc/wm_stream.h) against the float64
kernels on the same residuals and shifts, at the sizes where their work split changes:
full and part column strips and row chunks, tiles of one shift in groups of one to four,
tiles of mixed shifts, blocks of one and of four tiles.

Tolerance: a V-cycle here chains at most 40 rounded steps (smoothing, residual, transfer),
each within (taps + 6) 2^-24 <= 55 * 2^-24 of its result's size and none amplifying the
error (the smoother and the coarse correction contract it): 1.3e-4 of a system's largest
value.  A wrong neighbour, coefficient or shift changes a value by about its own size.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 40 * 55 * 2.0 ** -24


@pytest.fixture(scope="module")
def wm():
    import paper_2605_24882_gb300 as m
    return m


def shifts(pattern):
    """(systems of) runs of one shift, 0 standing for a run of distinct shifts."""
    out = []
    for k, (n, one) in enumerate(pattern):
        out += [25.0 * 3.0 ** k] * n if one else list(np.geomspace(0.5, 3e4, n))
    return np.array(out)


SHIFTS = {
    "one_system": [(1, 1)],
    "ragged_mixed": [(37, 0)],
    "full_group": [(128, 1)],
    "groups_of_4_3_2_1": [(128, 1), (96, 1), (64, 1), (32, 1)],
    "mixed_between_groups": [(128, 1), (50, 0), (14, 1), (100, 1)],
}
MESHES = [("sphere", 2, 8, 8, 3), ("sphere", 2, 16, 16, 4), ("sphere", 2, 64, 64, 6), ("sphere", 3, 16, 16, 4),
          ("sphere", 3, 64, 64, 6), ("torus", 2, 32, 16, 2), ("torus", 3, 64, 32, 3)]


@pytest.mark.parametrize("mesh", MESHES, ids=lambda m: "%s_p%d_%dx%d" % m[:4])
@pytest.mark.parametrize("pattern", sorted(SHIFTS))
def test_float_vcycle_matches_float64(wm, mesh, pattern):
    import torch
    kind, p, nu, nv, levels = mesh
    hier = wm.Hierarchy(wm.Geometry(kind, p, nu, nv), levels)
    sg = shifts(SHIFTS[pattern])
    g = torch.Generator(device="cuda").manual_seed(len(sg) + nu)
    r = torch.randn((len(sg), hier.num_dofs(0)), dtype=torch.float64, device="cuda", generator=g)
    for degree in (1, 2, 3):
        z = hier.vcycle(r, sg, precision="mixed", smoother_degree=degree)
        ref = hier.vcycle(r, sg, precision="fp64", smoother_degree=degree)
        err = (z - ref).abs().amax(dim=1) / ref.abs().amax(dim=1)
        assert bool(torch.isfinite(z).all()) and float(err.max()) < TOL, (degree, int(err.argmax()), float(err.max()))


@pytest.mark.parametrize("ns", [3, 32, 96, 160])
def test_inactive_tiles_of_a_group_keep_their_results(wm, ns):
    """Shifts that converge at different iterations leave groups with some tiles inactive;
    the fields agree with the float64 path within the solver tolerance."""
    hier = wm.Hierarchy(wm.Geometry("sphere", 2, 16), 4)
    kw = dict(kappa=2.0, beta=1.3, sinc_k=0.5, l_lo=-12, l_hi=12, n_samples=ns, seed=3, rtol=1e-10)
    u, st = hier.sample_fields(precision="mixed", **kw)
    ref, _ = hier.sample_fields(precision="fp64", **kw)
    d = u - ref
    assert st["n_not_converged"] == 0
    err = (d * hier.apply_mass(d)).sum(1) / (ref * hier.apply_mass(ref)).sum(1)
    assert float(err.max()) ** 0.5 < 1e-8


@pytest.mark.parametrize("p", [2, 3])
@pytest.mark.parametrize("ns", [5, 8, 11, 20, 31])
def test_true_residuals_of_tiles_with_a_few_shifts(wm, p, ns):
    """Ragged sample counts put up to four (ns >= 11) or more shifts into a tile: the
    double-float residuals of either kind accept the same solutions as the float64 path
    (both solved to 1e-9, far above the residuals' 2^-42 error)."""
    hier = wm.Hierarchy(wm.Geometry("sphere", p, 16), 4)
    kw = dict(kappa=2.0, beta=0.7, sinc_k=0.5, l_lo=-12, l_hi=12, n_samples=ns, seed=4, rtol=1e-9)
    u, st = hier.sample_fields(precision="mixed", **kw)
    ref, _ = hier.sample_fields(precision="fp64", **kw)
    assert st["n_not_converged"] == 0 and st["n_df_fallbacks"] == 0 and st["max_rel_residual"] <= 1e-9
    d = u - ref
    err = (d * hier.apply_mass(d)).sum(1) / (ref * hier.apply_mass(ref)).sum(1)
    assert float(err.max()) ** 0.5 < 1e-7


@pytest.mark.parametrize("surf", [("sphere", 2, 8, 8, 4), ("sphere", 3, 16, 16, 5), ("torus", 2, 16, 8, 1)])
@pytest.mark.parametrize("ns", [1, 40])
def test_float64_blocks_of_few_rows_keep_the_arithmetic(wm, surf, ns):
    """One system per launch (few blocks: two rows per block) and the same system among
    `ns` x 20 of other shifts (full blocks) give the same float64 V-cycle bit for bit."""
    import torch
    kind, p, nu, nv, levels = surf
    hier = wm.Hierarchy(wm.Geometry(kind, p, nu, nv), levels)
    g = torch.Generator(device="cuda").manual_seed(ns)
    r = torch.randn((20 * ns, hier.num_dofs(0)), dtype=torch.float64, device="cuda", generator=g)
    sg = np.geomspace(1.0, 1e4, 20 * ns)
    z = hier.vcycle(r, sg, precision="fp64", smoother_degree=3)
    pair = hier.vcycle(r[:2], sg[:2], precision="fp64", smoother_degree=3)
    assert torch.equal(z[:2], pair)
