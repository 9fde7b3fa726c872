"""The float steps of a solve do one arithmetic for a tile of 32 systems of one shift (rows
combined to S + sigma M) and one for a tile of several shifts (S z and M z apart), whatever
kernel, block and company the tile gets."""
import os

import numpy as np
import pytest
import torch

import paper_2605_24882_gb300 as wm

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "mixed_fields.txt")
MESHES = [("sphere", 2, 16, 16, 5), ("sphere", 3, 16, 16, 5), ("torus", 2, 32, 16, 2), ("torus", 3, 64, 32, 3)]
MIXED = list(np.geomspace(0.7, 2e4, 32))


def batches(first):
    """Lists of tiles: a number stands for 32 systems of that shift, None for a tile of the shifts
    MIXED.  The first one is looked at (a shift's smoother bound depends on its place in the list
    of shifts)."""
    other = [float(s) for s in np.geomspace(1.0, 1e4, 260)]
    return {"alone": [first], "pair": [first] * 2, "three": [first] * 3 + [3.0, None], "singles": [first, 3.0, 70.0, None],
            "many_mixed": [first, 25.0] + [None] * 40, "many_singles": [first] + other[:200] + [None] * 4,
            "many_pairs": [first] * 4 + [s for s in other for _ in range(2)] + [None] * 8,
            "only_pairs": [first] * 4 + [s for s in other[:30] for _ in range(2)]}


@pytest.mark.parametrize("mesh", MESHES, ids=lambda m: "%s_p%d_%dx%d" % m[:4])
@pytest.mark.parametrize("degree", [1, 2, 3])
@pytest.mark.parametrize("first", [25.0, None], ids=["one_shift", "shifts"])
def test_vcycle_of_a_tile_does_not_depend_on_its_company(mesh, degree, first):
    kind, p, nu, nv, levels = mesh
    hier = wm.Hierarchy(wm.Geometry(kind, p, nu, nv), levels)
    n = hier.num_dofs(0)
    g = torch.Generator(device="cuda").manual_seed(nu + degree)
    r0 = torch.randn((32, n), dtype=torch.float64, device="cuda", generator=g)
    z0 = None
    for name, tiles in batches(first).items():
        r = torch.randn((32 * len(tiles), n), dtype=torch.float64, device="cuda", generator=g)
        r[:32] = r0
        sg = sum(([s] * 32 if s is not None else MIXED for s in tiles), [])
        z = hier.vcycle(r, sg, precision="mixed", smoother_degree=degree)[:32].clone()
        z0 = z if z0 is None else z0
        assert torch.equal(z, z0), name


def test_fields_keep_their_values():
    """Fields recorded from the kernels that took a tile at a time.  The float steps being the
    same, only the order of float64 sums (1e-16) is free; a residual replacement turns that into
    flips of float roundings of a correction of 1e-4: 1e-11 is above a few of those."""
    rows = [l.split() for l in open(GOLDEN)]
    for (kind, p, nu, nv, levels), ns in ((MESHES[0], 60), (MESHES[3], 20)):
        hier = wm.Hierarchy(wm.Geometry(kind, p, nu, nv), levels)
        b = np.random.Generator(np.random.PCG64(40)).integers(-2 ** 20, 2 ** 20, size=(ns, hier.num_dofs(0)))
        u, _ = hier.sample_fields(b=torch.tensor(b.astype(np.float64) * 2.0 ** -24, device="cuda"), kappa=5.0, beta=0.75,
                                  n_samples=ns, precision="mixed")
        u = u.cpu().numpy()
        ref = [(int(s), int(i), float(v)) for k, q, s, i, v in rows if (k, int(q)) == (kind, p)]
        d = np.array([u[s, i] - v for s, i, v in ref])
        assert len(ref) > 50
        assert np.sqrt((d * d).mean()) < 1e-11 * np.sqrt(np.mean([v * v for _, _, v in ref]))


@pytest.mark.parametrize("mesh", MESHES, ids=lambda m: "%s_p%d_%dx%d" % m[:4])
@pytest.mark.parametrize("ns", [1, 20, 32, 60, 64, 96])
def test_iterations_of_the_mixed_solve(mesh, ns):
    """Wrong partial dot products (a chunk, a tile, a count left out) would show as steps of the
    wrong length: the mixed solve takes the float64 one's iterations and at most two more, one
    for each restart on a true residual."""
    kind, p, nu, nv, levels = mesh
    hier = wm.Hierarchy(wm.Geometry(kind, p, nu, nv), levels)
    kw = dict(kappa=3.0, beta=0.7, sinc_k=0.5, l_lo=-12, l_hi=12, n_samples=ns, seed=6, rtol=1e-8)
    _, st = hier.sample_fields(precision="mixed", **kw)
    _, ref = hier.sample_fields(precision="fp64", **kw)
    assert st["n_not_converged"] == 0 and st["max_iterations"] <= ref["max_iterations"] + 2


@pytest.mark.parametrize("split", [32, 64])
def test_dots_of_pairs_singles_and_remainders(split):
    """All systems in one solve and in solves of one or two tiles: whatever kernel forms a tile's
    dot products, its float sums are the same, and the fields agree far below the tolerance."""
    hier = wm.Hierarchy(wm.Geometry("sphere", 2, 16), 5)
    b = torch.randn((64, hier.num_dofs(0)), dtype=torch.float64, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(1))
    kw = dict(b=b, kappa=3.0, beta=0.7, sinc_k=0.5, l_lo=-12, l_hi=12, n_samples=64, precision="mixed")
    u, _ = hier.sample_fields(**kw)
    v, _ = hier.sample_fields(max_systems=split, **kw)
    assert float((u - v).norm() / u.norm()) < 1e-11


@pytest.mark.parametrize("cap", [499, 500, 501])
def test_caps_about_the_number_of_systems(cap):
    """500 systems of 20 samples: one solve from a cap of 500 on, below it whole tiles and a
    remainder tile of one shift.  The remainder's company does not enter the fields."""
    hier = wm.Hierarchy(wm.Geometry("sphere", 2, 16), 5)
    b = torch.randn((20, hier.num_dofs(0)), dtype=torch.float64, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(4))
    kw = dict(b=b, kappa=3.0, beta=0.7, sinc_k=0.5, l_lo=-12, l_hi=12, n_samples=20, precision="mixed")
    u, st = hier.sample_fields(**kw)
    v, sv = hier.sample_fields(max_systems=cap, **kw)
    assert st["n_batches"] == 1 and sv["n_batches"] == (1 if cap >= 500 else 2)
    assert float((u - v).norm() / u.norm()) < 1e-11


@pytest.mark.parametrize("surf", [("sphere", 2, 8, 4), ("sphere", 3, 16, 5)])
def test_thin_float64_row_blocks_keep_the_arithmetic(surf):
    """Levels of 152 and 218 rows: two tiles take blocks of two warps and two rows, 80 tiles
    (20 groups) blocks of 16 rows; the same float64 V-cycle bit for bit."""
    kind, p, nu, levels = surf
    hier = wm.Hierarchy(wm.Geometry(kind, p, nu), levels)
    g = torch.Generator(device="cuda").manual_seed(5)
    r = torch.randn((80 * 32, hier.num_dofs(0)), dtype=torch.float64, device="cuda", generator=g)
    sg = np.geomspace(1.0, 1e4, len(r))
    z = hier.vcycle(r, sg, precision="fp64", smoother_degree=3)
    few = hier.vcycle(r[:64], sg[:64], precision="fp64", smoother_degree=3)
    assert torch.equal(z[:64], few)


@pytest.mark.parametrize("shift", [1e30, 3e37])
def test_vcycle_at_the_end_of_the_float_range(shift):
    """Diagonals beyond 2^120, which the kernels' quotients do not take (elements of area 3)."""
    hier = wm.Hierarchy(wm.Geometry("torus", 2, 32, 16, 10.0, 4.0), 2)
    r = torch.randn((40, hier.num_dofs(0)), dtype=torch.float64, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(2))
    z = hier.vcycle(r, [shift] * 33 + [1.0] * 7, precision="mixed", smoother_degree=2)
    ref = hier.vcycle(r, [shift] * 33 + [1.0] * 7, precision="fp64", smoother_degree=2)
    err = (z - ref).abs().amax(dim=1) / ref.abs().amax(dim=1)
    assert bool(torch.isfinite(z).all()) and float(err.max()) < 40 * 55 * 2.0 ** -24
