"""A level of 16,777,216 DOFs: a tile of 32 systems takes 2^29 values there, so four tiles
are beyond 32-bit offsets."""
import pytest
import torch

import paper_2605_24882_gb300 as wm

pytestmark = pytest.mark.gpu


def test_torus_of_16_million_dofs():
    hier = wm.Hierarchy(wm.Geometry("torus", 2, 4096, 4096), 10)
    assert hier.num_dofs(0) == 2 ** 24
    kw = dict(b=hier.noise_loads(1, 1), kappa=3.0, beta=0.7, sinc_k=0.5, l_lo=-1, l_hi=1, n_samples=1)
    u, st = hier.sample_fields(precision="mixed", **kw)
    assert st["n_not_converged"] == 0
    ref, _ = hier.sample_fields(precision="fp64", rtol=1e-9, **kw)
    assert float((u - ref).norm() / ref.norm()) < 1e-6
    # the same residual in three tiles, two of one shift and one of two
    g = torch.Generator(device="cuda").manual_seed(3)
    r = torch.randn((66, 2 ** 24), dtype=torch.float64, device="cuda", generator=g)
    r[63] = r[64] = r[0]
    sg = [30.0] * 64 + [30.0, 2.0]
    z = hier.vcycle(r, sg, precision="mixed", smoother_degree=2)
    one = hier.vcycle(r[:1], sg[:1], precision="mixed", smoother_degree=2)[0]
    assert torch.equal(z[0], one) and torch.equal(z[63], one)
    assert float((z[64] - one).abs().max() / one.abs().max()) < 40 * 55 * 2.0 ** -24  # (float sums the other way)
