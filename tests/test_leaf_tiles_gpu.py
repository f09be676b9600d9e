"""The FP32 Q1 Jacobian of large meshes, regular bricks in tiles and the others swept, against
the sweep of all bricks that a forced strip height selects: the same bits, since both evaluate
every cell and nodal sum in the same order.

Sizes just above the two-pass limit of 650,000 cells: a uniform mesh whose last bricks are cut
by the domain's edge, and a refined one with hanging nodes; random active sets (fixed nodes on
tile edges), with and without a cell modulus."""
import numpy as np
import pytest

import synthetic as synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["box13_6_0", "box13_6_1"])
@pytest.mark.parametrize("modulus", [False, True])
def test_tiles_and_sweep_match_sweep_bitwise(name, modulus):
    import torch
    from paper_2404_03265_gb300 import PFF_OP_CONDENSED, PFF_OP_JACOBIAN, PFF_OP_TRANSPOSE, Mesh, Problem
    m = Mesh.from_recipe(synth.recipe(name)).finalize(1)
    assert m.info["n_leaf_cells"] > 650000
    X, Y, F = m.slots()
    valid = (F & 1) == 1
    ns = len(X)
    g = torch.Generator(device="cuda").manual_seed(31)
    ok = torch.tensor(valid, device="cuda")

    def rand(*shape):
        return torch.randn(*shape, ns, generator=g, device="cuda", dtype=torch.float64) * ok

    pb = Problem(m, E=1.0, nu=0.2, Gc=1.0, eps=2.0 * m.info["h_min"], kappa=1e-3, p=0.05)
    if modulus:
        nc = m.info["n_leaf_cells"]
        pb.set_cell_modulus(torch.exp(0.1 * torch.randn(nc, generator=g, device="cuda", dtype=torch.float64)))
    pb.set_state(rand(2) * 1e-2, rand().abs().clamp(max=1.0), rand().abs().clamp(max=1.0))
    pb.set_active(((rand() > 1.5) & ok).to(torch.uint8))
    x = rand(3).to(torch.float32)
    x[:, ~ok] = 1e30   # holes must be ignored
    for op in (PFF_OP_JACOBIAN, PFF_OP_TRANSPOSE, PFF_OP_CONDENSED):
        got = []
        for sched in (0, 15):
            pb.set_cell_loop(sched)
            y = torch.full_like(x, float("nan"))
            pb.apply(x[:2].contiguous(), x[2].contiguous(), y[:2], y[2], op=op)
            torch.cuda.synchronize()
            got.append(y)
        assert bool(torch.isfinite(got[0]).all()) and float(got[0].abs().max()) > 0
        assert torch.equal(got[0], got[1]), (op, float((got[0] - got[1]).abs().max()))
