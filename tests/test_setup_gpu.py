"""The multigrid set-up with all levels of a block in shared launches (FP32, Q1)
against one level at a time, which a forced strip height selects: the same estimates
of lambda_max and the same inverse diagonals, since the dots keep their partition and
every cell and nodal sum its order.

Meshes of one tile and of many, levels that end at a tile's edge and past it, irregular
bricks, active sets, with and without a cell modulus."""
import numpy as np
import pytest

import synthetic as synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["tiny", "small", "box5_4_2", "band4_2_4", "band9_3_3", "box1_5_1"])
@pytest.mark.parametrize("modulus", [False, True])
def test_levels_at_once_match_one_at_a_time(name, modulus):
    import torch
    from paper_2404_03265_gb300 import MG, PFF_F32, Mesh, Problem
    m = Mesh.from_recipe(synth.recipe(name)).finalize(1)
    X, Y, F = m.slots()
    valid = (F & 1) == 1
    ns = len(X)
    u, phi, phit = synth.linearisation(X[valid], Y[valid], m.info["x_max"], m.info["y_max"], seed=4, u_std=1e-3)
    rng = np.random.Generator(np.random.PCG64(29))

    def dev(a):
        out = np.zeros(a.shape[1:] + (ns,), dtype=a.dtype)
        out[..., valid] = np.moveaxis(a, 0, -1)
        return torch.tensor(out, device="cuda")

    act = dev((rng.uniform(size=valid.sum()) < 0.1).astype(np.uint8))
    E = torch.tensor(rng.lognormal(0.0, 0.1, m.info["n_leaf_cells"]), device="cuda")
    got = []
    for sched in (0, 15):
        pb = Problem(m, E=1.0, nu=0.2, Gc=1.0, eps=2.0 * m.info["h_min"], kappa=1e-3, p=0.05)
        pb.set_cell_loop(sched)
        if modulus:
            pb.set_cell_modulus(E)
        pb.set_state(dev(u), dev(phi), dev(phit))
        pb.set_active(act)
        mg = MG(pb, PFF_F32)
        for _ in range(2):   # the second set-up meets the buffers of the first
            mg.setup()
        got.append([mg.lam(b) for b in (0, 1)] +
                   [mg.inverse_diagonal(l, b)[0].cpu().numpy() for b in (0, 1) for l in range(mg.n_levels)])
    for x, y in zip(*got):
        assert np.all(np.isfinite(x)) and np.array_equal(x, y)
