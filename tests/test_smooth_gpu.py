"""The fused level smoothers of the FP32 V-cycle (one launch per level and direction)
against the sweeps that a forced strip height selects: the same bits, since both
evaluate every cell, nodal sum, Chebyshev step and transfer row in the same order.

The tile side (6, 10 or 15 nodes) goes by the tiles of a level; the larger meshes reach all
three on whole levels and on levels with refinement edges.

Meshes with one brick and with many, odd coarse grids (brick edges at every position
of the refinement edges), hanging levels, active sets, with and without a cell modulus."""
import numpy as np
import pytest

import synthetic as synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["tiny", "small", "box5_4_2", "band4_2_4", "band9_3_3", "box1_5_1"])
@pytest.mark.parametrize("modulus", [False, True])
@pytest.mark.parametrize("coarse", ["direct", "chebyshev"])
def test_tiles_match_sweeps_bitwise(name, modulus, coarse):
    import torch
    from paper_2404_03265_gb300 import MG, PFF_F32, Mesh, Problem
    m = Mesh.from_recipe(synth.recipe(name)).finalize(1)
    X, Y, F = m.slots()
    valid = (F & 1) == 1
    ns = len(X)
    u, phi, phit = synth.linearisation(X[valid], Y[valid], m.info["x_max"], m.info["y_max"], seed=2, u_std=1e-3)
    rng = np.random.Generator(np.random.PCG64(17))

    def dev(a):
        out = np.zeros(a.shape[1:] + (ns,), dtype=a.dtype)
        out[..., valid] = np.moveaxis(a, 0, -1)
        return torch.tensor(out, device="cuda")

    act = (rng.uniform(size=valid.sum()) < 0.1).astype(np.uint8)
    E = torch.tensor(rng.lognormal(0.0, 0.1, m.info["n_leaf_cells"]), device="cuda")
    r = {0: torch.tensor(rng.normal(size=(2, ns)), device="cuda"), 1: torch.tensor(rng.normal(size=ns), device="cuda")}
    out = {}
    for sched in (0, 15):
        pb = Problem(m, E=1.0, nu=0.2, Gc=1.0, eps=2.0 * m.info["h_min"], kappa=1e-3, p=0.05)
        pb.set_cell_loop(sched)
        if modulus:
            pb.set_cell_modulus(E)
        pb.set_state(dev(u), dev(phi), dev(phit))
        pb.set_active(dev(act))
        mg = MG(pb, PFF_F32, coarse=coarse)
        mg.setup()
        for b in (0, 1):
            for rep in range(2):   # the second cycle meets the buffers of the first
                z = torch.full_like(r[b], float("nan"))
                mg.vcycle(b, r[b], z)
            torch.cuda.synchronize()
            out.setdefault(b, []).append(z.cpu().numpy())
    for b in (0, 1):
        assert np.all(np.isfinite(out[b][0])) and np.abs(out[b][0]).max() > 0
        assert np.array_equal(out[b][0], out[b][1]), (b, np.abs(out[b][0] - out[b][1]).max())


def tile_sides(m):
    """The tile side of every level >= 1: the smallest of 6, 10, 15 whose tiles that hold a
    node are at most 2, 4, any number per streaming multiprocessor."""
    import torch
    from paper_2404_03265_gb300 import MG, PFF_F32, Problem
    pb = Problem(m)
    one = torch.ones(m.info["n_slots"], dtype=torch.float64, device="cuda")
    pb.set_state(torch.zeros((2, m.info["n_slots"]), dtype=torch.float64, device="cuda"), one, one)
    mg = MG(pb, PFF_F32)
    mg.setup()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    sides = []
    for l in range(1, mg.n_levels):
        node = (mg.inverse_diagonal(l, 1)[1] >= 0).reshape(-1, 30, 30)
        for t, most in ((6, 2), (10, 4), (15, None)):
            n = node.reshape(-1, 30 // t, t, 30 // t, t).any(axis=(2, 4)).sum()
            if most is None or n <= most * sms:
                break
        sides.append(t)
    return sides


@pytest.mark.parametrize("name", ["box9_5_1", "box9_4_4"])
@pytest.mark.parametrize("modulus", [False, True])
@pytest.mark.parametrize("coarse", ["direct", "chebyshev"])
def test_every_tile_side_matches_sweeps_bitwise(name, modulus, coarse):
    from paper_2404_03265_gb300 import Mesh
    assert set(tile_sides(Mesh.from_recipe(synth.recipe(name)).finalize(1))) == {6, 10, 15}
    test_tiles_match_sweeps_bitwise(name, modulus, coarse)
