"""The two-pass Q1 leaf operators (cells, then node slots) against the column sweep and
its fix-up kernel that a forced strip height selects: the same bits in both precisions,
since both evaluate every cell, nodal sum and condensation in the same order.

The Q2 FP64 passes against the brick kernel that pff_apply_noalloc runs: the same bits.

Meshes: one brick, refinement edges at odd positions of bricks, band refinement with
corner contacts two levels apart; random active sets; with and without a cell modulus."""
import numpy as np
import pytest

import synthetic as synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["tiny", "small", "box5_4_2", "band4_2_4", "band9_3_3", "box1_5_0"])
@pytest.mark.parametrize("modulus", [False, True])
@pytest.mark.parametrize("dtype", ["float64", "float32"])
def test_two_passes_match_sweep_bitwise(name, modulus, dtype):
    import torch
    from paper_2404_03265_gb300 import PFF_OP_CONDENSED, PFF_OP_JACOBIAN, PFF_OP_TRANSPOSE, Mesh, Problem
    m = Mesh.from_recipe(synth.recipe(name)).finalize(1)
    X, Y, F = m.slots()
    valid = (F & 1) == 1
    ns = len(X)
    u, phi, phit = synth.linearisation(X[valid], Y[valid], m.info["x_max"], m.info["y_max"], seed=2, u_std=1e-2)
    rng = np.random.Generator(np.random.PCG64(23))

    def dev(a):
        out = np.zeros(a.shape[1:] + (ns,), dtype=a.dtype)
        out[..., valid] = np.moveaxis(a, 0, -1)
        return torch.tensor(out, device="cuda")

    pb = Problem(m, E=1.0, nu=0.2, Gc=1.0, eps=2.0 * m.info["h_min"], kappa=1e-3, p=0.05)
    if modulus:
        pb.set_cell_modulus(torch.tensor(rng.lognormal(0.0, 0.1, m.info["n_leaf_cells"]), device="cuda"))
    pb.set_state(dev(u), dev(phi), dev(phit))
    pb.set_active(dev((rng.uniform(size=valid.sum()) < 0.1).astype(np.uint8)))
    dt = getattr(torch, dtype)
    x = torch.tensor(rng.normal(size=(3, ns)), device="cuda").to(dt)
    x[:, torch.tensor(~valid, device="cuda")] = 1e30   # holes must be ignored
    for op in (PFF_OP_JACOBIAN, PFF_OP_TRANSPOSE, PFF_OP_CONDENSED):
        got = []
        for sched in (0, 15):
            pb.set_cell_loop(sched)
            y = torch.full_like(x, float("nan"))
            pb.apply(x[:2].contiguous(), x[2].contiguous(), y[:2], y[2], op=op)
            torch.cuda.synchronize()
            got.append(y.cpu().numpy())
        assert np.all(np.isfinite(got[0])) and np.abs(got[0]).max() > 0
        assert np.array_equal(got[0], got[1]), (op, np.abs(got[0] - got[1]).max())


@pytest.mark.parametrize("name", ["tiny", "small", "box5_3_2", "band4_2_3", "band9_2_3", "box3_3_0"])
@pytest.mark.parametrize("modulus", [False, True])
def test_q2_two_passes_match_bricks_bitwise(name, modulus):
    import torch
    from paper_2404_03265_gb300 import (PFF_F64, PFF_OP_CONDENSED, PFF_OP_JACOBIAN, PFF_OP_TRANSPOSE, Mesh, Problem,
                                        _lib)
    m = Mesh.from_recipe(synth.recipe(name)).finalize(2)
    X, Y, F = m.slots()
    valid = (F & 1) == 1
    ns = len(X)
    u, phi, phit = synth.linearisation(X[valid], Y[valid], m.info["x_max"], m.info["y_max"], seed=2, u_std=1e-2)
    rng = np.random.Generator(np.random.PCG64(41))

    def dev(a):
        out = np.zeros(a.shape[1:] + (ns,), dtype=a.dtype)
        out[..., valid] = np.moveaxis(a, 0, -1)
        return torch.tensor(out, device="cuda")

    pb = Problem(m, E=1.0, nu=0.2, Gc=1.0, eps=2.0 * m.info["h_min"], kappa=1e-3, p=0.05)
    if modulus:
        pb.set_cell_modulus(torch.tensor(rng.lognormal(0.0, 0.1, m.info["n_leaf_cells"]), device="cuda"))
    pb.set_state(dev(u), dev(phi), dev(phit))
    pb.set_active(dev((rng.uniform(size=valid.sum()) < 0.1).astype(np.uint8)))
    x = torch.tensor(rng.normal(size=(3, ns)), device="cuda")
    x[:, torch.tensor(~valid, device="cuda")] = 1e30   # holes must be ignored
    for op in (PFF_OP_JACOBIAN, PFF_OP_TRANSPOSE, PFF_OP_CONDENSED):
        got = []
        for fn in (_lib.lib().pff_apply, _lib.lib().pff_apply_noalloc):
            y = torch.full_like(x, float("nan"))
            _lib.check(fn(pb._h, PFF_F64, op, _lib.ptr(x[:2]), _lib.ptr(x[2]), _lib.ptr(y[:2]), _lib.ptr(y[2]),
                          _lib.stream_ptr(None)))
            torch.cuda.synchronize()
            got.append(y.cpu().numpy())
        assert np.all(np.isfinite(got[0])) and np.abs(got[0]).max() > 0
        assert np.array_equal(got[0], got[1]), (op, np.abs(got[0] - got[1]).max())
