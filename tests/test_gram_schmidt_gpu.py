"""The Gram-Schmidt stages of GMRES over the row counts at which their loop changes: less
than a visit per thread, full groups of four visits and every rest.

With an orthonormal basis the residual estimate of the Givens rotations is the norm of the
preconditioned residual.  Both are formed in FP64 here (FP64 V-cycle and applies), so they
agree to the rounding of some ten steps on vectors of norm up to 1e2 times the final one:
1e-9 relative.  A row left out or taken twice in a dot or an update moves it by far more."""
import numpy as np
import pytest

import synthetic as synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,visits", [("tiny", 1), ("box8_5_1", 2), ("box10_5_1", 3), ("box12_5_1", 4),
                                         ("box14_5_1", 5), ("box16_5_1", 6), ("box9_6_1", 7)])
@pytest.mark.parametrize("transpose", [False, True])
def test_estimate_is_the_preconditioned_residual(name, visits, transpose):
    import torch
    from paper_2404_03265_gb300 import MG, PFF_F64, PFF_OP_JACOBIAN, PFF_OP_TRANSPOSE, Mesh, Problem, gmres
    m = Mesh.from_recipe(synth.recipe(name)).finalize(1)
    X, Y, F = m.slots()
    valid = (F & 1) == 1
    ns, rows = len(X), 3 * int(valid.sum())
    wave = 4 * 256 * torch.cuda.get_device_properties(0).multi_processor_count
    assert -(-rows // wave) == visits
    u, phi, phit = synth.linearisation(X[valid], Y[valid], m.info["x_max"], m.info["y_max"], seed=6, u_std=1e-3)

    def dev(a):
        out = np.zeros(a.shape[1:] + (ns,))
        out[..., valid] = np.moveaxis(a, 0, -1)
        return torch.tensor(out, device="cuda")

    pb = Problem(m, E=1.0, nu=0.2, Gc=1.0, eps=2.0 * m.info["h_min"], kappa=1e-2, p=0.01)
    pb.set_state(dev(u), dev(phi), dev(phit))
    mg = MG(pb, PFF_F64)
    mg.setup()
    b = dev(synth.vector(X[valid], Y[valid], seed=8))
    b[:, torch.tensor((F & 4) == 4, device="cuda")] = 0.0
    x, y, z = torch.zeros_like(b), torch.empty_like(b), torch.empty_like(b)
    r = gmres(pb, mg, b, x, rtol=0.05, restart=50, maxiter=50, transpose=transpose, check=False)
    assert r["converged"] and r["iterations"] >= 2
    pb.apply(x[:2], x[2], y[:2], y[2], op=PFF_OP_TRANSPOSE if transpose else PFF_OP_JACOBIAN)
    res = b - y
    mg.vcycle(0, res[:2], z[:2])
    mg.vcycle(1, res[2], z[2])
    true = float(z[:, torch.tensor(valid, device="cuda")].norm())
    assert abs(true - r["estimate"]) <= 1e-9 * true, (true, r["estimate"], r["iterations"])
