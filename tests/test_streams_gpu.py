"""Operators of one problem on several streams at once: the results are the bits of the same
calls one after the other.  On a mesh without refinement edges an apply has no scratch,
so any two may overlap; on other meshes an FP32 apply may overlap an FP64 operator.

The calls of the streams queue up behind a delay, so that they run side by side.

Fresh buffers are ready before a stream of the caller uses them: a multigrid, its set-up
and a solve made on a side stream while the default stream is busy.

An apply captured into a graph gives the bits of an eager one."""
import numpy as np
import pytest

import synthetic as synth

pytestmark = pytest.mark.gpu

F32, F64 = "float32", "float64"


def problem(name, k):
    import torch
    from paper_2404_03265_gb300 import Mesh, Problem
    m = Mesh.from_recipe(synth.recipe(name)).finalize(k)
    X, Y, F = m.slots()
    valid = (F & 1) == 1
    u, phi, phit = synth.linearisation(X[valid], Y[valid], m.info["x_max"], m.info["y_max"], seed=2, u_std=1e-2)

    def dev(a):
        out = np.zeros(a.shape[1:] + (len(X),))
        out[..., valid] = np.moveaxis(a, 0, -1)
        return torch.tensor(out, device="cuda")

    pb = Problem(m, E=1.0, nu=0.2, Gc=1.0, eps=2.0 * m.info["h_min"], kappa=1e-3, p=0.05)
    state = dev(u), dev(phi), dev(phit)
    pb.set_state(*state)
    rng = np.random.Generator(np.random.PCG64(31))
    xs = [torch.tensor(rng.normal(size=(3, len(X))), device="cuda") for _ in range(2)]
    return m, pb, state, xs


@pytest.mark.parametrize("name,k,calls", [
    ("box16_3_0", 1, (F64, F64)), ("box16_3_0", 1, (F32, F32)), ("box16_2_0", 2, (F64, F64)),
    ("box16_3_0", 1, (F64,) * 6), ("box8_3_0", 2, (F64, "residual", F64)),
    ("box9_4_2", 1, (F32, F64)), ("box9_4_2", 1, (F32, "residual")), ("box9_3_2", 2, (F32, F64)),
], ids=str)
def test_streams_match_one(name, k, calls):
    import torch
    from paper_2404_03265_gb300 import PFF_OP_JACOBIAN, PFF_OP_TRANSPOSE
    m, pb, state, xs = problem(name, k)
    assert (m.info["n_hanging"] == 0) == name.endswith("_0")
    n = 200 // len(calls)
    every = range(len(calls))
    streams = [torch.cuda.Stream() for _ in calls]
    xs = [xs[w % 2] * (1 + w) for w in every]
    xs = [x if c == "residual" else x.to(getattr(torch, c)) for x, c in zip(xs, calls)]

    def call(which, rep, y, stream):
        kind = calls[which]
        if kind == "residual":
            pb.residual(*state, y, stream=stream)
            return
        x = xs[which]
        op = PFF_OP_TRANSPOSE if (which + rep) % 2 else PFF_OP_JACOBIAN
        pb.apply(x[:2], x[2], y[:2], y[2], op=op, stream=stream)

    def outputs():
        dt = [torch.float64 if c == "residual" else getattr(torch, c) for c in calls]
        return [[torch.full(xs[0].shape, float("nan"), dtype=dt[w], device="cuda") for _ in range(n)] for w in every]

    want, got = outputs(), outputs()
    for w in every:
        for r in range(2):
            call(w, r, want[w][r], torch.cuda.current_stream())
    torch.cuda.synchronize()
    gate, go = torch.cuda.Stream(), torch.cuda.Event()
    with torch.cuda.stream(gate):
        torch.cuda._sleep(40_000_000)   # about 20 ms: longer than it takes to queue the calls
        go.record(gate)
    for s in streams:
        s.wait_event(go)
    for r in range(n):
        for w in every:
            call(w, r, got[w][r], streams[w])
    torch.cuda.synchronize()
    for w in every:
        for r in range(n):
            assert torch.equal(got[w][r], want[w][r % 2]), (calls[w], r)


@pytest.mark.parametrize("coarse", ["direct", "chebyshev"])
@pytest.mark.parametrize("k", [1, 2])
def test_fresh_solver_on_a_side_stream(k, coarse):
    import torch
    from paper_2404_03265_gb300 import MG, PFF_F32, gmres

    def solve(stream, busy):
        m, pb, state, xs = problem("box4_2_2", k)
        b = xs[0]
        z, x = torch.zeros_like(b[:2]), torch.zeros_like(b)
        torch.cuda.synchronize()
        if busy:
            torch.cuda._sleep(400_000_000)   # about 0.2 s on the default stream
        mg = MG(pb, PFF_F32, coarse=coarse)
        mg.setup(stream=stream)
        r = gmres(pb, mg, b, x, rtol=1e-6, stream=stream)
        torch.cuda.synchronize()             # whatever the default stream still held back
        mg.vcycle(0, b[:2], z, stream=stream)
        torch.cuda.synchronize()
        return [mg.lam(0), mg.lam(1), z.cpu().numpy(), x.cpu().numpy(), r["iterations"]]

    want = solve(torch.cuda.current_stream(), False)
    got = solve(torch.cuda.Stream(), True)
    for a, b in zip(want, got):
        assert np.all(np.isfinite(a)) and np.array_equal(a, b)


@pytest.mark.parametrize("name,k,dtype", [
    ("box9_4_2", 1, F64), ("box9_4_2", 1, F32), ("box9_3_2", 2, F64), ("box9_3_2", 2, F32),
    ("box16_3_0", 1, F64), ("box8_3_0", 2, F64),   # no refinement edges: the cell loop under capture
    ("box16_6_1", 1, F64),                         # contributions made by the first apply, here under capture
], ids=str)
def test_captured_apply_matches_eager(name, k, dtype):
    import torch
    from paper_2404_03265_gb300 import PFF_OP_TRANSPOSE
    m, pb, state, xs = problem(name, k)
    xs = [x.to(getattr(torch, dtype)) for x in xs]
    x, y = xs[0].clone(), torch.full_like(xs[0], float("nan"))
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        pb.apply(x[:2], x[2], y[:2], y[2], op=PFF_OP_TRANSPOSE)
    for v in xs:
        want = torch.full_like(v, float("nan"))
        pb.apply(v[:2], v[2], want[:2], want[2], op=PFF_OP_TRANSPOSE)
        x.copy_(v)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.isfinite(want).all() and torch.equal(y, want)
