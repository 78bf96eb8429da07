"""GPU: the stage launches of a step form a chain of programmatic dependent
launches, each of which may start before the one in front of it has ended.
Whatever surrounds the chain -- launches one at a time, a captured graph with
a memset, a copy and another stream's work in front of it -- the results are
the same bits; and the operator's point source, which the stage kernels add
themselves, reaches an element of a full block and one of the ragged last
block alike (FP64 oracle; FP32 1e-5, FP64 1e-12 of max |value|).
"""
import numpy as np
import pytest

import oracle as O
from synth import gaussian_pulse, jittered_delaunay_mesh, random_permittivity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1304_5546_gb300 import build as B
    B.build()
    import paper_1304_5546_gb300 as P
    return P


@pytest.mark.parametrize("N,prec,media", [(1, "fp32", True), (2, "fp32", False), (3, "fp32", False),
                                          (3, "fp32simt", True), (4, "fp64", False),
                                          (6, "fp32", True)])
def test_chain_under_capture_and_one_by_one(P, N, prec, media):
    import torch
    mesh = jittered_delaunay_mesh(30, seed=2)
    eps = random_permittivity(mesh[2].shape[0], seed=2) if media else None
    s = P.Solver(*mesh, N=N, precision=prec, eps=eps)
    dt = s.cfl_dt()
    P.dg_operator_set_source(s.op, (0.4, 0.6, 0.2 / dt, 3 * dt, 1.0))
    q0 = s.from_numpy(np.random.default_rng(5).uniform(-1, 1, (3, s.K, s.Np)))
    res = s.new_fields()
    want = q0.clone()
    s.step(want, res, dt, 5)
    one = q0.clone()
    for n in range(5):
        s.step(one, res, dt, 1, t0=n * dt)
        torch.cuda.synchronize()
    assert torch.equal(s.view(one), s.view(want))
    side, graph, q = torch.cuda.Stream(), torch.cuda.CUDAGraph(), q0.clone()
    with torch.cuda.graph(graph):
        main = torch.cuda.current_stream()
        q.zero_()
        side.wait_stream(main)
        with torch.cuda.stream(side):
            q.copy_(q0)
        main.wait_stream(side)
        s.step(q, res, dt, 5)
        out = q * 1.0
    for _ in range(3):
        q.fill_(7.0)
        res.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(s.view(out), s.view(want))
    P.dg_sync_check(s.op)
    s.close()


@pytest.mark.parametrize("where", ["first", "last"])
@pytest.mark.parametrize("N,prec", [(2, "fp32"), (3, "fp32tc"), (4, "fp32ept"), (5, "fp32tc"),
                                    (6, "fp32simt"), (5, "fp64")])
def test_source_in_a_full_and_in_the_ragged_block(P, N, prec, where):
    mesh = jittered_delaunay_mesh(14, seed=3)  # K = 392: no block size divides it
    d = O.Discretization(*mesh, N)
    k = 1 if where == "first" else d.K - 1
    xs, ys = (float(v[mesh[2][k]].mean()) for v in mesh[:2])
    s = P.Solver(*mesh, N=N, precision=prec)
    dt = s.cfl_dt()
    src = (xs, ys, 0.12 / dt, 2.2 * dt, 1.7)
    P.dg_operator_set_source(s.op, src)
    kk, w = O.point_source_weights(d, xs, ys)
    assert kk == k
    q0 = np.stack(gaussian_pulse(d.x, d.y, xs, ys, 0.2)).astype(np.float32).astype(np.float64)

    def rhs(u, t):
        return O.maxwell_rhs(d, u) + O.point_source_rhs(d, k, w, O.ricker(t, *src[2:]))
    want = q0
    for n in range(3):
        want = O.lsrk_step(d, want, n * dt, dt, rhs=rhs)
    q, res, out = s.from_numpy(q0), s.new_fields(), s.new_fields()
    P.dg_rhs(s.op, q, out, 2 * dt)
    s.step(q, res, dt, nsteps=3)
    P.dg_sync_check(s.op)
    tol = 1e-12 if prec == "fp64" else 1e-5
    for got, ref in ((s.to_numpy(out), rhs(q0, 2 * dt)), (s.to_numpy(q), want)):
        assert np.abs(got - ref).max() <= tol * np.abs(ref).max()
    s.close()
