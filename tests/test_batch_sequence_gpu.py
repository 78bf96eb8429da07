"""GPU: a batch whose orders run by themselves, beside each other, and change
between the two as problems join and leave; every problem has a point source,
whose times follow the steps since it joined.  Each is within 1e-5 of max
|value| of the oracle in the batch and alone, so within 2e-5 of a solver of
its own.
"""
import numpy as np
import pytest

from synth import gaussian_pulse, jittered_delaunay_mesh, random_permittivity

pytestmark = pytest.mark.gpu
TOL = 2e-5


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1304_5546_gb300 import build as B
    B.build()
    import paper_1304_5546_gb300 as P
    return P


class _Problem:
    def __init__(self, P, N, elems, seed):
        self.N, n = N, int(np.ceil(np.sqrt(elems / 2)))
        mesh = jittered_delaunay_mesh(n, seed=seed)
        eps = random_permittivity(mesh[2].shape[0], seed=seed)
        self.solver = P.Solver(*mesh, N=N, precision="fp32tc", eps=eps)
        self.dt = 0.8 * self.solver.cfl_dt()
        self.q0 = np.stack(gaussian_pulse(*self.solver.nodes(), 0.4, 0.6, 0.2))
        self.source = (0.37, 0.52, 0.15 / self.dt, 2.5 * self.dt, 1.7)

    def join(self, b):
        self.slot, self.steps = b.add(self.solver, self.dt, self.source), 0
        b.set_fields(self.slot, self.q0)

    def alone(self, P):
        s = self.solver
        P.dg_operator_set_source(s.op, self.source)
        q = s.from_numpy(self.q0)
        s.step(q, s.new_fields(), self.dt, self.steps)
        P.dg_sync_check(s.op)
        P.dg_operator_set_source(s.op, None)
        return s.to_numpy(q)


@pytest.mark.parametrize("graph", [True, False])
def test_orders_alone_and_side_by_side(P, graph):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    a = _Problem(P, 3, 80 * sms + 90, 1)       # just over one block a multiprocessor
    b = _Problem(P, 7, 40 * sms + 50, 2)
    c = _Problem(P, 2, 200, 3)                 # a few blocks
    d = _Problem(P, 5, 4 * 40 * sms + 50, 4)   # over four
    cap = [0] * 7
    for p in (a, b, c, d):
        cap[p.N - 1] += (p.solver.K + 3) // 4 * 4
    bt = P.Batch(cap, graph=graph)
    here = []

    def step(*counts):
        for n in counts:
            bt.step(n)
            for p in here:
                p.steps += n

    def check():
        bt.sync_check()
        for p in here:
            want, got = p.alone(P), bt.get_fields(p.slot)
            assert np.abs(got - want).max() <= TOL * np.abs(want).max(), (p.N, p.steps)

    for joins in ([a, b], [c], [d]):
        for p in joins:
            p.join(bt)
            here.append(p)
        step(3, 1, 0, 2)   # a and b alone; all side by side; d alone, the others beside it
        check()
    bt.remove(c.slot)
    here.remove(c)
    step(3)                # all alone
    c.join(bt)             # an order that has not stepped meanwhile
    here.append(c)
    step(2, 3)
    check()
    bt.close()
