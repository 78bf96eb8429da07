"""GPU: the kernels of small FP32 meshes: where the dispatch takes them, the
block sizes on either side of each line with a ragged last block, and their
results in a partition and under capture.  The reference is the kernel taken
above the lines (each is within 1e-5 of max |value| of the oracle, so they are
within 2e-5 of each other).
"""
import numpy as np
import pytest

from synth import jittered_delaunay_mesh, random_permittivity

pytestmark = pytest.mark.gpu
TOL = 2e-5
PER_SM = {1: 32, 2: 32, 3: 56, 4: 32, 5: 16, 6: 8, 7: 8}  # elements per multiprocessor
SMALL_BLOCKS = {N: min(24, e) for N, e in zip(range(1, 8), (64, 32, 32, 32, 24, 16, 12))}


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1304_5546_gb300 import build as B
    B.build()
    import paper_1304_5546_gb300 as P
    return P


def _sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


def _mesh(K):
    n = int(np.ceil(np.sqrt(K / 2)))
    VX, VY, E = jittered_delaunay_mesh(n, seed=5)
    used, E = np.unique(E[:K], return_inverse=True)
    return VX[used], VY[used], E.reshape(-1, 3).astype(np.int32)


def _close(a, b):
    assert np.abs(a - b).max() <= TOL * np.abs(b).max(), np.abs(a - b).max() / np.abs(b).max()


def _other(N):
    return ("element threads", 32) if N <= 2 else ("tensor cores", 80 if N == 3 else 40)


@pytest.mark.parametrize("N", range(1, 8))
def test_dispatch(P, N):
    nodes = ("cuda cores", {1: 64, 2: 32, 3: 32, 4: 32, 5: 24, 6: 16, 7: 12}[N])
    K = PER_SM[N] * _sms()
    small, above = P.Solver(*_mesh(K), N=N), P.Solver(*_mesh(K + 1), N=N)
    assert small.kernel() == nodes
    assert above.kernel() == (("element threads", 32) if N == 3 else _other(N))
    if N == 3:
        K = 224 * _sms()
        assert P.Solver(*_mesh(K), N=3).kernel() == ("element threads", 32)
        assert P.Solver(*_mesh(K + 1), N=3).kernel() == ("tensor cores", 80)
    P.dg_operator_set_block_elems(small.op, _other(N)[1])
    assert small.kernel() == _other(N)
    P.dg_operator_set_block_elems(small.op, 0)
    assert small.kernel() == nodes
    if N >= 3:
        P.dg_operator_set_face_pairs(small.op, True)
        assert small.kernel()[0] == "tensor cores"
        assert P.Solver(*_mesh(100), N=N, precision="fp32tc").kernel()[0] == "tensor cores"


@pytest.mark.parametrize("form", ["plain", "media", "alpha"])
@pytest.mark.parametrize("N", range(1, 8))
def test_steps_with_source(P, N, form):
    sms, Np = _sms(), (N + 1) * (N + 2) // 2
    sizes = [2, SMALL_BLOCKS[N] * sms - 1, SMALL_BLOCKS[N] * sms, PER_SM[N] * sms - 3]
    for K in sizes + ([60 * sms + 5] if N == 3 else []):
        mesh = _mesh(K)
        eps = random_permittivity(K, seed=3) if form == "media" else None
        q0 = np.random.default_rng(N).uniform(-1, 1, (3, K, Np))
        got = {}
        for prec in ("fp32", "fp32ept" if N <= 2 else "fp32tc"):
            s = P.Solver(*mesh, N=N, precision=prec, eps=eps)
            if form == "alpha":
                P.dg_operator_set_alpha(s.op, 0.5)
            dt = s.cfl_dt()
            got[prec] = []
            for k in (0, K - 1):  # a source in the first block and in the last one
                xs, ys = (float(v[mesh[2][k]].mean()) for v in mesh[:2])
                P.dg_operator_set_source(s.op, (xs, ys, 0.12 / dt, 2.2 * dt, 1e-3))
                q, res, out = s.from_numpy(q0), s.new_fields(), s.new_fields()
                P.dg_rhs(s.op, q, out, 2 * dt)
                s.step(q, res, dt, 3)
                P.dg_sync_check(s.op)
                got[prec] += [s.to_numpy(out), s.to_numpy(q)]
            s.close()
        for a, b in zip(*got.values()):
            _close(a, b)


@pytest.mark.parametrize("N,per_sm,media", [(1, 28, False), (3, 50, True), (3, 100, False),
                                            (3, 100, True), (4, 30, False), (7, 8, False)])
def test_partition_and_capture_are_bit_equal(P, N, per_sm, media):
    import torch
    mesh = _mesh(per_sm * _sms())
    eps = random_permittivity(mesh[2].shape[0], seed=3) if media else None
    s = P.Solver(*mesh, N=N, eps=eps)
    assert s.kernel()[0] == ("element threads" if per_sm == 100 else "cuda cores")
    dt = s.cfl_dt()
    q0 = s.from_numpy(np.random.default_rng(1).uniform(-1, 1, (3, s.K, s.Np)))
    res, want, got = s.new_fields(), q0.clone(), s.new_fields()
    s.step(want, res, dt, 4)
    part = P.Partition(s, 3)  # parts below a line on block sizes: the same kernel
    part.set_fields(q0)
    part.step(dt, 4)
    part.get_fields(got)
    part.sync_check()
    assert torch.equal(s.view(got), s.view(want))
    graph, q = torch.cuda.CUDAGraph(), q0.clone()
    with torch.cuda.graph(graph):
        q.copy_(q0)
        s.step(q, res, dt, 4)
    for _ in range(2):
        graph.replay()
    P.dg_sync_check(s.op)
    assert torch.equal(s.view(q), s.view(want))
    s.close()
