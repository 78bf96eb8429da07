"""GPU: the element-row FP32 kernel (large meshes at N = 3..5): where the
dispatch takes it, its ragged last block, its point source and its results in
a partition and under capture.  Oracle parity at K = 51,842 and 101,250 is in
test_parity_large_gpu.py; here the node-thread FP32 kernel is the reference
(each is within 1e-5 of max |value| of the oracle, so they are within 2e-5 of
each other).
"""
import numpy as np
import pytest

from synth import jittered_delaunay_mesh, random_permittivity

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


def _mesh(n, drop=0):
    VX, VY, E = jittered_delaunay_mesh(n, seed=5)
    if drop:  # the last triangles, and the vertices only they have
        used, E = np.unique(E[:-drop], return_inverse=True)
        VX, VY, E = VX[used], VY[used], E.reshape(-1, 3).astype(np.int32)
    return VX, VY, E


def _close(a, b):
    assert np.abs(a - b).max() <= TOL * np.abs(b).max(), np.abs(a - b).max() / np.abs(b).max()


@pytest.mark.parametrize("N", [3, 4, 5])
def test_dispatch_and_block_sizes(P, N):
    sms = __import__("torch").cuda.get_device_properties(0).multi_processor_count
    n = int(np.ceil(np.sqrt(128 * sms)))  # 2 n^2 >= 256 elements per multiprocessor
    other = 80 if N == 3 else 40
    big, small = P.Solver(*_mesh(n), N=N), P.Solver(*_mesh(n - 2), N=N)
    assert small.kernel() == ("tensor cores", other)
    assert big.kernel() == ("tensor cores", 128)
    q = big.from_numpy(np.random.default_rng(N).uniform(-1, 1, (3, big.K, big.Np)))
    er = big.to_numpy(big.rhs(q))
    P.dg_operator_set_block_elems(big.op, other)
    assert big.kernel() == ("tensor cores", other)
    _close(er, big.to_numpy(big.rhs(q)))
    P.dg_operator_set_block_elems(big.op, 0)
    assert big.kernel() == ("tensor cores", 128)
    np.testing.assert_array_equal(er, big.to_numpy(big.rhs(q)))
    P.dg_operator_set_alpha(big.op, 0.5)  # two flux scalars: the other kernel
    assert big.kernel() == ("tensor cores", other)
    P.dg_sync_check(big.op)


@pytest.mark.parametrize("media", [False, True])
@pytest.mark.parametrize("N", [3, 4, 5])
@pytest.mark.parametrize("drop", [0, 1, 83])  # last block of 104, 103 and 21 elements
def test_steps_with_source(P, N, media, drop):
    mesh = _mesh(158, drop)
    K = mesh[2].shape[0]
    eps = random_permittivity(K, seed=3) if media else None
    q0 = np.random.default_rng(N).uniform(-1, 1, (3, K, (N + 1) * (N + 2) // 2))
    got = {}
    for prec in ("fp32", "fp32simt"):
        s = P.Solver(*mesh, N=N, precision=prec, eps=eps)
        dt = s.cfl_dt()
        got[prec] = []
        for k in (1, K - 1):  # a source in a full block and in the last one
            xs, ys = (float(v[mesh[2][k]].mean()) for v in mesh[:2])
            P.dg_operator_set_source(s.op, (xs, ys, 0.12 / dt, 2.2 * dt, 1e-3))
            q, res, out = s.from_numpy(q0), s.new_fields(), s.new_fields()
            P.dg_rhs(s.op, q, out, 2 * dt)
            s.step(q, res, dt, 3)
            P.dg_sync_check(s.op)
            got[prec] += [s.to_numpy(out), s.to_numpy(q)]
        if prec == "fp32":
            assert s.kernel() == ("tensor cores", 128)
        s.close()
    for a, b in zip(got["fp32"], got["fp32simt"]):
        _close(a, b)


@pytest.mark.parametrize("N,media", [(3, True), (4, False), (5, False), (5, True)])
def test_partition_and_capture_are_bit_equal(P, N, media):
    import torch
    mesh = _mesh(158)
    eps = random_permittivity(mesh[2].shape[0], seed=3) if media else None
    s = P.Solver(*mesh, N=N, eps=eps)
    assert s.kernel() == ("tensor cores", 128)
    dt = s.cfl_dt()
    q0 = s.from_numpy(np.random.default_rng(1).uniform(-1, 1, (3, s.K, s.Np)))
    res, want, got = s.new_fields(), q0.clone(), s.new_fields()
    s.step(want, res, dt, 4)
    part = P.Partition(s, 3)  # parts below the dispatch's line run the same kernel
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
        torch.cuda.synchronize()
        assert torch.equal(s.view(q), s.view(want))
    P.dg_sync_check(s.op)


# LIFT is one block-diagonal tile, whose zeros meet what a face's flux holds:
# a value that is not finite must reach the elements that it reaches in the
# other tensor-core kernel, whole, and no other element
@pytest.mark.parametrize("media", [False, True])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("N", [3, 4, 5])
def test_non_finite_values_stay_where_they_reach(P, N, bad, media):
    mesh = _mesh(158, 83)
    K = mesh[2].shape[0]
    s = P.Solver(*mesh, N=N, eps=random_permittivity(K, seed=3) if media else None)
    assert s.kernel() == ("tensor cores", 128)
    q = np.random.default_rng(N).uniform(-1, 1, (3, K, s.Np))
    run = lambda: s.to_numpy(s.rhs(s.from_numpy(q)))
    clean = run()
    ks = [0, 127, 128, 20000, K - 1]  # first and last of a block, and of the ragged one
    for k, field in zip(ks, (2, 0, 1, 2, 2)):
        q[field, k, 0] = bad
    got = run()
    P.dg_operator_set_block_elems(s.op, 80 if N == 3 else 40)
    other = run()
    hit = np.unique(np.nonzero(~np.isfinite(got))[1])
    np.testing.assert_array_equal(hit, np.unique(np.nonzero(~np.isfinite(other))[1]))
    assert set(ks) <= set(hit.tolist()) and len(hit) <= 4 * len(ks)
    rest = np.setdiff1d(np.arange(K), hit)
    np.testing.assert_array_equal(got[:, rest], clean[:, rest])
    P.dg_sync_check(s.op)
    s.close()
