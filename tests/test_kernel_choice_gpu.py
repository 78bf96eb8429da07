"""GPU: the kernel and block size of an FP32 operator as its caller sees and
sets them (dg_operator_kernel, dg_operator_set_block_elems, dg_operator_tune),
and partitions of an operator on a size that was set.
"""
import numpy as np
import pytest

from synth import jittered_delaunay_mesh, random_permittivity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1304_5546_gb300 import build as B
    B.build()
    import paper_1304_5546_gb300 as P
    return P


def _mesh(K):
    n = int(np.ceil(np.sqrt(K / 2)))
    VX, VY, E = jittered_delaunay_mesh(n, seed=5)
    used, E = np.unique(E[:K], return_inverse=True)
    return VX[used], VY[used], E.reshape(-1, 3).astype(np.int32)


# an operator of the element-row kernel on the other tensor-core kernel: in
# its default and in its alternative size, whose parts must run that one too
@pytest.mark.parametrize("N,elems,media", [(3, 40, False), (3, 80, False), (4, 80, False),
                                           (4, 40, True), (4, 80, True), (5, 40, False)])
def test_partition_runs_the_kernel_that_was_set(P, N, elems, media):
    import torch
    mesh = _mesh(40000)
    eps = random_permittivity(40000, seed=3) if media else None
    s = P.Solver(*mesh, N=N, eps=eps)
    assert s.kernel() == ("tensor cores", 128)
    P.dg_operator_set_block_elems(s.op, elems)
    assert s.kernel() == ("tensor cores", elems)
    q0 = s.from_numpy(np.random.default_rng(1).uniform(-1, 1, (3, s.K, s.Np)))
    res, want, got, dt = s.new_fields(), q0.clone(), s.new_fields(), s.cfl_dt()
    s.step(want, res, dt, 2)
    part = P.Partition(s, 3)
    part.set_fields(q0)
    part.step(dt, 2)
    part.get_fields(got)
    part.sync_check()
    P.dg_sync_check(s.op)
    assert torch.equal(s.view(got), s.view(want))
    s.close()


# the reported size keeps the kernel, on either side of every line of the
# dispatch; N = 2's node threads and element threads both have blocks of 32
@pytest.mark.parametrize("K", [100, 9000, 25000, 40000])
@pytest.mark.parametrize("N", range(1, 8))
def test_reported_block_size_is_accepted(P, N, K):
    s = P.Solver(*_mesh(K), N=N)
    first = s.kernel()
    P.dg_operator_set_block_elems(s.op, first[1])
    assert s.kernel() == (("element threads", 32) if N == 2 else first)
    other = {1: 32, 2: 32, 3: 40, 4: 80, 5: 40, 6: 40, 7: 40}[N]
    for size in (other, first[1]):  # away and back
        P.dg_operator_set_block_elems(s.op, size)
        assert s.kernel()[1] == size
    assert s.kernel() == (("element threads", 32) if N == 2 else first)
    P.dg_operator_set_block_elems(s.op, 0)
    assert s.kernel() == first
    with pytest.raises(P.DGError) as ex:
        P.dg_operator_set_block_elems(s.op, 20)
    assert ex.value.status == P._lib.DG_ERR_ARG
    s.close()


# every kernel of the operator is a candidate, and 0 brings the set-up's back
@pytest.mark.parametrize("N,K,cands", [(1, 300, 4), (2, 300, 4), (3, 300, 4), (3, 12000, 4),
                                       (4, 300, 4), (5, 300, 3), (7, 300, 2), (3, 40000, 5),
                                       (4, 40000, 5), (5, 40000, 4)])
def test_tune_times_every_kernel_and_can_be_undone(P, N, K, cands):
    s = P.Solver(*_mesh(K), N=N)
    first = s.kernel()
    assert (first[1] == 128) == (K == 40000)
    n0 = P.dg_launch_count(s.op)
    ms_tc, ms_cc = s.tune(reps=2)
    assert ms_tc > 0 and ms_cc > 0
    assert P.dg_launch_count(s.op) - n0 == 3 * cands
    kernel, elems = s.kernel()
    P.dg_operator_set_block_elems(s.op, elems)  # the choice can be set again
    assert s.kernel() == (kernel, elems)
    if kernel != "tensor cores" and elems != 128:
        with pytest.raises(P.DGError):  # blocks of a kernel that does not run
            P.dg_operator_set_block_elems(s.op, 128)
    P.dg_operator_set_block_elems(s.op, 0)
    assert s.kernel() == first
    s.close()
