"""GPU: the FP64 stage kernel (fixed-point products, kernels_f64.cuh) at the
sizes and values where it can go wrong: one element, less and more than a
block, blocks of every size the dispatch picks; every flux form; and operand
vectors that have no fixed-point form (infinite, NaN, out of range), whose
elements take the products in FP64.  FP64 oracle, 1e-12 of max |value|.
"""
import numpy as np
import pytest

import oracle as O
from synth import jittered_delaunay_mesh, random_permittivity

pytestmark = pytest.mark.gpu
TOL = 1e-12


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1304_5546_gb300 import build as B
    B.build()
    import paper_1304_5546_gb300 as P
    return P


def _rhs(P, s, q):
    out = s.to_numpy(s.rhs(s.from_numpy(q)))
    P.dg_sync_check(s.op)
    return out


def _close(a, b):
    assert np.abs(a - b).max() <= TOL * np.abs(b).max(), np.abs(a - b).max() / np.abs(b).max()


@pytest.mark.parametrize("form", ["upwind", "alpha", "media"])
@pytest.mark.parametrize("N", range(1, 8))
@pytest.mark.parametrize("n", [1, 9, 24])
def test_rhs_and_step_match_oracle(P, N, n, form):
    mesh = jittered_delaunay_mesh(n, seed=7)
    if n == 1:  # one element alone: every face a wall
        mesh = (mesh[0][mesh[2][0]], mesh[1][mesh[2][0]], np.array([[0, 1, 2]], np.int32))
    d = O.Discretization(*mesh, N)
    eps = random_permittivity(d.K, seed=2) if form == "media" else None
    s = P.Solver(*mesh, N=N, precision="fp64", eps=eps)
    alpha = 0.25 if form == "alpha" else 1.0
    if form == "alpha":
        P.dg_operator_set_alpha(s.op, alpha)
    # magnitudes from 1e-9 to 1 within an element
    rng = np.random.default_rng(N)
    q = rng.uniform(-1, 1, (3, d.K, d.Np)) * 10.0 ** rng.uniform(-9, 0, (3, d.K, d.Np))
    rhs = (lambda u: O.maxwell_rhs(d, u, alpha=alpha)) if eps is None else \
        (lambda u: O.maxwell_rhs_media(d, u, eps))
    _close(_rhs(P, s, q), rhs(q))
    dt = s.cfl_dt()
    want = O.lsrk_step(d, q, 0.0, dt, rhs=lambda u, t: rhs(u))
    f, res = s.from_numpy(q), s.new_fields()
    s.step(f, res, dt, 1)
    _close(s.to_numpy(f), want)
    s.close()


@pytest.mark.parametrize("N", [1, 4, 7])
@pytest.mark.parametrize("scale", [1e-300, 1e-290, 1e285, 0.0])
def test_fields_beyond_the_fixed_point_range(P, N, scale):
    mesh = jittered_delaunay_mesh(5, seed=3)
    d = O.Discretization(*mesh, N)
    s = P.Solver(*mesh, N=N, precision="fp64")
    q = np.random.default_rng(N).uniform(-1, 1, (3, d.K, d.Np))
    want = _rhs(P, s, q)
    if scale == 0.0:
        assert not _rhs(P, s, 0.0 * q).any()
    else:
        _close(_rhs(P, s, scale * q) / scale, want)
        part = q.copy()  # in some elements only: their neighbours see both
        part[:, : d.K // 2] *= 1e-300
        _close(_rhs(P, s, part), O.maxwell_rhs(d, part))
    s.close()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("N", [1, 4, 7])
def test_non_finite_values_stay_where_they_reach(P, N, bad):
    mesh = jittered_delaunay_mesh(5, seed=3)
    d = O.Discretization(*mesh, N)
    s = P.Solver(*mesh, N=N, precision="fp64")
    q = np.random.default_rng(N).uniform(-1, 1, (3, d.K, d.Np))
    clean = _rhs(P, s, q)
    k = d.K // 2
    q[2, k, 0] = bad  # a vertex node: on two faces
    got = _rhs(P, s, q)
    reach = {k} | {int(d.EToE[k, f]) for f in range(3)}
    hit = set(np.nonzero(~np.isfinite(got))[1].tolist())
    assert k in hit and hit <= reach
    rest = np.setdiff1d(np.arange(d.K), sorted(reach))
    np.testing.assert_array_equal(got[:, rest], clean[:, rest])
    assert not np.isfinite(got[:2, k]).any()
    s.close()
