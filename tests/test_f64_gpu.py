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


def _rhs_and_size(P, s, q, alpha, eps):
    """The right-hand side from the operator's own tables and geometry in
    extended precision, and the sum of the absolute values of its terms."""
    LD = np.longdouble
    R, G = P.dg_get_reference(s.op), P.dg_get_geometry(s.op)
    vM, vP = P.dg_get_maps(s.op)
    wall = vM == vP
    N, Nfp = s.N, R["Fmask"].shape[1]
    q = q.astype(LD)
    out = []
    for absolute in (False, True):
        sg = (lambda v: np.abs(v)) if absolute else (lambda v: v)
        minus = LD(1 if absolute else -1)  # the sign of a subtracted term
        Dr, Ds, L = (sg(R[k].astype(LD)) for k in ("Dr", "Ds", "LIFT"))
        rx, ry, sx, sy = (sg(G[k].astype(LD))[:, None] for k in ("rx", "ry", "sx", "sy"))
        nx, ny, F = (sg(np.repeat(G[k].astype(LD), Nfp, axis=1)) for k in ("nx", "ny", "Fscale"))
        u = [sg(c) for c in q]
        # a field is its linear interpolant (derivatives half the vertex
        # differences) and the rest
        lam2, lam3 = ((1 + R[k].astype(LD)) / 2 for k in ("r", "s"))
        rest, gr, gs = [], [], []
        for c in u:
            v1, d2, d3 = c[:, :1], c[:, N:N + 1] + minus * c[:, :1], c[:, -1:] + minus * c[:, :1]
            rest.append(c + minus * v1 + minus * (d2 * lam2 + d3 * lam3))
            gr.append(d2 / 2)
            gs.append(d3 / 2)
        dx, dy, dz = (c.ravel()[vM] + minus * c.ravel()[vP] for c in u)
        dx, dy = (np.where(wall, LD(0), d) for d in (dx, dy))
        dz = np.where(wall, 2 * u[2].ravel()[vM], dz)
        Ht = ny * dx + minus * nx * dy
        if eps is None:
            fh, fz = F / 2 * (LD(alpha) * Ht + minus * dz), F / 2 * (Ht + minus * LD(alpha) * dz)
            zm = sH = sE = LD(1)
        else:
            Z = 1 / np.sqrt(eps.astype(LD))
            zM, zP = np.repeat(Z[:, None], 3 * Nfp, axis=1), Z[vP // s.Np]
            fh = fz = F / (zM + zP) * (zP * Ht + minus * dz)
            zm, sH, sE = zM, LD(1), 1 / eps.astype(LD)[:, None]
        hx, hy, ez = rest
        zr, zs = ez @ Dr.T + gr[2], ez @ Ds.T + gs[2]
        A, B = rx * hy + minus * ry * hx, sx * hy + minus * sy * hx
        lin = rx * gr[1] + minus * ry * gr[0] + sx * gs[1] + minus * sy * gs[0]
        out.append(np.stack([
            sH * (minus * (ry * zr + sy * zs) + minus * (zm * ny * fh) @ L.T),
            sH * (rx * zr + sx * zs + (zm * nx * fh) @ L.T),
            sE * (A @ Dr.T + B @ Ds.T + lin + fz @ L.T)]))
    return out


# Every component to within 32 roundings (2^-53) of the sum of its own terms'
# sizes: a term meets at most 16 on its way (operands 5, coefficients 4,
# product 1, chain rule, update of the sum and row scale 6).  Bubbles with
# entries over nine decades on zero vertices, which deflation leaves as they
# are; and one element far above its neighbours, on axis-aligned faces: where
# a normal's component is zero, a large flux has no part in that row.
@pytest.mark.parametrize("form", ["upwind", "alpha", "media"])
@pytest.mark.parametrize("N", range(1, 8))
@pytest.mark.parametrize("kind", ["bubbles", "one large"])
def test_small_components_keep_their_precision(P, kind, N, form):
    from synth import square_grid_mesh
    mesh = jittered_delaunay_mesh(6, seed=4) if kind == "bubbles" else square_grid_mesh(5, 5)
    s = P.Solver(*mesh, N=N, precision="fp64",
                 eps=random_permittivity(mesh[2].shape[0], seed=2) if form == "media" else None)
    alpha = 0.25 if form == "alpha" else 1.0
    if form == "alpha":
        P.dg_operator_set_alpha(s.op, alpha)
    rng = np.random.default_rng(N)
    shape = (3, s.K, s.Np)
    q = rng.uniform(0.5, 1, shape) * rng.choice([-1.0, 1.0], shape)
    if kind == "bubbles":
        q *= 10.0 ** rng.uniform(-9, 0, shape)
        q[:, :, [0, N, s.Np - 1]] = 0.0
    else:
        q *= 1e-8
        q[:, 22] *= 1e8
    eps = random_permittivity(s.K, seed=2) if form == "media" else None
    want, size = _rhs_and_size(P, s, q, alpha, eps)
    got = _rhs(P, s, q)
    s.close()
    assert (np.abs(got - want) <= 32 * 2.0 ** -53 * size).all(), \
        float((np.abs(got - want)[size > 0] / size[size > 0]).max() * 2 ** 53)


def _solver_and_oracle(P, N, form):
    mesh = jittered_delaunay_mesh(5, seed=3)
    d = O.Discretization(*mesh, N)
    eps = random_permittivity(d.K, seed=2) if form == "media" else None
    s = P.Solver(*mesh, N=N, precision="fp64", eps=eps)
    if form == "alpha":
        P.dg_operator_set_alpha(s.op, 0.25)
        return d, s, lambda u: O.maxwell_rhs(d, u, alpha=0.25)
    return d, s, lambda u: O.maxwell_rhs_media(d, u, eps)


# the products in FP64 with the second flux scalar and with a permittivity
@pytest.mark.parametrize("form", ["alpha", "media"])
@pytest.mark.parametrize("N", range(1, 8))
@pytest.mark.parametrize("scale", [1e-300, 1e285])
def test_fp64_products_in_the_other_flux_forms(P, N, form, scale):
    d, s, rhs = _solver_and_oracle(P, N, form)
    q = np.random.default_rng(N).uniform(-1, 1, (3, d.K, d.Np))
    _close(_rhs(P, s, scale * q) / scale, rhs(q))
    part = q.copy()
    part[:, : d.K // 2] *= 1e-300
    _close(_rhs(P, s, part), rhs(part))
    dt = s.cfl_dt()
    f, res = s.from_numpy(scale * q), s.new_fields()
    s.step(f, res, dt, 1)
    _close(s.to_numpy(f) / scale, O.lsrk_step(d, q, 0.0, dt, rhs=lambda u, t: rhs(u)))
    s.close()


@pytest.mark.parametrize("form", ["alpha", "media"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("N", [1, 4, 7])
@pytest.mark.parametrize("field", [0, 2])
def test_non_finite_values_in_the_other_flux_forms(P, N, form, bad, field):
    d, s, _ = _solver_and_oracle(P, N, form)
    q = np.random.default_rng(N).uniform(-1, 1, (3, d.K, d.Np))
    clean = _rhs(P, s, q)
    k = d.K // 2
    q[field, k, 0] = bad
    got = _rhs(P, s, q)
    reach = {k} | {int(d.EToE[k, f]) for f in range(3)}
    hit = set(np.nonzero(~np.isfinite(got))[1].tolist())
    assert k in hit and hit <= reach
    rest = np.setdiff1d(np.arange(d.K), sorted(reach))
    np.testing.assert_array_equal(got[:, rest], clean[:, rest])
    s.close()
