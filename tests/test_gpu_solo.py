"""The on-chip CG (the AUTO engine's inner solve of meshes that fit) against the
two-kernel engine and the oracle, over the forms a mesh can take: the smallest
meshes (one block), open and closed stars, odd sizes, arbitrary numberings,
periodic and lumped operators, no Dirichlet nodes, no preconditioner."""
import numpy as np
import pytest

import oracle
from oracle.lumped import LumpedMatrix
from oracle.periodic import PeriodicMatrix
from paper_2301_08357_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_2301_08357_gb300 import build
    build.build()
    from paper_2301_08357_gb300 import pressure as P
    ctx = P.ps_ctx_create(0)
    yield P, torch, ctx
    P.ps_ctx_destroy(ctx)


def _free(case):
    case.dirichlet[:] = 0
    return case


FORMS = [
    ("square_1", lambda: S.make_c1(1), {}),
    ("square_9", lambda: S.make_c1(9), {}),
    ("square_83_shuffled", lambda: S.shuffle_case(S.make_c1(83)), {}),
    ("cube_1", lambda: S.make_c2(1), {}),
    ("cube_7_free", lambda: _free(S.make_c2(7)), {}),
    ("cube_11_shuffled", lambda: S.shuffle_case(S.make_c2(11)), {}),
    ("cube_19", lambda: S.make_c2(19), {}),
    ("cube_10_small_chunks", lambda: S.make_c2(10), {"chunk_elems": 40}),
    ("square_37_periodic", lambda: S.make_periodic_case(2, 37), {"periodic": True}),
    ("cube_9_periodic", lambda: S.make_periodic_case(3, 9), {"periodic": True}),
    ("square_29_lumped", lambda: S.make_c1(29), {"lumped": True}),
    ("cube_12_lumped", lambda: S.make_c2(12), {"lumped": True}),
]


@pytest.mark.parametrize("precond", [1, 0], ids=["jacobi", "plain"])
@pytest.mark.parametrize("mode", [1, 0], ids=["mixed", "fp64"])
@pytest.mark.parametrize("name,make,how", FORMS, ids=[f[0] for f in FORMS])
def test_on_chip_matches_two_kernels(env, name, make, how, mode, precond):
    P, torch, ctx = env
    case = make()
    master = case.extra["master"] if how.get("periodic") else None
    m = P.ps_mesh_upload(ctx, case.dim, case.coords, case.conn, case.dirichlet, periodic=master,
                         chunk_elems=how.get("chunk_elems", 0))
    try:
        P.ps_coeff_set(m, case.alpha, case.beta, case.dt2)
        args = (case.dim, case.coords, case.conn, case.dirichlet)
        if how.get("lumped"):
            P.ps_mesh_set_mass(m, P.PS_MASS_LUMPED)
            A = LumpedMatrix(*args, case.alpha, case.beta, case.dt2)
        elif master is not None:
            A = PeriodicMatrix(*args, master, case.alpha, case.beta, case.dt2)
        else:
            A = oracle.PressureMatrix.from_case(case)
        b = torch.as_tensor(case.b, device="cuda")
        out = []
        for engine in (P.PS_ENGINE_AUTO, P.PS_ENGINE_AUTO, P.PS_ENGINE_GRAPH):
            x = torch.zeros_like(b)
            st, info = P.ps_pressure_solve(m, b, x, P.make_opts(mode=mode, precond=precond, engine=engine, tol=1e-13,
                                                                max_outer=20))
            assert st == P.PS_OK, (engine, info.as_dict())
            out.append((x.cpu().numpy(), info))
        auto, again, two = out
        assert np.array_equal(auto[0], again[0])                        # bitwise reproducible
        if two[1].iters_inner > 8:                                      # one launch per inner run
            assert auto[1].kernel_launches < two[1].kernel_launches
        # both solve the same system to 1e-13 of its right-hand side
        err = np.linalg.norm(auto[0] - two[0]) / np.linalg.norm(two[0])
        assert err <= 1e-9, err
        assert A.residual(case.b, auto[0]) <= 1.05e-10
        # an iteration cap is reported with the iterations done
        x = torch.zeros_like(b)
        st, info = P.ps_pressure_solve(m, b, x, P.make_opts(mode=mode, precond=precond, tol=1e-13, max_iters=2))
        assert st == (P.PS_ENOTCONV if two[1].iters_inner > 2 else P.PS_OK) and info.iters_inner <= 2
    finally:
        P.ps_mesh_free(m)


def test_batch_on_chip(env):
    """Every form at once, with enough blocks for more than one launch and one
    mesh that does not fit on chip: each solution meets the oracle's residual
    and is bitwise the one of the mesh alone."""
    P, torch, ctx = env
    forms = FORMS + [("square_150_%d" % k, lambda: S.make_c1(150), {}) for k in range(18)] + [
        ("cube_44", lambda: S.make_c2(44), {}), ("cube_72", lambda: S.make_c2(72), {})]
    ms, cases, As = [], [], []
    try:
        for name, make, how in forms:
            case = make()
            master = case.extra["master"] if how.get("periodic") else None
            m = P.ps_mesh_upload(ctx, case.dim, case.coords, case.conn, case.dirichlet, periodic=master,
                                 chunk_elems=how.get("chunk_elems", 1536))
            ms.append(m)
            P.ps_coeff_set(m, case.alpha, case.beta, case.dt2)
            args = (case.dim, case.coords, case.conn, case.dirichlet)
            if how.get("lumped"):
                P.ps_mesh_set_mass(m, P.PS_MASS_LUMPED)
                A = LumpedMatrix(*args, case.alpha, case.beta, case.dt2)
            elif master is not None:
                A = PeriodicMatrix(*args, master, case.alpha, case.beta, case.dt2)
            else:
                A = oracle.PressureMatrix.from_case(case)
            cases.append(case)
            As.append(A)
        bs = [torch.as_tensor(c.b, device="cuda") for c in cases]
        xs = [torch.zeros_like(b) for b in bs]
        opts = P.make_opts(tol=1e-10)
        st, infos = P.ps_batch_solve(ms, bs, xs, opts)
        assert st == P.PS_OK
        for f, c, A, x in zip(forms, cases, As, xs):
            assert A.residual(c.b, x.cpu().numpy()) <= 1.05e-10, f[0]
        for k in (0, 1, 5, 8, 10, 12, len(ms) - 2, len(ms) - 1):
            x = torch.zeros_like(bs[k])
            st, info = P.ps_batch_solve([ms[k]], [bs[k]], [x], opts)
            assert st == P.PS_OK and torch.equal(x, xs[k]), forms[k][0]
            assert info[0].iters_inner == infos[k].iters_inner
        # a cap on the iterations is reported for the meshes that need more
        xs = [torch.zeros_like(b) for b in bs]
        st, capped = P.ps_batch_solve(ms, bs, xs, P.make_opts(tol=1e-10, max_iters=3))
        for i, c in zip(infos, capped):
            assert c.iters_inner <= 3 and c.status == (P.PS_OK if i.iters_inner <= 3 else P.PS_ENOTCONV)
    finally:
        for m in ms:
            P.ps_mesh_free(m)


@pytest.mark.parametrize("make", [lambda: S.shuffle_case(S.make_c1(13)), lambda: S.shuffle_case(S.make_c2(5))],
                         ids=["square", "cube"])
def test_infinite_entry_reaches_its_neighbours_only(env, make):
    """An infinite or NaN value reaches the rows its element matrices couple it
    to, and no others (2D stars of every size share one code path; an open
    star's two ends are no neighbours)."""
    P, torch, ctx = env
    c = make()
    m = P.ps_mesh_upload(ctx, c.dim, c.coords, c.conn, c.dirichlet)
    try:
        P.ps_coeff_set(m, c.alpha, c.beta, c.dt2)
        rng = np.random.default_rng(3)
        for bad in (np.inf, np.nan):
            for v in rng.choice(np.flatnonzero(c.dirichlet == 0), 24, replace=False):
                x = rng.standard_normal(c.n_nodes)
                x[v] = bad
                near = np.zeros(c.n_nodes, bool)
                near[np.unique(c.conn[(c.conn == v).any(axis=1)])] = True
                for prec, dt in ((P.PS_F64, torch.float64), (P.PS_F32, torch.float32)):
                    xd = torch.as_tensor(x, dtype=dt, device="cuda")
                    y = torch.empty_like(xd)
                    P.ps_pressure_apply(m, xd, y, prec)
                    assert np.all(np.isfinite(y.cpu().numpy()[~near]))
    finally:
        P.ps_mesh_free(m)
