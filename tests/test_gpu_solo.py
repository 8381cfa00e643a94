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
