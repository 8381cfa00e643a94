"""The scalars of the on-chip FP64 run at the ends of their range: right-hand
sides of any size, and a residual that reaches zero."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("precond", [1, 0], ids=["jacobi", "plain"])
@pytest.mark.parametrize("make", [lambda: S.make_c1(21), lambda: S.make_c2(8)], ids=["square", "cube"])
def test_size_of_the_right_hand_side(env, make, precond):
    """A power of two in b is the same power of two in x, bit by bit, as long as
    the dot products r.r and r.D^-1 r can be represented (their products, of
    which the quotients are formed, need not be)."""
    P, torch, ctx = env
    c = make()
    m = P.ps_mesh_upload(ctx, c.dim, c.coords, c.conn, c.dirichlet)
    try:
        P.ps_coeff_set(m, c.alpha, c.beta, c.dt2)
        out = {}
        for k in (0, -380, -300, -150, 150, 300, 440):
            b = torch.as_tensor(np.ldexp(c.b, k), device="cuda")
            x = torch.zeros_like(b)
            st, info = P.ps_pressure_solve(m, b, x, P.make_opts(mode=P.PS_MODE_FP64, precond=precond))
            assert st == P.PS_OK, (k, info.as_dict())
            out[k] = np.ldexp(x.cpu().numpy(), -k), info.iters_inner
        for k, (x, it) in out.items():
            assert it == out[0][1] and np.array_equal(x, out[0][0]), k
    finally:
        P.ps_mesh_free(m)


def test_residual_that_reaches_zero(env):
    """One free vertex, every number of the run exact: the residual is 0 after
    one iteration, which is convergence (the next quotient would be 0 / 0)."""
    P, torch, ctx = env
    X = np.array([[0.0, 0.0], [1.0, 0.0], [0.0, 1.0]])
    m = P.ps_mesh_upload(ctx, 2, X, np.array([[0, 1, 2]], np.int32), np.array([0, 1, 1], np.uint8))
    try:
        P.ps_coeff_set(m, np.full(3, 6.0), np.array([3.0]), 1.0)
        P.ps_mesh_set_mass(m, P.PS_MASS_LUMPED)        # A = 6 / 6 + 3 = 4
        b = torch.tensor([1.0, 0.0, 0.0], dtype=torch.float64, device="cuda")
        for mode in (P.PS_MODE_FP64, P.PS_MODE_MIXED):
            x = torch.zeros_like(b)
            st, info = P.ps_pressure_solve(m, b, x, P.make_opts(mode=mode))
            assert st == P.PS_OK, info.as_dict()
            assert x.cpu().numpy().tolist() == [0.25, 0.0, 0.0] and info.iters_inner == 1
    finally:
        P.ps_mesh_free(m)
