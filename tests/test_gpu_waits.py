"""Limits of the on-chip kernels' waits (ps_solve_opts.grid_spin_limit): the
limit bounds one wait, not a run, and a wait that reaches it is reported and
recovered from.  A wait that gives up returns from the kernel; nothing is left
waiting."""
import numpy as np
import pytest

import oracle
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


def _upload(P, ctx, c):
    m = P.ps_mesh_upload(ctx, c.dim, c.coords, c.conn, c.dirichlet, chunk_elems=1536)
    P.ps_coeff_set(m, c.alpha, c.beta, c.dt2)
    return m


def _stretched(n, factor):
    """The square with a stiffer operator: more iterations on the same mesh."""
    c = S.make_c1(n)
    c.beta = c.beta * factor
    return c


def test_limit_bounds_one_wait_not_a_run(env):
    P, torch, ctx = env
    c = _stretched(150, 1e3)
    m = _upload(P, ctx, c)
    try:
        b = torch.as_tensor(c.b, device="cuda")
        x = torch.zeros_like(b)
        limit = 150        # far above one exchange (a few polls), far below all of a run's
        st, infos = P.ps_batch_solve([m], [b], [x], P.make_opts(grid_spin_limit=limit))
        assert st == P.PS_OK
        # (every iteration of a run polls at least once)
        assert infos[0].iters_inner / infos[0].iters_outer > limit
        assert oracle.PressureMatrix.from_case(c).residual(c.b, x.cpu().numpy()) <= 1.05e-10
    finally:
        P.ps_mesh_free(m)


def test_blocks_may_wait_for_busy_ones(env):
    """More meshes than the SMs hold at once, some slow: a mesh's blocks start
    when the thread blocks they are placed on are free, and the time until then
    is no wait between running blocks."""
    P, torch, ctx = env
    cases = [_stretched(130 + 4 * (k % 6), 1e3 if k % 3 == 0 else 1.0) for k in range(48)]
    ms = [_upload(P, ctx, c) for c in cases]
    try:
        bs = [torch.as_tensor(c.b, device="cuda") for c in cases]
        xs = [torch.zeros_like(b) for b in bs]
        st, infos = P.ps_batch_solve(ms, bs, xs, P.make_opts(grid_spin_limit=150))
        assert st == P.PS_OK
        for k in (0, 1, 20, 47):
            A = oracle.PressureMatrix.from_case(cases[k])
            assert A.residual(cases[k].b, xs[k].cpu().numpy()) <= 1.05e-10
    finally:
        for m in ms:
            P.ps_mesh_free(m)


@pytest.mark.parametrize("mode", [1, 0], ids=["mixed", "fp64"])
@pytest.mark.parametrize("make", [lambda: S.make_c1(48), lambda: S.make_c2(12)], ids=["square", "cube"])
def test_single_solve_reports_and_recovers(env, make, mode):
    P, torch, ctx = env
    c = make()
    A = oracle.PressureMatrix.from_case(c)
    m = _upload(P, ctx, c)
    try:
        b = torch.as_tensor(c.b, device="cuda")
        x = torch.zeros_like(b)
        P.ps_pressure_solve(m, b, x, P.make_opts(mode=mode))     # (words with tags of an earlier run)
        with pytest.raises(P.PressureError) as e:
            x.zero_()
            P.ps_pressure_solve(m, b, x, P.make_opts(mode=mode, grid_spin_limit=1))
        assert e.value.status == P.PS_ETIMEOUT
        out = []
        for _ in range(2):
            x = torch.zeros_like(b)
            st, info = P.ps_pressure_solve(m, b, x, P.make_opts(mode=mode))
            assert st == P.PS_OK and A.residual(c.b, x.cpu().numpy()) <= 1.05e-10
            out.append(x)
        assert torch.equal(*out)
    finally:
        P.ps_mesh_free(m)
