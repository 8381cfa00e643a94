"""Sums of the on-chip kernel's dot-product shares over its blocks: the sizes run
through block counts around every multiple of 32 (the lanes of the warp that
reads the shares) up to one block per SM.  After a fixed number of iterations the
iterate is compared with the two-kernel engine's, whose sums take another path: a
share lost or counted twice changes every step length from the first one on."""
import numpy as np
import pytest

from paper_2301_08357_gb300 import synthetic as S

pytestmark = pytest.mark.gpu

ITERS = 10


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_2301_08357_gb300 import build
    build.build()
    from paper_2301_08357_gb300 import pressure as P
    ctx = P.ps_ctx_create(0)
    yield P, torch, ctx
    P.ps_ctx_destroy(ctx)


# (a shared mesh takes part in a batch of one too: PS_ENGINE_PERSISTENT)
@pytest.mark.parametrize("n", [6, 20, 42, 46, 62, 63, 64, 65, 66, 88, 90, 92, 107, 109, 111, 124, 127, 130, 150, 260])
def test_iterates_match_the_two_kernel_engine(env, n):
    P, torch, ctx = env
    case = S.make_c1(n)
    m = P.ps_mesh_upload(ctx, case.dim, case.coords, case.conn, case.dirichlet)
    try:
        P.ps_coeff_set(m, case.alpha, case.beta, case.dt2)
        b = torch.as_tensor(case.b, device="cuda")
        for mode, engines, tol in ((P.PS_MODE_FP64, (P.PS_ENGINE_AUTO,), 1e-10),
                                   (P.PS_MODE_MIXED, (P.PS_ENGINE_AUTO, P.PS_ENGINE_PERSISTENT), 1e-4)):
            def run(engine):
                x = torch.zeros_like(b)
                _, info = P.ps_pressure_solve(m, b, x, P.make_opts(mode=mode, engine=engine, tol=1e-30, inner_tol=1e-30,
                                                                   max_iters=ITERS, max_outer=1))
                assert info.iters_inner == ITERS
                return x.cpu().numpy()
            want = run(P.PS_ENGINE_GRAPH)
            for engine in engines:
                # ten iterations of the same recurrence: rounding (2^-53, 2^-24) times the
                # growth over the iterations, far below the effect of one block's share
                err = np.linalg.norm(run(engine) - want) / np.linalg.norm(want)
                assert err <= tol, (mode, engine, err)
    finally:
        P.ps_mesh_free(m)
