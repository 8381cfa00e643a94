"""The autotuner offers what the solver does by default: on a mesh that fits on
chip the settings it returns are no slower than the default ones."""
import time

import numpy as np
import pytest

from paper_2301_08357_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make", [lambda: S.make_c2(28), lambda: S.make_c1(120)], ids=["cube", "square"])
def test_tuned_settings_are_no_slower_than_the_default(make):
    import torch
    from paper_2301_08357_gb300 import autotune, build
    build.build()
    from paper_2301_08357_gb300 import pressure as P
    case = make()
    ctx = P.ps_ctx_create(0)
    try:
        res = autotune.tune(P, ctx, case, chunks=(0, 1536), reps=5)
        kinds = {(r["operator_kernel"], r["operator_threads"]) for r in res["table"]}
        assert kinds == ({(1, 0), (2, 0), (2, 128), (2, 256)} if case.dim == 3 else {(1, 0)})
        assert {s["engine"] for s in res["solves"]} >= {P.PS_ENGINE_AUTO}
        ms = []
        for kw, opts in (({}, P.make_opts()),
                         ({k: res[k] for k in ("chunk_elems", "pipeline", "operator_kernel", "operator_threads")},
                          P.make_opts(engine=res["engine"], inner_tol=res["inner_tol"]))):
            m = P.ps_mesh_upload(ctx, case.dim, case.coords, case.conn, case.dirichlet, **kw)
            P.ps_coeff_set(m, case.alpha, case.beta, case.dt2)
            b = torch.as_tensor(case.b, device="cuda")
            ts = []
            for _ in range(8):
                x = torch.zeros_like(b)
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                st, _ = P.ps_pressure_solve(m, b, x, opts)
                torch.cuda.synchronize()
                ts.append(time.perf_counter() - t0)
                assert st == P.PS_OK
            ms.append(np.min(ts[1:]))
            P.ps_mesh_free(m)
        # (the kernel-by-kernel engines take two to three times as long here)
        assert ms[1] <= 1.2 * ms[0], ms
    finally:
        P.ps_ctx_destroy(ctx)
