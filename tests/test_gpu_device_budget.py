"""Device memory at its limit: what a context's budget leaves no room for is
done without, and requests are charged for what they use."""
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
    return P, torch


def test_batch_without_room_for_exchanged_words(env):
    """The words that blocks of a mesh exchange on chip (some 100 bytes per pair
    of blocks) are the batch's largest buffer; without room for them the
    meshes run chunk by chunk."""
    P, torch = env
    cases = [S.make_c2(30) for _ in range(3)]

    def run(budget):
        ctx = P.ps_ctx_create(0, budget)
        try:
            ms = [P.ps_mesh_upload(ctx, c.dim, c.coords, c.conn, c.dirichlet, chunk_elems=1536) for c in cases]
            for m, c in zip(ms, cases):
                P.ps_coeff_set(m, c.alpha, c.beta, c.dt2)
            bs = [torch.as_tensor(c.b, device="cuda") for c in cases]
            xs = [torch.zeros_like(b) for b in bs]
            st, infos = P.ps_batch_solve(ms, bs, xs, P.make_opts())
            assert st == P.PS_OK
            held = P.ps_ctx_bytes_in_use(ctx)
            for m in ms:
                P.ps_mesh_free(m)
            return held, [x.cpu().numpy() for x in xs], [i.kernel_launches for i in infos]
        finally:
            P.ps_ctx_destroy(ctx)

    held, want, launches = run(0)
    # meshes, workspaces and layouts, and 64 KB for the task lists
    tight, got, more = run(held + (64 << 10))
    A = oracle.PressureMatrix.from_case(cases[0])
    for c, x in zip(cases, got):
        assert A.residual(c.b, x) <= 1.05e-10
    assert tight <= held and more[0] > launches[0]
