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


def _vectors(st):
    """At most these bytes of solver vectors, partial sums and dot products."""
    sh = st.chunk_node_refs - (st.n_nodes - st.n_shared) + 3 * st.n_chunks
    return (st.n_nodes + 4096) * (5 * 8 + 12 * 4) + sh * 16 + st.n_chunks * 48


def test_only_meshes_with_a_layout_of_their_own_are_charged_for_one(env):
    P, torch = env
    ctx = P.ps_ctx_create(0)
    try:
        small, large = S.make_c2(24), S.make_c2(72)
        ms = [P.ps_mesh_upload(ctx, c.dim, c.coords, c.conn, c.dirichlet, chunk_elems=1536) for c in (small, large)]
        st = [P.ps_mesh_get_stats(m) for m in ms]
        assert st[0].solve_bytes > _vectors(st[0]) - 4096 * 88        # a layout of its own in a batch
        assert st[1].solve_bytes <= _vectors(st[1])                   # too large for one
        # requests that the server solves alone need none either
        P.ps_coeff_set(ms[0], small.alpha, small.beta, small.dt2)
        srv = P.ps_server_create(ctx, opts=P.make_opts(), single_nodes=1000, hbm_budget_bytes=_vectors(st[0]))
        try:
            t = P.ps_solve_submit(srv, P.ps_server_add_case(srv, ms[0]), small.b)
            status, info = P.ps_solve_wait(srv, t)
            assert status == P.PS_OK and P.ps_server_get_stats(srv).single_solves == 1
        finally:
            P.ps_server_destroy(srv)
        for m in ms:
            P.ps_mesh_free(m)
    finally:
        P.ps_ctx_destroy(ctx)
