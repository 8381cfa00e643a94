"""The batch's chunk-by-chunk kernel (meshes that do not fit on chip): task
orders, threads per block, epochs that end in the middle of an inner solve, and
the expiry of its grid barrier.

A chunk of a handful of elements still takes a whole group of 32 star records,
so small meshes cut into such chunks are too large for the on-chip layout.  An
inner solve on chip runs to its end in one epoch whatever the epoch's length;
here shorter epochs have to take more launches, which shows that the chunked
kernel ran."""
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
    cases = [S.make_c2(11), S.make_c1(45), S.shuffle_case(S.make_c2(9)), S.make_c1(60)]
    ctx = P.ps_ctx_create(0)
    ms = []
    for c in cases:
        m = P.ps_mesh_upload(ctx, c.dim, c.coords, c.conn, c.dirichlet, chunk_elems=6 if c.dim == 3 else 4)
        P.ps_coeff_set(m, c.alpha, c.beta, c.dt2)
        ms.append(m)
    bs = [torch.as_tensor(c.b, device="cuda") for c in cases]
    yield P, torch, cases, ms, bs
    for m in ms:
        P.ps_mesh_free(m)
    P.ps_ctx_destroy(ctx)


def _solve(env, **kw):
    P, torch, cases, ms, bs = env
    xs = [torch.zeros_like(b) for b in bs]
    st, infos = P.ps_batch_solve(ms, bs, xs, P.make_opts(**kw))
    assert st == P.PS_OK
    return [x.cpu().numpy() for x in xs], infos


def _gate(env, xs):
    for c, x in zip(env[2], xs):
        assert oracle.PressureMatrix.from_case(c).residual(c.b, x) <= 1.05e-10


@pytest.mark.parametrize("threads", [128, 256])
def test_orders_and_epochs_give_the_same_bits(env, threads):
    want, infos = _solve(env, batch_threads=threads, batch_order=0)
    _gate(env, want)
    for order in (0, 1):
        for graph_iters in (1, 32):
            got, other = _solve(env, batch_threads=threads, batch_order=order, graph_iters=graph_iters)
            assert all(np.array_equal(a, b) for a, b in zip(want, got)), (order, graph_iters)
            assert [i.iters_inner for i in other] == [i.iters_inner for i in infos]
            if graph_iters == 1:      # epochs of 8 iterations
                assert other[0].kernel_launches >= 2 * infos[0].kernel_launches


def test_barrier_expiry_is_reported_and_recovered(env):
    P = env[0]
    for order in (0, 1):
        with pytest.raises(P.PressureError) as e:
            _solve(env, batch_order=order, grid_spin_limit=1)
        assert e.value.status == P.PS_ETIMEOUT
        xs, _ = _solve(env, batch_order=order)
        _gate(env, xs)
