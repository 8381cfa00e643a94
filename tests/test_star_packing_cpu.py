"""Star patches of 2D meshes (no GPU): every element lies in exactly one star
whatever the vertices' degrees."""
import numpy as np
import pytest

from paper_2301_08357_gb300 import synthetic as S


@pytest.fixture(scope="module")
def P():
    from paper_2301_08357_gb300 import build
    build.build()
    from paper_2301_08357_gb300 import pressure
    return pressure


def _fan(k):
    """k triangles around one vertex."""
    t = 2 * np.pi * np.arange(k) / k
    X = np.vstack([[0.0, 0.0], np.c_[np.cos(t), np.sin(t)]])
    C = np.array([[0, 1 + j, 1 + (j + 1) % k] for j in range(k)], dtype=np.int32)
    return X, C


def _delaunay(n, seed):
    from scipy.spatial import Delaunay
    X = np.random.default_rng(seed).random((n, 2))
    C = Delaunay(X).simplices.astype(np.int32)
    a, b, c = X[C[:, 0]], X[C[:, 1]], X[C[:, 2]]
    area = (b - a)[:, 0] * (c - a)[:, 1] - (b - a)[:, 1] * (c - a)[:, 0]
    C = C[np.abs(area) > 1e-9]
    used = np.unique(C)
    new = np.full(n, -1, np.int32)
    new[used] = np.arange(used.size)
    return X[used], new[C]


@pytest.mark.parametrize("make", [lambda: _fan(3), lambda: _fan(7), lambda: _fan(14), lambda: _fan(61),
                                  lambda: _delaunay(40, 1), lambda: _delaunay(3000, 2)],
                         ids=["fan3", "fan7", "fan14", "fan61", "delaunay40", "delaunay3000"])
@pytest.mark.parametrize("chunk", [0, 40, 1536])
def test_irregular_meshes_hold_the_layout_rules(P, make, chunk):
    X, C = make()
    X, C = np.ascontiguousarray(X), np.ascontiguousarray(C, dtype=np.int32)
    # (the call checks every rule of the layout and raises at the first fault)
    st = P.ps_debug_prepare(2, X, C, np.zeros(len(X), np.uint8), chunk_elems=chunk)
    assert st.n_elems == len(C)


def test_squares_and_shuffled_squares(P):
    for c in (S.make_c1(37), S.shuffle_case(S.make_c1(37))):
        st = P.ps_debug_prepare(2, c.coords, c.conn, c.dirichlet, chunk_elems=1536)
        assert st.n_elems == c.conn.shape[0]
