"""Row pass of the graph build at the edges of its cell grid, against the oracle
edge for edge: the three ways of splitting cells, boxes just wider than four
E_nb and as wide as allowed (coordinate differences modulo 2^32), open boxes,
cells of one to many hubs, rows filled in chunks. And the pair kernel's table
of configurations, which only uneven bins reach now."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_parity import edge_set_from_gpu, edge_set_from_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gs():
    import torch
    assert torch.cuda.is_available()
    import paper_2607_06604_gb300 as m
    return m


def points(kind, n, box):
    rng = np.random.default_rng(n)
    X = rng.integers(0, box, size=(n, 3))
    if kind == "faces":  # most points near a face, some on it
        X[::2] = np.where(rng.random((len(X[::2]), 3)) < 0.5, X[::2] % 3000, box - 1 - X[::2] % 3000)
        X[::20] = np.where(X[::20] < box // 2, 0, box - 1)
    if kind == "uneven":  # a few dense cells beside empty ones
        X[: n // 2] = box // 3 + rng.integers(-200, 201, size=(n // 2, 3))
    return np.mod(X, box).astype(np.int32)


# cells of side E_nb; n against their number decides the split: (1, 1, 1), (2, 1, 1), (4, 2, 2)
@pytest.mark.parametrize("kind", ["uniform", "faces", "uneven"])
@pytest.mark.parametrize("n,box,rmax", [
    (300, 40_005, 10_000), (600, 40_001, 10_000), (4000, 40_001, 10_000), (3000, 400_003, 40_000),
    (6001, 90_000, 10_000), (5001, 2**31 - 1, 2**19 - 1), (6001, 2_200_000, 2**19 - 1)])
@pytest.mark.parametrize("windows", [0, 3])
def test_rows(gs, kind, n, box, rmax, windows):
    X = points(kind, n, box)
    edges = np.array([0, rmax // 7, rmax // 2, rmax], dtype=np.int64)
    for box_u in (box, 0):
        if not box_u and box > 1 << 30:
            X = (X.astype(np.int64) % (1 << 30)).astype(np.int32)  # an open box's limit
        g = gs.gs_build_graph(X, box_u, edges, force_windows=windows)
        ref = edge_set_from_oracle(oracle.Graph(X, box_u, edges))
        got, deg, ptr, nbr = edge_set_from_gpu(gs, g)
        assert np.array_equal(got, ref)
        assert all(np.all(np.diff(nbr[p:p + d]) > 0) for p, d in zip(ptr[:-1], deg))
        info = gs.gs_graph_info(g)
        assert info["edges"] == len(ref) and info["max_degree"] == deg.max()


@pytest.mark.parametrize("edges", [
    np.array([0, 1500, 2000, 4000, 4100, 9000]),  # buckets, none linear
    np.array([0, 1, 2, 9000]),                    # bins too narrow for buckets
    np.arange(64) * 140,                          # more even bins than the tiles take
])
def test_pair_kernel_of_uneven_bins(gs, edges):
    edges = edges.astype(np.int64)
    rng = np.random.default_rng(len(edges))
    X = rng.integers(0, 60_000, size=(4000, 3)).astype(np.int32)
    X[:500] = 30_000 + rng.integers(-1500, 1501, size=(500, 3))
    w = (rng.uniform(0.5, 1.5, len(X)) * np.where(rng.random(len(X)) < 0.4, -1, 1)).astype(np.float32)
    for box_u in (60_000, 0):
        rc, rw = oracle.Graph(X, box_u, edges).count_3pcf(w)
        g = gs.gs_build_graph(X, box_u, edges)
        for variant in (0, 4):
            assert np.array_equal(gs.gs_count_3pcf(g, variant=variant), rc)
            c, s = gs.gs_count_3pcf(g, w, variant=variant)
            assert np.array_equal(c, rc) and np.array_equal(s, rw)
