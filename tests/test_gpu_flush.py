"""Shared counters emptied by one group of warps while the others count on:
variant 1024 flushes before every hub, on catalogues whose counts the kernels
decide in integers (points on a mesh or in planes: volumes of zero, pairs on
bin edges), with one warp to half a CTA per hub. Against the oracle bit for
bit."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gs():
    import torch
    assert torch.cuda.is_available()
    import paper_2607_06604_gb300 as m
    return m


def mesh(m):
    at = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3) * 1000
    return at.astype(np.int32), m * 1000


def planes(n, box_u):
    """Uniform points on planes 2,500 apart."""
    X = np.random.default_rng(n).integers(0, box_u, size=(n, 3))
    X[:, 2] = X[:, 2] // 2500 * 2500
    return X.astype(np.int32), box_u


def patch(n, box_u):
    """Uniform points, one in 20 on a plane."""
    X = np.random.default_rng(n).integers(0, box_u, size=(n, 3))
    X[::20, 2] = 5000
    return X.astype(np.int32), box_u


# rows of about 15, 27, 60 and 100: 1, 4, 8 and 16 warps per hub
CATALOGUES = [(mesh, (20,), 2100), (mesh, (18,), 2300), (mesh, (14,), 3100), (mesh, (15,), 3700),
              (planes, (7000, 40_000), 4000), (planes, (13_000, 40_000), 4000),
              (planes, (12_000, 30_000), 4000), (planes, (3700, 17_000), 4000)]


@pytest.mark.parametrize("kind,args,rmax", CATALOGUES)
def test_parity_flush_between_groups(gs, kind, args, rmax):
    X, box_u = kind(*args)
    edges = np.linspace(0, rmax, 6).astype(np.int64)
    re, ro = oracle.Graph(X, box_u, edges).count_4pcf()
    g = gs.gs_build_graph(X, box_u, edges)
    for _ in range(3):
        ge, go = gs.gs_count_4pcf_parity(g, variant=1024)
        assert np.array_equal(ge, re) and np.array_equal(go, ro)
    assert np.array_equal(gs.gs_count_4pcf(g, variant=1024), re)


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("kind,args,rmax", CATALOGUES)
@pytest.mark.parametrize("rmin", [0, 1000])
def test_3pcf_flush_between_groups(gs, kind, args, rmax, rmin, weighted):
    """Bins of 200 units: on the mesh many pairs lie on an edge."""
    X, box_u = kind(*args)
    edges = np.arange(rmin, rmax + 1, 200, dtype=np.int64)
    og, g = oracle.Graph(X, box_u, edges), gs.gs_build_graph(X, box_u, edges)
    if weighted:
        rng = np.random.default_rng(3)
        w = (rng.uniform(0.5, 1.5, len(X)) * np.where(rng.random(len(X)) < 0.4, -1, 1)).astype(np.float32)
        rc, rw = og.count_3pcf(w)
        for _ in range(3):
            c, s = gs.gs_count_3pcf(g, w, variant=1024)
            assert np.array_equal(c, rc) and np.array_equal(s, rw)
    else:
        ref = og.count_3pcf()
        for _ in range(3):
            assert np.array_equal(gs.gs_count_3pcf(g, variant=1024), ref)


@pytest.mark.parametrize("nb", [3, 5, 9])
@pytest.mark.parametrize("kind,args,rmax", [CATALOGUES[k] for k in (0, 2, 4, 6)] + [
    (planes, (3, 17_000), 4000), (planes, (12, 17_000), 4000), (planes, (150, 17_000), 4000),
    (patch, (1000, 17_000), 4000)])
def test_volumes_of_zero(gs, kind, args, rmax, nb):
    """V = 0 tetrahedra in even and odd numbers per orbit, unweighted (all orbits
    or 64 in shared memory, rows in global memory) and with weights of both
    signs (cells for V = 0 on planes and meshes, none for a few coplanar points
    among others)."""
    X, box_u = kind(*args)
    edges = np.linspace(0, rmax, nb + 1).astype(np.int64)
    og, g = oracle.Graph(X, box_u, edges), gs.gs_build_graph(X, box_u, edges)
    rng = np.random.default_rng(8)
    w = (rng.uniform(0.5, 1.5, len(X)) * np.where(rng.random(len(X)) < 0.5, -1, 1)).astype(np.float32)
    for pix in (False, True):
        ref = og.count_4pcf(w, pixel=pix)
        for variant in (0, 1, 8, 1024, 1024 + 8):
            got = gs.gs_count_4pcf_parity(g, w, pix=pix, variant=variant)
            for a, b in zip(got, ref):
                assert np.array_equal(a, b), (pix, variant)
            got = gs.gs_count_4pcf_parity(g, pix=pix, variant=variant)
            assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1]), (pix, variant)


@pytest.mark.parametrize("signed", [False, True])
@pytest.mark.parametrize("nb", [5, 10, 12])
def test_orbits_without_shared_cells(gs, nb, signed):
    """Weighted sums of orbits that have no cells in shared memory: 64 orbits in
    it (variant 8), launches of 256 hubs (1024), weights of the full 30 bits."""
    X, box_u = planes(3000, 17_000) if nb == 5 else patch(2500, 17_000)
    edges = np.linspace(0, 4000, nb + 1).astype(np.int64)
    og, g = oracle.Graph(X, box_u, edges), gs.gs_build_graph(X, box_u, edges)
    rng = np.random.default_rng(nb)
    w = 2.0 ** rng.uniform(-4.9, 0.0, len(X)) * np.where(rng.random(len(X)) < 0.5 * signed, -1.0, 1.0)
    w = w.astype(np.float32)
    ref = og.count_4pcf(w)
    for variant in (0, 8, 1024, 1024 + 8):
        for a, b in zip(gs.gs_count_4pcf_parity(g, w, variant=variant), ref):
            assert np.array_equal(a, b), variant
        even, weven = gs.gs_count_4pcf(g, w, variant=variant)
        assert np.array_equal(even, ref[0]) and np.array_equal(weven, ref[2]), variant


def test_weighted_rows_beyond_352(gs):
    """Few bins: all orbits have shared cells beside the workspace of rows of
    more than 352."""
    X = (50_000 + np.random.default_rng(2).integers(-2500, 2501, size=(368, 3))).astype(np.int32)
    edges = np.array([0, 4000, 9000], dtype=np.int64)
    w = np.random.default_rng(3).uniform(0.5, 1.5, len(X)).astype(np.float32)
    g = gs.gs_build_graph(X, 200_000, edges)
    assert gs.gs_graph_info(g)["max_degree"] > 352
    for a, b in zip(gs.gs_count_4pcf_parity(g, w), oracle.Graph(X, 200_000, edges).count_4pcf(w)):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("n", [500, 511, 520, 2040, 2060])
@pytest.mark.parametrize("kind", ["span", "uniform"])
def test_3pcf_rows_at_the_count_fields_limit(gs, n, kind):
    """Complete rows on both sides of the lengths up to which the weighted tiles
    can count pairs beside the sums (512 for weights of 30 bits, 2,048 for weights
    within a factor of two)."""
    rng = np.random.default_rng(n)
    X = (50_000 + rng.integers(-2500, 2501, size=(n, 3))).astype(np.int32)
    edges = 2560 * np.arange(5, dtype=np.int64)
    w = 2.0 ** rng.uniform(-4.9, 0.0, n) * np.where(rng.random(n) < 0.5, -1, 1) if kind == "span" \
        else rng.uniform(0.5, 1.5, n)
    w = w.astype(np.float32)
    rc, rw = oracle.Graph(X, 200_000, edges).count_3pcf(w)
    c, s = gs.gs_count_3pcf(gs.gs_build_graph(X, 200_000, edges), w)
    assert np.array_equal(c, rc) and np.array_equal(s, rw)
