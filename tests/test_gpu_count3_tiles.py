"""Tiled pair kernel (3pCF with evenly spaced bins) at the edges of its tiles
and launch rules, against the oracle bit for bit: rows around multiples of 32,
every group size, rows beyond the shared staging, pairs exactly on bin edges
(which single precision cannot place), coincident points, bins that start
above zero or are rounded to the lattice, and weights of every width and sign
the exact sums take."""
import numpy as np
import pytest

import catalogs
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gs():
    import torch
    assert torch.cuda.is_available()
    import paper_2607_06604_gb300 as m
    return m


def weights(kind, n, seed):
    rng = np.random.default_rng(seed)
    if kind == "one":
        return np.ones(n, np.float32)
    w = rng.uniform(0.5, 1.5, n)
    if kind == "signed":
        w *= np.where(rng.random(n) < 0.4, -1.0, 1.0)
    if kind == "span":  # the full 30 bits of the direct path
        w = 2.0 ** rng.uniform(-4.9, 0.0, n) * np.where(rng.random(n) < 0.5, -1.0, 1.0)
    return w.astype(np.float32)


def check(gs, X, box_u, edges, kinds=("uniform",), **opts):
    og = oracle.Graph(X, box_u, edges)
    g = gs.gs_build_graph(X, box_u, edges, **opts)
    ref = og.count_3pcf()
    assert np.array_equal(gs.gs_count_3pcf(g), ref)
    for k, kind in enumerate(kinds):
        w = weights(kind, len(X), 40 + k)
        rc, rw = og.count_3pcf(w)
        gc, gw = gs.gs_count_3pcf(g, w)
        assert np.array_equal(gc, rc) and np.array_equal(gw, rw), kind
        (bc, bw), = gs.gs_count_3pcf_batch([g], [w])
        assert np.array_equal(bc, rc) and np.array_equal(bw, rw), kind
    (bc, _), = gs.gs_count_3pcf_batch([g])
    assert np.array_equal(bc, ref)
    return ref


@pytest.mark.parametrize("n", [3, 32, 33, 34, 64, 65, 97, 129, 300])
def test_complete_rows(gs, n):
    rng = np.random.default_rng(n)
    X = (50_000 + rng.integers(-2500, 2501, size=(n, 3))).astype(np.int32)
    edges = 2560 * np.arange(5, dtype=np.int64)  # wider than the clump's diagonal
    ref = check(gs, X, 200_000, edges, ("uniform", "signed", "span"))
    assert ref.sum() == n * (n - 1) * (n - 2) // 6


@pytest.mark.parametrize("edges", [
    1000 * np.arange(8),                                # pairs on every edge
    np.array([0, 999, 2001, 3000, 4000, 5001, 6000]),   # rounded edges
    np.array([1000, 2000, 3000, 4000, 5000]),           # bins from above zero
    np.array([700, 2100, 3500, 4900, 6300, 7700]),
])
@pytest.mark.parametrize("box_u", [0, 64_000])
def test_pairs_on_bin_edges(gs, edges, box_u):
    """A lattice of spacing 1000 (some points off by one, some twice): most
    axis-parallel pairs lie on, just below or just above an edge."""
    rng = np.random.default_rng(len(edges))
    at = np.stack(np.meshgrid(*[np.arange(12)] * 3, indexing="ij"), -1).reshape(-1, 3) * 1000
    X = at[rng.permutation(len(at))[:900]]
    X = np.concatenate([X, X[:300] + rng.integers(-1, 2, size=(300, 3)), X[:40]])
    X = np.mod(X + 60_000 if box_u else X + 5000, box_u or 1 << 20).astype(np.int32)
    check(gs, X, box_u, edges.astype(np.int64), ("signed",))


@pytest.mark.parametrize("mean", [6, 50, 120, 250, 500])
def test_group_sizes(gs, mean):
    """Mean row lengths on both sides of every rule that picks the warps per
    hub, with a clump of longer rows (global staging)."""
    box_u = 100 * 1024
    rng = np.random.default_rng(mean)
    rmax = 12_000
    n = int(2 * mean * box_u ** 3 / (4.18879 * rmax ** 3)) if mean < 400 else 9000
    X = np.concatenate([rng.integers(0, box_u, size=(n, 3)),
                        50_000 + rng.integers(-3000, 3001, size=(5 * mean, 3))]).astype(np.int32)
    nb = 6
    check(gs, X, box_u, np.linspace(0, rmax, nb + 1).astype(np.int64), ("uniform",))


@pytest.mark.parametrize("nb", [1, 2, 13, 22, 30])
def test_bin_counts(gs, nb):
    box_u = 60 * 1024
    X = oracle.quantize(catalogs.neyman_scott(4000, 60.0, seed=nb, sigma=1.5), box_u, True)
    check(gs, X, box_u, catalogs.bin_edges_u(0.0, 9.0, nb), ("one", "signed"))


def test_batch_of_unequal_catalogues_and_windows(gs):
    box_u = 80 * 1024
    edges = catalogs.bin_edges_u(0.0, 9.0, 7)
    Xs = [oracle.quantize(catalogs.neyman_scott(n, 80.0, seed=n, sigma=1.5), box_u, True)
          for n in (5, 900, 7000, 40, 3001)]
    ws = [weights("signed", len(X), 3) for X in Xs]
    graphs = [gs.gs_build_graph(X, box_u, edges) for X in Xs]
    refs = [oracle.Graph(X, box_u, edges).count_3pcf(w) for X, w in zip(Xs, ws)]
    for (c, _), (rc, _) in zip(gs.gs_count_3pcf_batch(graphs), refs):
        assert np.array_equal(c, rc)
    for (c, s), (rc, rw) in zip(gs.gs_count_3pcf_batch(graphs, ws), refs):
        assert np.array_equal(c, rc) and np.array_equal(s, rw)
    g = gs.gs_build_graph(Xs[2], box_u, edges, force_windows=3)
    c, s = gs.gs_count_3pcf(g, ws[2])
    assert np.array_equal(c, refs[2][0]) and np.array_equal(s, refs[2][1])
    parts = [gs.gs_count_3pcf(graphs[2], shard=k, shards=3) for k in range(3)]
    assert np.array_equal(sum(parts), refs[2][0])


@pytest.mark.parametrize("n", [33, 64, 130])
@pytest.mark.parametrize("nmu", [1, 5, 62, 64])
@pytest.mark.parametrize("flat", [False, True])
def test_mu_rows_and_degenerate_normals(gs, n, nmu, flat):
    """Rows around multiples of 32; a coarse lattice (normals exactly on mu
    edges, collinear and coincident points) or a plate two units thick."""
    rng = np.random.default_rng(n + nmu)
    d = rng.integers(-2, 3, size=(n, 3)) * 800
    if flat:
        d = rng.integers(-2500, 2501, size=(n, 3))
        d[:, 1] = rng.integers(0, 3, size=n)
    X = (50_000 + d).astype(np.int32)
    for edges in (1600 * np.arange(6), np.array([500, 1901, 3300, 4700, 6100])):
        edges = edges.astype(np.int64)
        ref = oracle.Graph(X, 200_000, edges).count_3pcf_mu(nmu)
        ref = ref[0] if isinstance(ref, tuple) else ref
        got = gs.gs_count_3pcf_mu(gs.gs_build_graph(X, 200_000, edges), nmu)
        assert np.array_equal(got, np.asarray(ref).reshape(got.shape))


@pytest.mark.parametrize("n", [2, 33, 64, 130, 700])
@pytest.mark.parametrize("kind", ["uniform", "signed", "span"])
def test_equilateral_and_weighted_pairs(gs, n, kind):
    """One, few and many neighbours per bin, pairs exactly on bin edges, uneven
    bins, more bins than lanes."""
    rng = np.random.default_rng(n)
    X = (50_000 + np.concatenate([rng.integers(-3, 4, size=(n // 2, 3)) * 1000,
                                  rng.integers(-2500, 2501, size=(n - n // 2, 3))])).astype(np.int32)
    w = weights(kind, len(X), 9)
    for edges in (np.array([0, 20_000]), 1000 * np.arange(12), np.array([0, 700, 1000, 5000, 5001, 9000]),
                  np.linspace(0, 11_000, 41)):
        edges = edges.astype(np.int64)
        og = oracle.Graph(X, 200_000, edges)
        g = gs.gs_build_graph(X, 200_000, edges)
        rc, rw = oracle.equilateral_3pcf(og, w)
        assert np.array_equal(gs.gs_count_3pcf_equilateral(g), rc)
        gc, gw = gs.gs_count_3pcf_equilateral(g, w)
        assert np.array_equal(gc, rc) and np.array_equal(gw, rw)
        rr = np.ones(len(edges) - 1)
        rp, rsum = og.pairs(w)
        gp, gxi, _ = gs.gs_disconnected_4pcf(g, w, rr=rr, zeta=False)
        assert np.array_equal(gp, rp) and np.array_equal(gxi, rsum - 1.0)
