"""4pCF kernel at the edges of its tiles and launch rules, against the oracle
bit for bit: complete neighbourhoods whose rows end at, before and after
multiples of 32 (lanes, chunks), every group size (one warp to a whole CTA
per hub), two- and four-byte table entries, plates whose volumes are zero or
so small that single precision cannot sign them."""
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


def clumps(sizes, spread, box_u, seed, flat):
    """Clumps far apart; flat: points on a plate of thickness 0..2 units."""
    rng = np.random.default_rng(seed)
    out = []
    for k, n in enumerate(sizes):
        d = rng.integers(-spread, spread + 1, size=(n, 3))
        if flat:
            d[:, 2] = rng.integers(0, 3, size=n)
        at = np.array([k % 8, (k // 8) % 8, k // 64]) * (box_u // 8) + box_u // 16
        out.append(at + d)
    X = np.concatenate(out)
    return X[rng.permutation(len(X))].astype(np.int32)


def check(gs, X, box_u, edges, pix=(False, True)):
    og = oracle.Graph(X, box_u, edges)
    g = gs.gs_build_graph(X, box_u, edges)
    for p in pix:
        re, ro = og.count_4pcf(pixel=p)
        ge, go = gs.gs_count_4pcf_parity(g, pix=p)
        assert np.array_equal(ge, re) and np.array_equal(go, ro), p
    assert np.array_equal(gs.gs_count_4pcf(g), re)
    return re


@pytest.mark.parametrize("nb", [1, 3, 8, 9])
@pytest.mark.parametrize("flat", [False, True])
@pytest.mark.parametrize("sizes", [[4, 5], [33, 34], [65, 66, 97], [130]])
def test_complete_rows(gs, nb, flat, sizes):
    box_u, spread = 400_000, 3000
    edges = np.linspace(0, 10_500, nb + 1).astype(np.int64)  # wider than a clump's diagonal
    X = clumps(sizes, spread, box_u, 7 * nb + len(sizes), flat)
    total = check(gs, X, box_u, edges).sum()
    assert total == sum(n * (n - 1) * (n - 2) * (n - 3) // 24 for n in sizes)


@pytest.mark.parametrize("n", [7, 61, 121, 251, 361])
def test_group_sizes(gs, n):
    """Mean row lengths on both sides of every rule that picks the warps per
    hub, with one clump of longer rows (the second launch)."""
    box_u = 500_000
    X = clumps([n] * (1 if n > 200 else 4) + [n + n // 2], 2500, box_u, n, False)
    check(gs, X, box_u, np.array([0, 1500, 3000, 5000], dtype=np.int64))


def test_weighted_signed(gs):
    """Weights of both signs on flat clumps: V = 0, cells of either sign."""
    box_u = 400_000
    X = clumps([40, 70], 3000, box_u, 5, True)
    rng = np.random.default_rng(6)
    w = (rng.uniform(0.5, 1.5, len(X)) * np.where(rng.random(len(X)) < 0.5, -1, 1)).astype(np.float32)
    edges = np.array([0, 2000, 4000, 6000, 10_500], dtype=np.int64)
    og = oracle.Graph(X, box_u, edges)
    g = gs.gs_build_graph(X, box_u, edges)
    for pix in (False, True):
        ref = og.count_4pcf(w, pixel=pix)
        got = gs.gs_count_4pcf_parity(g, w, pix=pix)
        for a, b in zip(got, ref):
            assert np.array_equal(a, b)
