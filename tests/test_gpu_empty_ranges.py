"""Calls without a hub to count (no points, one point, shards that get no hub):
all results are zero, on the paths that relabel orbits too."""
import numpy as np
import pytest

import catalogs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gs():
    import torch
    assert torch.cuda.is_available()
    import paper_2607_06604_gb300 as m
    return m


@pytest.mark.parametrize("nb", [2, 8, 10])
@pytest.mark.parametrize("n", [0, 1, 2])
def test_no_hubs(gs, n, nb):
    X = np.full((n, 3), 5000, np.int32)
    w = np.ones(n, np.float32)
    g = gs.gs_build_graph(X, 100_000, catalogs.bin_edges_u(0.0, 9.0, nb))
    for opts in ({}, dict(shard=3, shards=4), dict(shard=0, shards=4), dict(variant=8)):
        for pix in (False, True):
            outs = list(gs.gs_count_4pcf_parity(g, pix=pix, **opts))
            if n:
                outs += gs.gs_count_4pcf_parity(g, w, pix=pix, **opts)
            assert all(not o.any() for o in outs)
        outs = [gs.gs_count_4pcf(g, **opts)]
        if n:
            outs += list(gs.gs_count_4pcf(g, w, **opts)) + list(gs.gs_count_3pcf(g, w, **opts))
        assert all(not o.any() for o in outs)
