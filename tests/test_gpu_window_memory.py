"""Device memory of calls on graphs streamed in windows: what a call allocates
for long rows does not grow with the number of windows."""
import threading

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_mod():
    import torch
    assert torch.cuda.is_available()
    return torch


@pytest.fixture(scope="module")
def gs():
    import paper_2607_06604_gb300 as m
    return m


def stars(n_stars, rays):
    """Background points and, per star, a hub with `rays` neighbours on the half
    sphere ahead of it in x."""
    rng = np.random.default_rng(5)
    box_u, r = 200_000, 9500
    out = [rng.integers(0, box_u, size=(20_000, 3))]
    for k in range(n_stars):
        at = np.array([(2 * k + 1) * box_u // (2 * n_stars), 100_000, 100_000])
        d = rng.normal(size=(rays, 3))
        d *= r / np.linalg.norm(d, axis=1)[:, None]
        d[:, 0] = np.abs(d[:, 0])
        out += [at[None], at + np.rint(d).astype(np.int64)]
    return np.mod(np.concatenate(out), box_u).astype(np.int32), box_u


def peak(torch, call):
    """Most device memory taken during call(), sampled beside it."""
    torch.cuda.synchronize()
    base = low = torch.cuda.mem_get_info()[0]
    done = threading.Event()

    def sample():
        nonlocal low
        while not done.is_set():
            low = min(low, torch.cuda.mem_get_info()[0])

    t = threading.Thread(target=sample)
    t.start()
    out = call()
    low = min(low, torch.cuda.mem_get_info()[0])
    done.set()
    t.join()
    torch.cuda.synchronize()
    return out, base - low


def test_4pcf_workspace_is_one_for_all_windows(gs, torch_mod):
    """Variant 1: every hub's workspace is in global memory, 152 CTAs of
    more than 1,000^2 / 2 bytes."""
    X, box_u = stars(8, 1500)
    edges = np.array([9000, 9400, 10_000], dtype=np.int64)
    ref = oracle.Graph(X, box_u, edges).count_4pcf()
    used = {}
    for windows in (2, 2, 10):
        g = gs.gs_build_graph(X, box_u, edges, force_windows=windows)
        info = gs.gs_graph_info(g)
        assert info["windows"] >= windows and info["max_degree"] > 1000
        for variant in (0, 1):
            got, used[windows] = peak(torch_mod, lambda: gs.gs_count_4pcf_parity(g, variant=variant))
            assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])
    assert used[2] > 80 << 20
    assert used[10] < 1.25 * used[2] + (32 << 20), used


def test_streamed_calls_fit_beside_little_memory(gs, torch_mod):
    """Rows of thousands beside short ones: the staging for long rows of every
    group of warps would take 0.6 GB and makes do with less, but only after the
    window buffers (2 of 60 MB) are there."""
    torch = torch_mod
    rng = np.random.default_rng(6)
    box_u = 1_000_000
    X = np.concatenate([rng.integers(0, box_u, size=(400_000, 3)),
                        500_000 + rng.integers(-1500, 1501, size=(6500, 3))]).astype(np.int32)
    edges = np.array([0, 2500, 5000], dtype=np.int64)
    g = gs.gs_build_graph(X, box_u, edges, force_windows=2)
    info = gs.gs_graph_info(g)
    assert info["max_degree"] > 6000 and info["edges"] / len(X) < 64
    w = rng.uniform(0.5, 1.5, len(X)).astype(np.float32)
    calls = [lambda: gs.gs_count_3pcf(g), lambda: gs.gs_count_3pcf_mu(g, 2),
             lambda: gs.gs_count_3pcf_equilateral(g), lambda: gs.gs_count_3pcf_equilateral(g, w)[1]]
    refs = [c() for c in calls]
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    for spare in (240, 300, 360, 480):  # MB
        free = torch.cuda.mem_get_info()[0]
        held = torch.empty(free - (spare << 20), dtype=torch.uint8, device="cuda")
        for call, ref in zip(calls, refs):
            assert np.array_equal(call(), ref), spare
        del held
        torch.cuda.empty_cache()


def test_wide_weights_hold_one_evaluations_scratch(gs, torch_mod):
    """Wide weights make five weighted 4pCF evaluations; their scratch (hundreds of
    MB at 14 bins) is that of one."""
    rng = np.random.default_rng(8)
    X = rng.integers(0, 60_000, size=(3000, 3)).astype(np.int32)
    edges = np.linspace(0, 9000, 15).astype(np.int64)
    g = gs.gs_build_graph(X, 60_000, edges)
    narrow = rng.uniform(0.5, 1.5, len(X)).astype(np.float32)
    wide = (2.0 ** rng.uniform(-9, 1, len(X))).astype(np.float32)
    gs.gs_count_4pcf_parity(g, narrow)
    one = peak(torch_mod, lambda: gs.gs_count_4pcf_parity(g, narrow))[1]
    got, five = peak(torch_mod, lambda: gs.gs_count_4pcf_parity(g, wide))
    for a, b in zip(got, oracle.Graph(X, 60_000, edges).count_4pcf(wide)):
        assert np.array_equal(a, b)
    # beside it the evaluations' own sums, 10 x 24 bytes an orbit
    orbits = gs.gs_num_configs(4, 14)
    assert five < 1.3 * one + 240 * orbits + (64 << 20), (one, five)
