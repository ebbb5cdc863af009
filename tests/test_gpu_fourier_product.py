"""tau -> iw on a non-equidistant grid: the product with the Fourier weights (exact
digit products) and the FFTs that serve captures and large grids, both against the
oracle, at the edges of their tiles: one to three blocks of 256 nodes, frequency
counts around the blocks of 32, matrices of 1 to 169 elements (128-row tiles).

Tolerance: the weights and the samples are rounded once, the sums are exact to
2^-56 of the largest product per block, and the oracle's weights carry a phase error
of up to theta 2^-53 (theta = w h of the longest interval, at most a few hundred);
2^-44 of the sum of absolute terms covers both.
"""

import numpy as np
import pytest
import torch

from oracle import grids
from oracle import transforms as ot

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import os

    import paper_1405_3273_gb300 as g
    from paper_1405_3273_gb300 import build
    if not os.path.exists(g.LIB_PATH):
        build.build()
    g.lib()
    return g


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def both_paths(g, n, M, idx, n_iw, beta, X):
    """(product, FFT): the first call of a context under capture cannot build the planes."""
    Xd, out = dev(X), torch.zeros(n_iw, n, n, dtype=torch.complex128, device="cuda")
    with g.Context(n, None, n_iw, beta, grid=(M, idx)) as ctx:
        graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=side):
            g.gf2_set_stream(ctx.handle)
            g.gf2_fft_tau_to_iw(ctx.handle, Xd, out)
        graph.replay()
        torch.cuda.synchronize()
        fft = out.cpu().numpy()
        out.zero_()
        g.gf2_set_stream(ctx.handle)
        g.gf2_fft_tau_to_iw(ctx.handle, Xd, out)
        return out.cpu().numpy(), fft


@pytest.mark.parametrize("n,p,u,n_iw", [(1, 2, 2, 1), (5, 2, 2, 31), (12, 3, 8, 32), (13, 3, 8, 33), (4, 7, 16, 300),
                                        (4, 3, 32, 64), (3, 7, 32, 1000)])
def test_product_and_ffts_match_oracle(g, n, p, u, n_iw):
    M, idx = grids.power_mesh(p, u)
    beta = 40.0
    X = np.random.default_rng(n * 1000 + n_iw).uniform(-1.0, 1.0, (len(idx), n, n))
    X[:, 0, 0] *= 10.0 ** -np.arange(len(idx), dtype=float).clip(max=30)  # one element over many decades
    ref = ot.tau_to_iw_grid(X, beta, M, idx, n_iw)
    size = ot.tau_to_iw_grid(np.abs(X), beta, M, idx, 1)  # |weights| <= those of the lowest frequency, up to the cubic's 1.6
    bound = 2.0 ** -44 * 2.0 * np.abs(size[0]).max()
    for got in both_paths(g, n, M, idx, n_iw, beta, X):
        assert np.abs(got - ref).max() <= bound


def test_non_finite_sample_reaches_its_element_only(g):
    M, idx = grids.power_mesh(3, 8)
    X = np.random.default_rng(5).uniform(-1.0, 1.0, (len(idx), 4, 4))
    X[7, 1, 2] = np.inf
    got, _ = both_paths(g, 4, M, idx, 50, 10.0, X)
    bad = np.zeros((4, 4), bool)
    bad[1, 2] = True
    assert not np.isfinite(got[:, 1, 2]).any() and np.isfinite(got[:, ~bad]).all()


def test_large_frequency_count_takes_the_ffts(g):
    """n_tau n_iw beyond the product's range: the same numbers as a context within it."""
    M, idx, n = 64, list(range(65)), 3
    X = np.random.default_rng(6).uniform(-1.0, 1.0, (65, n, n))
    outs = []
    for n_iw in (300, 3000):
        with g.Context(n, None, n_iw, 10.0, grid=(M, idx)) as ctx:
            o = torch.empty(n_iw, n, n, dtype=torch.complex128, device="cuda")
            g.gf2_fft_tau_to_iw(ctx.handle, dev(X), o)
            outs.append(o.cpu().numpy()[:300])
    assert np.abs(outs[0] - outs[1]).max() <= 2.0 ** -44 * np.abs(outs[0]).max()


@pytest.mark.parametrize("p,u", [(11, 2), (9, 8), (7, 32), (12, 1)])
def test_end_nodes_of_steep_meshes_keep_their_digits(g, p, u):
    """Single samples at the ends, where the intervals are up to 2^11 times shorter than in the
    middle: X(i w_n) is that node's weight.  It is made of at most three intervals of
    similar length with w h < 1, so neither the oracle's sum nor the library's cancels:
    a few dozen roundings, 2^-47 of its size, cover both."""
    M, idx = grids.power_mesh(p, u)
    beta, n_iw, n, nt = 100.0, 8, 2, len(idx)
    X = np.zeros((nt, n * n))
    X[0, 0], X[-1, 1], X[1, 2], X[-2, 3] = 1.0, -1.0, 3.0, 1e-9
    X = X.reshape(nt, n, n)
    ref = ot.tau_to_iw_grid(X, beta, M, idx, n_iw)
    got, _ = both_paths(g, n, M, idx, n_iw, beta, X)
    assert np.all(np.abs(got - ref) <= 2.0 ** -47 * np.abs(ref))


def test_first_call_beside_a_capture_on_another_stream(g):
    """The first call of a context builds its planes also while another stream is under capture
    in the strictest mode, and leaves that capture alone."""
    M, idx = grids.power_mesh(11, 2)
    X = np.random.default_rng(7).uniform(-1.0, 1.0, (len(idx), 3, 3))
    Xd, out = dev(X), torch.zeros(50, 3, 3, dtype=torch.complex128, device="cuda")
    y, own, side = torch.zeros(4, device="cuda"), torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(own):
        ctx = g.Context(3, None, 50, 10.0, grid=(M, idx))
    with ctx:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side, capture_error_mode="global"):
            y.add_(1.0)
            g.gf2_fft_tau_to_iw(ctx.handle, Xd, out)  # on the context's stream, not captured
            y.add_(1.0)
        torch.cuda.synchronize()
        first = out.cpu().numpy()
        graph.replay()
        g.gf2_fft_tau_to_iw(ctx.handle, Xd, out)
        torch.cuda.synchronize()
    assert np.array_equal(first, out.cpu().numpy()) and float(y[0]) == 2.0
    assert np.abs(first - ot.tau_to_iw_grid(X, 10.0, M, idx, 50)).max() <= 2.0 ** -44 * np.abs(first).max()


def test_the_rule_takes_the_faster_way(g):
    """Few elements on a short grid go through the FFTs, short meshes with many frequencies and
    long ones through the product; the slower way takes at least 1.3 times as long."""
    import ctypes
    f = g.lib().gf2_test_fourier_path
    f.argtypes, f.restype = [ctypes.c_void_p, ctypes.c_int], ctypes.c_int
    for n, (p, u), n_iw, product in ((10, (2, 64), 256, False), (4, (3, 8), 64, False), (32, (3, 8), 8192, True),
                                     (4, (7, 32), 256, True), (64, (2, 64), 2048, True)):
        M, idx = grids.power_mesh(p, u)
        X = torch.randn(len(idx), n, n, dtype=torch.float64, device="cuda")
        out = torch.empty(n_iw, n, n, dtype=torch.complex128, device="cuda")
        us = []
        with g.Context(n, None, n_iw, 40.0, grid=(M, idx)) as ctx:
            for path in (0, 1, 2):
                assert f(ctx.handle, path) == 0
                best = []
                for _ in range(9):
                    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                    a.record()
                    for _ in range(8):
                        g.gf2_fft_tau_to_iw(ctx.handle, X, out)
                    b.record()
                    torch.cuda.synchronize()
                    best.append(a.elapsed_time(b) / 8e-3)
                us.append(min(best))
        print(n, M, len(idx), n_iw, "rule %.1f product %.1f FFTs %.1f us" % tuple(us))
        fast, slow = (us[1], us[2]) if product else (us[2], us[1])
        assert slow > 1.3 * fast and us[0] < 1.15 * fast, us


@pytest.mark.parametrize("n,p,u,n_iw", [(1, 2, 2, 1), (5, 2, 2, 31), (12, 3, 8, 32), (13, 3, 8, 33), (4, 7, 16, 300),
                                        (4, 3, 32, 64), (3, 7, 32, 1000), (11, 3, 2, 65), (2, 2, 64, 97)])
def test_product_at_the_edges_of_its_tiles(g, n, p, u, n_iw):
    """As test_product_and_ffts_match_oracle, by the product whatever the rule would take."""
    import ctypes
    f = g.lib().gf2_test_fourier_path
    f.argtypes, f.restype = [ctypes.c_void_p, ctypes.c_int], ctypes.c_int
    M, idx = grids.power_mesh(p, u)
    X = np.random.default_rng(n * 1000 + n_iw + 1).uniform(-1.0, 1.0, (len(idx), n, n))
    out = torch.zeros(n_iw, n, n, dtype=torch.complex128, device="cuda")
    with g.Context(n, None, n_iw, 40.0, grid=(M, idx)) as ctx:
        assert f(ctx.handle, 1) == 0
        g.gf2_fft_tau_to_iw(ctx.handle, dev(X), out)
        got = out.cpu().numpy()
    ref = ot.tau_to_iw_grid(X, 40.0, M, idx, n_iw)
    size = ot.tau_to_iw_grid(np.abs(X), 40.0, M, idx, 1)
    assert np.abs(got - ref).max() <= 2.0 ** -44 * 2.0 * np.abs(size[0]).max()
