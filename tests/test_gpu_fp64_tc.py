"""The FP64 Sigma as exact digit products on the tensor cores, against the
oracle's Eq. Sigma.

Sizes lie at the edges of the 16-wide K steps, the 32-column accumulators and
the 128-row tiles (N = 1 .. 64), with G and v that have no symmetry at all,
signed zeros and blocks of zeros, entries spread over many decades, and scales
whose products leave the range of the fast exponent arithmetic.

Tolerance.  A stage's digit arithmetic errs by at most K 2^-56 (row maximum)
(column maximum) and its result is rounded once (2^-53); for entries spread
uniformly over their range the product of the maxima is about four times the
mean product, so four stages stay within 4 (1 + 4 / 8) 2^-53 < 2^-50 of the sum of
absolute terms.  The oracle's own sums round too (blocked, up to N^3 terms):
2^-47 of that sum bounds both sides.
"""

import numpy as np
import pytest
import torch

import gf2_inputs as gi
from oracle import sigma as osg

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


def run(g, G, v, k0=0, count=None):
    nt, n, _ = G.shape
    count = nt if count is None else count
    with g.Context(n, nt, 8, 10.0) as ctx:
        g.gf2_set_integrals(ctx.handle, dev(v))
        out = torch.full((count, n, n), 7.0, dtype=torch.float64, device="cuda")
        g.gf2_sigma_tau_points(ctx.handle, dev(G), k0, count, out, g.GF2_PREC_FP64)
        return out.cpu().numpy()


def check(got, G, v, points, k0=0, factor=2.0 ** -47):
    W = osg.exchange_combination(v)
    aW = 2.0 * np.abs(v) + np.abs(v.transpose(2, 1, 0, 3))
    for k in points:
        ref = osg.sigma_factored(G[k], osg.gbar_from_grid(G, k), v, W)
        size = np.abs(osg.sigma_factored(np.abs(G[k]), np.abs(osg.gbar_from_grid(G, k)), np.abs(v), aW))
        assert np.all(np.abs(got[k - k0] - ref) <= factor * size + 1e-300), (k, np.abs(got[k - k0] - ref).max())


@pytest.mark.parametrize("n,n_tau", [(1, 9), (2, 17), (3, 9), (15, 9), (16, 65), (17, 9), (31, 9), (32, 9), (33, 9),
                                     (48, 9), (49, 9), (63, 9), (64, 9), (65, 9), (80, 9), (97, 9), (128, 9)])
def test_every_edge_without_any_symmetry(g, n, n_tau):
    rng = np.random.default_rng(1000 + n)
    G = rng.uniform(-1.0, 1.0, (n_tau, n, n))
    v = rng.uniform(-1.0, 1.0, (n, n, n, n))
    check(run(g, G, v), G, v, range(n_tau) if n < 33 else (0, 3, n_tau - 1) if n <= 64 else (3,))


@pytest.mark.parametrize("k0,count", [(0, 129), (1, 3), (64, 1), (127, 2)])
def test_sub_ranges_and_many_tiles_per_cta(g, k0, count):
    G, v = gi.random_symmetric_g(20, 129, seed=7), gi.random_eri(20, seed=8)
    check(run(g, G, v, k0, count), G, v, {k0, k0 + count // 2, k0 + count - 1}, k0)


def test_chunks_of_the_workspace(g):
    """N = 64: the 2 GB workspace holds 8 time points, so 17 run as 8, 8 and 1."""
    G, v = gi.random_symmetric_g(64, 17, seed=9), gi.random_eri(64, seed=10)
    check(run(g, G, v), G, v, (0, 7, 8, 15, 16))


@pytest.mark.parametrize("n", [10, 40])
def test_zero_blocks_signed_zeros_and_decades(g, n):
    rng = np.random.default_rng(n)
    G = rng.uniform(-1.0, 1.0, (9, n, n))
    v = rng.uniform(-1.0, 1.0, (n, n, n, n))
    G[3] = 0.0
    G[4][: n // 2] = -0.0
    v[:, :, 1] *= -0.0
    v[2] = 0.0
    v *= 10.0 ** rng.integers(-6, 1, (n, 1, 1, n))
    # entries far below their row's largest are rounded to 2^-63 of it: covered by the
    # ratio of the maxima's product to the mean product, 10^6 here instead of 4 in two stages
    got = run(g, G, v)
    check(got, G, v, (0, 3, 4, 8), factor=2.0 ** -47 + 2.0 * n * 4.0e6 * 2.0 ** -62)
    assert np.all(got[3] == 0.0) and not np.any(np.signbit(got[3]) & (got[3] != 0.0))


@pytest.mark.parametrize("sv,sg", [(1e-120, 1e30), (1e100, 1e-60), (1e60, 1e20)])
def test_scales_beyond_the_fast_exponent_arithmetic(g, sv, sg):
    """Intermediates near both ends of the FP64 range; Sigma itself scales as v^2 G^3."""
    G, v = gi.random_symmetric_g(12, 9, seed=11), gi.random_eri(12, seed=12)
    check(run(g, G * sg, v * sv), G * sg, v * sv, range(9))


@pytest.mark.parametrize("n,bad", [(10, np.nan), (10, np.inf), (36, np.nan), (36, -np.inf)])
def test_non_finite_input_reaches_its_points_only(g, n, bad):
    G, v = gi.random_symmetric_g(n, 17, seed=13), gi.random_eri(n, seed=14)
    H = G.copy()
    H[5, 1, 2] = bad
    got = run(g, H, v)
    for k in range(17):
        assert np.isfinite(got[k]).all() == (k not in (5, 11)), k
    check(got, G, v, (0, 8))


def test_new_integrals_under_capture(g):
    """Planes that become stale outside a capture are rebuilt inside it and, not
    having run yet, again by the next call."""
    n, nt = 24, 17
    G = gi.random_symmetric_g(n, nt, seed=15)
    v1, v2 = gi.random_eri(n, seed=16), gi.random_eri(n, seed=17)
    Gd, out = dev(G), torch.zeros(nt, n, n, dtype=torch.float64, device="cuda")
    with g.Context(n, nt, 8, 10.0) as ctx:
        g.gf2_set_integrals(ctx.handle, dev(v1))
        g.gf2_sigma_tau(ctx.handle, Gd, out, g.GF2_PREC_FP64)
        check(out.cpu().numpy(), G, v1, (0, 16))
        g.gf2_set_integrals(ctx.handle, dev(v2))
        torch.cuda.synchronize()
        graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(graph, stream=side):
            g.gf2_set_stream(ctx.handle)
            g.gf2_sigma_tau(ctx.handle, Gd, out, g.GF2_PREC_FP64)
        g.gf2_set_stream(ctx.handle)
        g.gf2_sigma_tau(ctx.handle, Gd, out, g.GF2_PREC_FP64)
        check(out.cpu().numpy(), G, v2, (0, 16))
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        check(out.cpu().numpy(), G, v2, (0, 16))


@pytest.mark.parametrize("n,n_tau", [(1, 9), (2, 17), (3, 9), (15, 9), (16, 65), (17, 9), (31, 9), (32, 9), (33, 9),
                                     (48, 9), (49, 9), (63, 9), (64, 9), (65, 9)])
def test_integrals_symmetric_in_the_bra_only(g, n, n_tau):
    """v[i][m] = v[m][i] to the last bit: two axes run over the pairs i <= m.  One entry off
    by one unit in the last place takes all of them again."""
    rng = np.random.default_rng(2000 + n)
    G = rng.uniform(-1.0, 1.0, (n_tau, n, n))
    v = rng.uniform(-1.0, 1.0, (n, n, n, n))
    low = np.tril(np.ones((n, n), dtype=bool))
    v = np.where(low[:, :, None, None], v, v.transpose(1, 0, 2, 3))
    assert np.array_equal(v, v.transpose(1, 0, 2, 3))
    points = range(n_tau) if n < 33 else (0, 3, n_tau - 1)
    got = run(g, G, v)
    check(got, G, v, points)
    if n > 1:
        u = v.copy()
        u[0, n - 1, n - 1, 0] = np.nextafter(u[0, n - 1, n - 1, 0], 9.0)
        check(run(g, G, u), G, u, points)


@pytest.mark.parametrize("n", [24, 40, 80])
def test_a_captured_call_follows_new_integrals(g, n):
    """The planes were ready when the call was captured; the integrals change between
    symmetric ones and ones without any symmetry."""
    nt = 9
    G = gi.random_symmetric_g(n, nt, seed=18)
    v1 = np.random.default_rng(19).uniform(-1.0, 1.0, (n, n, n, n))
    v2 = v1 + v1.transpose(1, 0, 2, 3)
    Gd, out = dev(G), torch.zeros(nt, n, n, dtype=torch.float64, device="cuda")
    with g.Context(n, nt, 8, 10.0) as ctx:
        g.gf2_set_integrals(ctx.handle, dev(v2))
        g.gf2_sigma_tau(ctx.handle, Gd, out, g.GF2_PREC_FP64)
        torch.cuda.synchronize()
        graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(graph, stream=side):
            g.gf2_set_stream(ctx.handle)
            g.gf2_sigma_tau(ctx.handle, Gd, out, g.GF2_PREC_FP64)
        g.gf2_set_stream(ctx.handle)
        for v in (v1, v2):
            g.gf2_set_integrals(ctx.handle, dev(v))
            out.zero_()
            graph.replay()
            torch.cuda.synchronize()
            check(out.cpu().numpy(), G, v, (3,))


def graded(n, spread, kind):
    """Powers of two for n basis functions, 2^spread apart: rising, alternating or one alone."""
    e = {"rising": np.round(np.linspace(0, spread, n)), "alternating": spread * (np.arange(n) % 2),
         "one": spread * (np.arange(n) == n // 2)}[kind].astype(int)
    return np.ldexp(1.0, e - spread // 2)


@pytest.mark.parametrize("n,spread,kind", [(5, 16, "rising"), (8, 12, "alternating"), (20, 8, "rising"), (31, 30, "one"),
                                           (40, 16, "alternating"), (64, 12, "rising"), (70, 12, "alternating")])
@pytest.mark.parametrize("symmetric", [False, True])
def test_basis_functions_of_different_norm(g, n, spread, kind, symmetric):
    """v -> d d d d v and G -> G / (d d): rows of v grow along the contracted index where columns
    of G shrink.  Eq. Sigma is covariant, and the sum of absolute terms that the
    tolerance is taken of scales with the result: the same tolerance as everywhere."""
    rng = np.random.default_rng(3000 + n)
    G, v = rng.uniform(-1.0, 1.0, (9, n, n)), rng.uniform(-1.0, 1.0, (n, n, n, n))
    if symmetric:
        v = v + v.transpose(1, 0, 2, 3)
    d = graded(n, spread, kind)
    v *= d[:, None, None, None] * d[:, None, None] * d[:, None] * d
    G /= d[:, None] * d
    check(run(g, G, v), G, v, (0, 3, 8) if n < 60 else (3,))


def test_integrals_with_empty_and_tiny_diagonals(g):
    """No scale can be read off v[i][i]: functions without any integral, and a diagonal that is
    tiny beside the rest, leave the others as accurate as they are."""
    n = 24
    rng = np.random.default_rng(77)
    G, v = rng.uniform(-1.0, 1.0, (9, n, n)), rng.uniform(-1.0, 1.0, (n, n, n, n))
    for i in range(n):
        v[i, i] *= 2.0 ** -60
    for i in (3, 11):
        v[i], v[:, i], v[:, :, i], v[..., i] = 0.0, 0.0, 0.0, 0.0
    v *= 2.0 ** -80
    check(run(g, G, v), G, v, range(9))


@pytest.mark.parametrize("n,m", [(6, 20), (40, 50)])
def test_factor_order_with_basis_functions_of_different_norm(g, n, m):
    rng = np.random.default_rng(n)
    G, B = rng.uniform(-1.0, 1.0, (9, n, n)), rng.uniform(-1.0, 1.0, (m, n, n))
    d = graded(n, 14, "alternating")
    B *= d[:, None] * d
    G /= d[:, None] * d
    v = np.tensordot(B, B, axes=(0, 0))
    out = torch.empty(9, n, n, dtype=torch.float64, device="cuda")
    with g.Context(n, 9, 8, 10.0) as ctx:
        g.gf2_set_df_integrals(ctx.handle, dev(B))
        g.gf2_sigma_tau_df(ctx.handle, dev(G), 0, 9, out)
        got = out.cpu().numpy()
    # the library sums m products of B where the oracle is given v: that v's own rounding is
    # m 2^-53 of the sums of absolute products, in the two v of Eq. Sigma
    aW = np.tensordot(np.abs(B), np.abs(B), axes=(0, 0))
    W = osg.exchange_combination(v)
    for k in (0, 4, 8):
        ref = osg.sigma_factored(G[k], osg.gbar_from_grid(G, k), v, W)
        size = np.abs(osg.sigma_factored(np.abs(G[k]), np.abs(osg.gbar_from_grid(G, k)), aW,
                                         2.0 * aW + aW.transpose(2, 1, 0, 3)))
        assert np.all(np.abs(got[k] - ref) <= (2.0 ** -47 + 4 * m * 2.0 ** -53) * size)


@pytest.mark.parametrize("n,m", [(12, 30), (40, 50)])
def test_a_captured_factor_order_follows_new_integrals(g, n, m):
    """Captured with its planes ready; the factor changes, its number of functions does not.
    The replay gives what an eager call gives, up to the order of the last atomic sums."""
    G = dev(gi.random_symmetric_g(n, 9, seed=20))
    rng = np.random.default_rng(21)
    out = torch.zeros(9, n, n, dtype=torch.float64, device="cuda")
    with g.Context(n, 9, 8, 10.0) as ctx:
        g.gf2_set_df_integrals(ctx.handle, dev(rng.uniform(-1.0, 1.0, (m, n, n))))
        g.gf2_sigma_tau_df(ctx.handle, G, 0, 9, out)
        torch.cuda.synchronize()
        graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(graph, stream=side):
            g.gf2_set_stream(ctx.handle)
            g.gf2_sigma_tau_df(ctx.handle, G, 0, 9, out)
        g.gf2_set_stream(ctx.handle)
        g.gf2_set_df_integrals(ctx.handle, dev(rng.uniform(-1.0, 1.0, (m, n, n))))
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        replayed = out.cpu().numpy()
        g.gf2_sigma_tau_df(ctx.handle, G, 0, 9, out)
        eager = out.cpu().numpy()
    assert np.abs(replayed - eager).max() <= 2.0 ** -44 * np.abs(eager).max()


def test_integrals_set_by_a_graph_that_precedes_the_planes(g):
    """gf2_set_integrals captured before the first FP64 call (N > 64, where it can be): calls
    follow its replays, and pay for new planes only after one."""
    n, nt = 96, 9
    G = gi.random_symmetric_g(n, nt, seed=22)
    v1, v2 = gi.random_eri(n, seed=23), gi.random_eri(n, seed=24)
    Gd, vd, out = dev(G), dev(v1), torch.zeros(1, n, n, dtype=torch.float64, device="cuda")

    def timed(ctx):
        ms = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            g.gf2_sigma_tau_points(ctx.handle, Gd, 3, 1, out, g.GF2_PREC_FP64)
            b.record()
            torch.cuda.synchronize()
            ms.append(a.elapsed_time(b))
        return min(ms)

    with g.Context(n, nt, 8, 10.0) as ctx:
        g.gf2_set_integrals(ctx.handle, vd)
        torch.cuda.synchronize()
        graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(graph, stream=side):
            g.gf2_set_stream(ctx.handle)
            g.gf2_set_integrals(ctx.handle, vd)
        g.gf2_set_stream(ctx.handle)
        for v in (v1, v2, v1):
            vd.copy_(dev(v))
            graph.replay()
            g.gf2_sigma_tau_points(ctx.handle, Gd, 3, 1, out, g.GF2_PREC_FP64)
            check(out.cpu().numpy(), G, v, (3,), k0=3)
        after_graph = timed(ctx)
    with g.Context(n, nt, 8, 10.0) as ctx:
        g.gf2_set_integrals(ctx.handle, vd)
        plain = timed(ctx)
    assert after_graph <= 1.15 * plain, (after_graph, plain)


@pytest.mark.parametrize("n,blocks", [(65, 33), (66, 1123), (100, 1000)])
def test_planes_of_w_a_part_at_a_time(g, n, blocks):
    """N > 64 where memory is short: the last stage in parts of `blocks` blocks of 256, the last
    part smaller or a single block, and again after new integrals."""
    import ctypes
    f = g.lib().gf2_test_wide_blocks
    f.argtypes, f.restype = [ctypes.c_void_p, ctypes.c_int], ctypes.c_int
    G = gi.random_symmetric_g(n, 9, seed=25)
    out = torch.empty(2, n, n, dtype=torch.float64, device="cuda")
    with g.Context(n, 9, 8, 10.0) as ctx:
        assert f(ctx.handle, blocks) == 0
        for seed in (26, 27):
            v = gi.random_eri(n, seed=seed)
            g.gf2_set_integrals(ctx.handle, dev(v))
            g.gf2_sigma_tau_points(ctx.handle, dev(G), 3, 2, out, g.GF2_PREC_FP64)
            check(out.cpu().numpy(), G, v, (3, 4), k0=3)
    assert f(None, 1) == 1
