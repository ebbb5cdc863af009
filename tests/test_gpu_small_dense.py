"""The small dense FP64 kernels behind the tail moments: the cluster-wide inverse
(N over eight CTAs, some of them empty) and the small-tile product, at the edges
of both (1, 8, 9, 16, 17, 64, 65, 128), against numpy.

Tolerance: S = 1 + small symmetric part has a condition number below 3; an
elimination without pivoting on such a matrix errs by at most about n kappa 2^-53
per entry of order one, a product of n terms by n 2^-53 of the sum of absolute
terms, and G3, G4 chain up to five of them: 8 (n + 8) 2^-53 of the largest product
of absolute values bounds all four moments.
"""

import numpy as np
import pytest
import torch

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


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 15, 16, 17, 63, 64, 65, 127, 128])
def test_tail_moments_at_every_edge(g, n):
    rng = np.random.default_rng(n)
    a = rng.normal(size=(n, n)) / np.sqrt(n)
    S = np.eye(n) + 0.1 * (a + a.T)
    F, s1, s2 = rng.normal(size=(3, n, n))
    F = F + F.T
    mu, dev = 0.3, lambda x: torch.as_tensor(np.ascontiguousarray(x), device="cuda")
    mom = torch.full((4, n, n), 7.0, dtype=torch.float64, device="cuda")
    with g.Context(n, 9, 8, 10.0) as ctx:
        g.gf2_tail_moments(ctx.handle, dev(S), dev(F), mu, dev(np.stack([s1 + s1.T, s2 + s2.T])), mom)
        mom = mom.cpu().numpy()
    Si = np.linalg.inv(S)

    def moments(Si, X, s1, s2):
        return [Si, Si @ X @ Si, Si @ (X @ Si @ X + s1) @ Si,
                Si @ (X @ Si @ X @ Si @ X + X @ Si @ s1 + s1 @ Si @ X + s2) @ Si]

    ref = moments(Si, F - mu * S, s1 + s1.T, s2 + s2.T)
    size = moments(np.abs(Si), np.abs(F) + mu * np.abs(S), np.abs(s1 + s1.T), np.abs(s2 + s2.T))
    for k in range(4):
        assert np.abs(mom[k] - ref[k]).max() <= 8.0 * (n + 8) * 2.0 ** -53 * size[k].max(), k


@pytest.mark.parametrize("n", [1, 2, 7, 9, 31, 32, 33, 63, 64, 65, 96, 97])
def test_fock_at_the_edges_of_its_columns_and_ranges(g, n):
    """v and P without symmetry.  Each entry is a sum of at most 2 N^2 + 1 rounded terms: it
    errs by (2 N^2 + 16) 2^-53 of the sum of their absolute values on either side."""
    rng = np.random.default_rng(300 + n)
    v, P, h = rng.uniform(-1, 1, (n, n, n, n)), rng.uniform(-1, 1, (n, n)), rng.uniform(-1, 1, (n, n))
    F, dev = torch.empty(n, n, dtype=torch.float64, device="cuda"), lambda x: torch.as_tensor(x, device="cuda")
    with g.Context(n, 9, 8, 10.0) as ctx:
        g.gf2_set_integrals(ctx.handle, dev(v))
        g.gf2_fock(ctx.handle, dev(h), dev(P), F)
    J = np.tensordot(v, P, axes=([3, 2], [0, 1]))            # sum_kl P_kl v_ijlk
    K = np.tensordot(v, P, axes=([1, 2], [0, 1]))            # sum_kl P_kl v_iklj
    size = np.abs(h) + np.tensordot(np.abs(v), np.abs(P), axes=([3, 2], [0, 1])) + np.tensordot(
        np.abs(v), np.abs(P), axes=([1, 2], [0, 1]))
    assert np.all(np.abs(F.cpu().numpy() - (h + J - 0.5 * K)) <= 2.0 * (2 * n * n + 16) * 2.0 ** -53 * size)


@pytest.mark.parametrize("n", [8, 64, 127])
def test_inverse_is_the_same_whenever_its_ctas_start(g, n):
    """The eight CTAs of the inverse write into each other's shared memory from the first pivot
    on.  Beside work that fills the chip, so that they start at different times, it gives
    the bits that it gives alone: nothing in it depends on the order of their start."""
    rng = np.random.default_rng(n)
    a = rng.normal(size=(n, n)) / np.sqrt(n)
    dev = lambda x: torch.as_tensor(np.ascontiguousarray(x), device="cuda")
    S, F = dev(np.eye(n) + 0.1 * (a + a.T)), dev(a + a.T)
    big = torch.ones(1 << 26, dtype=torch.float32, device="cuda")
    side = torch.cuda.Stream()
    mom = [torch.zeros(4, n, n, dtype=torch.float64, device="cuda") for _ in range(33)]
    with g.Context(n, 9, 8, 10.0) as ctx:
        g.gf2_tail_moments(ctx.handle, S, F, 0.3, None, mom[0])
        torch.cuda.synchronize()
        for m in mom[1:]:
            with torch.cuda.stream(side):
                for _ in range(4):
                    big.mul_(1.0)
            g.gf2_tail_moments(ctx.handle, S, F, 0.3, None, m)
        torch.cuda.synchronize()
    for m in mom[1:]:
        assert torch.equal(m, mom[0])


@pytest.mark.parametrize("n", [1, 2, 10, 11, 15, 16, 22, 23, 33, 34, 35, 36, 47, 48, 52, 53, 65, 66, 71, 72, 92, 93, 100,
                               101, 128])
def test_dyson_at_the_edges_of_its_layouts(g, n):
    """Either side of every size at which dyson_kernel changes its threads or elements per
    thread, with and without Sigma.  A = (i w + mu) S - F - Sigma has an imaginary part that is
    definite, so elimination without pivoting grows by at most a few: it errs by
    16 n 2^-53 of |A^-1| |A| |A^-1| on either side."""
    rng = np.random.default_rng(400 + n)
    a = rng.normal(size=(n, n)) / np.sqrt(n)
    S, beta, n_iw, mu = np.eye(n) + 0.1 * (a + a.T), 10.0, 5, 0.2
    F = rng.normal(size=(n, n)) / np.sqrt(n)
    F = F + F.T
    w = (2 * np.arange(n_iw) + 1) * np.pi / beta
    sig = rng.normal(size=(n_iw, n, n)) / np.sqrt(n)
    sig = 0.1 * (sig + sig.transpose(0, 2, 1)) - 0.05j * S / w[:, None, None]
    dev = lambda x: torch.as_tensor(np.ascontiguousarray(x), device="cuda")
    G = torch.empty(n_iw, n, n, dtype=torch.complex128, device="cuda")
    with g.Context(n, 9, n_iw, beta) as ctx:
        for X in (None, sig):
            g.gf2_dyson(ctx.handle, mu, dev(S), dev(F), None if X is None else dev(X), G)
            A = (1j * w[:, None, None] + mu) * S - F - (0.0 if X is None else X)
            ref = np.linalg.inv(A)
            bound = 2 * 16 * n * 2.0 ** -53 * (np.abs(ref) @ np.abs(A) @ np.abs(ref)).max()
            assert np.abs(G.cpu().numpy() - ref).max() <= bound
