"""The uniform transforms and iw -> tau on meshes, element by element: matrix elements of very
different size, exact zeros, non-finite samples and symmetric matrices beside each
other, an odd number of elements, the shortest and longest grids, fewer and more
frequencies than grid points.

Tolerance: each element is a sum of its own samples with weights of known size, through
an FFT (at most 13 passes, a few roundings each); 2^-44 of the sum of the absolute
terms of that element covers both sides.  Nothing of another element enters.
"""

import numpy as np
import pytest
import torch

from oracle import grids
from oracle import transforms as ot

pytestmark = pytest.mark.gpu

BETA = 20.0


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


def sizes(n):
    """Magnitudes of the elements: neighbours up to 10^14 apart, every fifth element zero."""
    s = 10.0 ** -np.array([0.0, 12.0, 3.0, 14.0, 7.0])[np.arange(n * n) % 5]
    s[4::5] = 0.0
    return s.reshape(n, n)


def tau_to_iw(g, n, M, n_iw, X):
    out = torch.zeros(n_iw, n, n, dtype=torch.complex128, device="cuda")
    with g.Context(n, M + 1, n_iw, BETA) as ctx:
        g.gf2_fft_tau_to_iw(ctx.handle, dev(X), out)
        return out.cpu().numpy()


def iw_to_tau(g, n, M, n_iw, X, mom, mesh=None):
    with g.Context(n, M + 1, n_iw, BETA, grid=mesh) as ctx:
        out = torch.zeros(ctx.n_tau, n, n, dtype=torch.float64, device="cuda")
        g.gf2_fft_iw_to_tau(ctx.handle, dev(X), dev(mom), out)
        return out.cpu().numpy()


CASES = [(1, 8, 3), (3, 8, 40), (3, 16, 16), (2, 1024, 100), (5, 4096, 9000), (3, 8192, 700)]


@pytest.mark.parametrize("n,M,n_iw", CASES)
def test_tau_to_iw_per_element(g, n, M, n_iw):
    X = np.random.default_rng(M + n).uniform(-1.0, 1.0, (M + 1, n, n)) * sizes(n)
    got, ref = tau_to_iw(g, n, M, n_iw, X), ot.tau_to_iw(X, BETA, n_iw)
    # |weights| <= h sum |Lagrange polynomials| < 2 h, the end terms' up to 15 h on eight samples
    size = (BETA / M) * (2.0 * np.abs(X).sum(0) + 15.0 * (np.abs(X[:4]) + np.abs(X[-4:])).sum(0))
    assert np.all(np.abs(got - ref).max(0) <= 2.0 ** -44 * size)
    assert np.all(got[:, sizes(n) == 0.0] == 0.0)


@pytest.mark.parametrize("n,M,n_iw", CASES + [(3, (3, 8), 50), (5, (7, 32), 300)])
def test_iw_to_tau_per_element(g, n, M, n_iw):
    rng = np.random.default_rng(n_iw + n)
    mesh = None
    if isinstance(M, tuple):
        mesh = grids.power_mesh(*M)
        M = mesh[0]
    X = (rng.uniform(-1, 1, (n_iw, n, n)) + 1j * rng.uniform(-1, 1, (n_iw, n, n))) * sizes(n)
    mom = rng.uniform(-1, 1, (4, n, n)) * sizes(n)
    got, ref = iw_to_tau(g, n, M, n_iw, X, mom, mesh), ot.iw_to_tau(
        X, mom, BETA, M + 1, taus=mesh and list(mesh[1]))
    # the tail (z - 1)^-r and its image are below 1 and beta^3 in size, its four coefficients
    # at most eight moments each
    size = (2.0 / BETA) * np.abs(X).sum(0) + 32.0 * BETA ** 3 * np.abs(mom).sum(0)
    assert np.all(np.abs(got - ref).max(0) <= 2.0 ** -44 * size)
    assert np.all(got[:, sizes(n) == 0.0] == 0.0)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("n,M", [(2, 16), (3, 4096)])
def test_non_finite_sample_stays_in_its_element(g, n, M, bad):
    rng = np.random.default_rng(5)
    hit = np.zeros((n, n), bool)
    hit[1, 0] = True
    hit[2:, 2:] = True  # n = 3: the last element, which has no neighbour
    X = rng.uniform(-1, 1, (M + 1, n, n))
    X[5, hit] = bad
    got = tau_to_iw(g, n, M, 30, X)
    assert not np.isfinite(got[:, hit]).all(0).any() and np.isfinite(got[:, ~hit]).all()
    Y = rng.uniform(-1, 1, (30, n, n)) + 1j * rng.uniform(-1, 1, (30, n, n))
    Y[7, hit] = bad
    for mesh in (None, grids.power_mesh(2, 2)):
        got = iw_to_tau(g, n, M if mesh is None else mesh[0], 30, Y, np.zeros((4, n, n)), mesh)
        assert not np.isfinite(got[:, hit]).all(0).any() and np.isfinite(got[:, ~hit]).all()


@pytest.mark.parametrize("n,M,n_iw", [(3, 16, 40), (6, 4096, 500)])
def test_symmetric_matrices_stay_symmetric_to_the_bit(g, n, M, n_iw):
    rng = np.random.default_rng(M)
    X = rng.uniform(-1, 1, (M + 1, n, n))
    X = X + X.transpose(0, 2, 1)
    got = tau_to_iw(g, n, M, n_iw, X)
    assert np.array_equal(got, got.transpose(0, 2, 1))
    Y = rng.uniform(-1, 1, (n_iw, n, n)) + 1j * rng.uniform(-1, 1, (n_iw, n, n))
    mom = rng.uniform(-1, 1, (4, n, n))
    got = iw_to_tau(g, n, M, n_iw, Y + Y.transpose(0, 2, 1), mom + mom.transpose(0, 2, 1))
    assert np.array_equal(got, got.transpose(0, 2, 1))
