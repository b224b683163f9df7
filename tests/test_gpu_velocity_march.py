"""Shape velocity on grids above the size from which its Chebyshev steps are
marched through z by strips of four rows and windows of 30 columns (4e5 node
values over all vectors), against the exact inverse: the periodic operator is
diagonal under the discrete Fourier transform.

Shapes (nz, ny, nx): rows that are no whole number of strips (ny = 83, 54, 2,
3, 5), columns whose sequence of nx + 2 positions is no whole number of windows,
z sizes that are no multiple of the chunk, one and four vectors.  Bound: 1e-10
of the largest value, that of the small grids' comparison (the iteration
reduces the A-norm error by 1e-13).
"""
import numpy as np
import pytest
import torch

import cellgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_03148_gb300 import load
    return load()


def representers(shape, alpha, ds):
    """A^-1 d with A = alpha^2 K + M in Q1 on the periodic unit cell."""
    s, m = [], []
    for n in shape:
        c = np.cos(2.0 * np.pi * np.arange(n) / n)
        s.append((2.0 - 2.0 * c) * n)
        m.append((4.0 + 2.0 * c) / (6.0 * n))
    o = lambda a, b, c: a[:, None, None] * b[None, :, None] * c[None, None, :]
    lam = alpha ** 2 * (o(s[0], m[1], m[2]) + o(m[0], s[1], m[2]) + o(m[0], m[1], s[2])) + o(*m)
    return [np.fft.ifftn(np.fft.fftn(d) / lam).real for d in ds]


def velocity(shape, alpha, dJ, dCs, Cs, wJ, wC):
    """Null-space step from the representers (Gram matrix, Cholesky)."""
    ds = [dJ] + dCs
    g = representers(shape, alpha, ds)
    G = np.array([[float((a * b).sum()) for b in ds] for a in g])
    G = 0.5 * (G + G.T)
    n = len(dCs)
    coef, norm2, mu = np.zeros(n), G[0, 0], np.zeros(0)
    if n:
        R = np.linalg.cholesky(G[1:, 1:]).T
        p = np.linalg.solve(R.T, G[1:, 0])
        norm2 -= p @ p
        mu = np.linalg.solve(R.T, wC * np.array(Cs))
        coef = np.linalg.solve(R, mu - wJ * p / np.sqrt(norm2))
    norm = np.sqrt(norm2)
    return wJ * g[0] / norm + sum(c * gi for c, gi in zip(coef, g[1:])), norm, mu


@pytest.mark.parametrize("shape,ncons", [((61, 83, 85), 0), ((37, 54, 61), 3), ((150, 2, 1400), 0), ((89, 3, 388), 3),
                                         ((31, 5, 2700), 0), ((2, 180, 290), 3)])
def test_large_grids_match_the_fourier_inverse(shape, ncons):
    from paper_2410_03148_gb300 import Cell
    assert np.prod(shape) * (1 + ncons) >= 400000
    rng = np.random.default_rng(51)
    dev = "cuda:0"
    cell = Cell(torch.as_tensor(cellgen.random_rho(shape, seed=2), device=dev), cellgen.pzt5h_class(), kind="rho",
                autotune=0, restart=1, load_mask=1)
    dJ = rng.standard_normal(shape)
    dCs = [np.ones(shape) + 0.2 * rng.standard_normal(shape) for _ in range(ncons)]
    Cs = list(0.1 * rng.standard_normal(ncons))
    alpha = 4.0 / max(shape)
    t = lambda a: torch.as_tensor(a, device=dev)
    v, norm, _, mu = cell.hilbert_velocity(t(dJ), [t(d) for d in dCs], Cs, alpha=alpha, wJ=1.3, wC=0.6)
    want, n_want, mu_want = velocity(shape, alpha, dJ, dCs, Cs, 1.3, 0.6)
    assert np.abs(v.cpu().numpy() - want).max() < 1e-10 * np.abs(want).max()
    assert abs(norm - n_want) < 1e-10 * n_want
    assert np.allclose(mu, mu_want, rtol=1e-9, atol=1e-12 * np.abs(mu_want).max(initial=1.0))
