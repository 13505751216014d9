"""The FP64 path's fixed-point pair arithmetic where it could go wrong: tile
edges, close pairs on both sides of the distance the grid resolves, mass ratios
and velocities of very different size, far outliers, extreme units, values its
formats do not take.

Bound.  One fixed-point pair is within 2^-50 of its exact value (acceleration
and potential of their own size, jerk of m (|w| + 3 |r.w| |r| / s^2) / s^3, plus
2^-54 m Vmax / s^3 for the grid of the velocities), and so is the oracle's FP64
pair; both sum without further error to speak of.  So each result may differ by
2^-49 of the sum of the terms' sizes; twice that is allowed.
"""
import numpy as np
import pytest

import oracle
from paper_0709_4552_gb300 import inputs
from _util import gpu_forces

pytestmark = pytest.mark.gpu


def _sizes(m, x, v, eps, idx):
    """Sums of the sizes of the terms of each result, and of the velocity grid's unit."""
    A, J, P = np.zeros(len(idx)), np.zeros(len(idx)), np.zeros(len(idx))
    vmax = np.abs(v).max()
    for k, i in enumerate(idx):
        d, w = x - x[i], v - v[i]
        s2 = (d * d).sum(1) + eps * eps
        keep = np.arange(len(m)) != i
        d, w, s2, mm = d[keep], w[keep], s2[keep], np.abs(m[keep])
        r, s = np.sqrt((d * d).sum(1)), np.sqrt(s2)
        A[k] = (mm * r / s ** 3).sum()
        J[k] = (mm * (np.sqrt((w * w).sum(1)) + 3 * np.abs((d * w).sum(1)) * r / s2 + vmax / 64) / s ** 3).sum()
        P[k] = (mm / s).sum()
    return A, J, P


def _system(kind, N):
    m, x, v = inputs.plummer(N, 500 + N, "salpeter")
    rng = np.random.default_rng(N)
    eps = 1.0 / 512
    if kind == "unsoftened":
        eps = 0.0
    elif kind == "close_pairs":  # distances from far below to far above 2^(g-8) of any grid here
        k = N // 2
        u = rng.normal(size=(k, 3))
        u /= np.linalg.norm(u, axis=1)[:, None]
        x[k:2 * k] = x[:k] + u * 2.0 ** rng.uniform(-30, -2, (k, 1))
        eps = 2.0 ** -20
    elif kind == "masses":  # ratio up to 2^60, massless and (in FP64 arithmetic no error) negative ones
        m = m * 2.0 ** rng.uniform(-60, 0, N)
        m[::7] = 0.0
        m[3::11] *= -1.0
    elif kind == "outliers":  # tiles of very different extent and speed
        x[::50] *= 2.0 ** 30
        v[::50] *= 2.0 ** 20
        x[N // 2:] *= 2.0 ** -20
        v[N // 4:N // 2] = 0.0
    elif kind == "large_softening":
        eps = 64.0
    elif kind == "big_units":
        x, v, eps = x * 2.0 ** 200, v * 2.0 ** 90, eps * 2.0 ** 200
    elif kind == "small_units":
        x, v, eps = x * 2.0 ** -180, v * 2.0 ** -100, eps * 2.0 ** -180
    elif kind == "planar":
        x[:, 2] = 0.0
        v[:, 2] = 0.0
    return m, x, v, eps


@pytest.mark.parametrize("kind", ["plain", "unsoftened", "close_pairs", "masses", "outliers", "large_softening",
                                  "big_units", "small_units", "planar"])
@pytest.mark.parametrize("N,j_tile", [(2, 64), (33, 32), (64, 64), (129, 128), (1100, 64)])
def test_fixed_point_pairs(nbl, kind, N, j_tile):
    m, x, v, eps = _system(kind, N)
    idx = np.arange(N)
    a, j, p = gpu_forces(nbl, nbl.NB_FP64, m, x, v, eps, idx, tuning=dict(j_tile=j_tile, n_split=1 + N // 500))
    ar, jr, pr = oracle.forces(m, x, v, eps, compensated=True)
    A, J, P = _sizes(m, x, v, eps, idx)
    for got, ref, size in ((a, ar, A), (j, jr, J), (p[:, None], pr[:, None], P)):
        off = np.linalg.norm(got - ref, axis=1)
        assert (off <= 2.0 ** -48 * size).all(), (kind, N, (off / np.maximum(size, 1e-300)).max())
    if kind == "planar":  # exact zeros stay zero
        assert np.all(a[:, 2] == 0.0) and np.all(j[:, 2] == 0.0)


@pytest.mark.parametrize("scale", [2.0 ** 320, 2.0 ** -330])
def test_units_beyond_the_formats(nbl, scale):
    # exponents the fixed-point formats do not take: FP64 arithmetic throughout.
    # Only the positions are scaled: 1/s and s^2 stay inside FP64's range here.
    N = 70
    m, x, v = inputs.plummer(N, 77)
    a, j, p = gpu_forces(nbl, nbl.NB_FP64, m, x * scale, v, 0.0, np.arange(N))
    _, _, pr = oracle.forces(m, x, v, 0.0, compensated=True)
    assert (np.abs(p * scale - pr) <= 2.0 ** -48 * np.abs(pr)).all()


def test_result_does_not_depend_on_the_rest_of_the_block(nbl):
    # the grid belongs to the j-tiles: a particle's result is the same bits in any block
    N, eps = 3000, 1 / 256
    m, x, v = inputs.plummer(N, 78, "salpeter")
    x[::100] *= 50.0
    tuning = dict(n_split=3)
    full = gpu_forces(nbl, nbl.NB_FP64, m, x, v, eps, np.arange(N), tuning=tuning)
    idx = inputs.sample_indices(N, 37, 5)
    part = gpu_forces(nbl, nbl.NB_FP64, m, x, v, eps, idx, tuning=tuning)
    for f, q in zip(full, part):
        assert np.array_equal(f[idx], q)
