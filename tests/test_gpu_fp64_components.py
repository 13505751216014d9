"""The FP64 path's results component by component, on systems whose components or
masses differ so much that the fixed-point pair's integers could run out of bits:
a star among light companions, thin discs (one far from the origin too), needles,
cold velocities; through the kernels of every group count and the allocation-free
call.

Bound.  With u = 2^-53, an FP64 evaluation of a component's term is good to about
16 u of its size: the differences 1 each, s^2 6, 1/s and its powers 10 at most,
the products 4 (jerk: r.v to 3 u of sum |r_k v_k|, within the size used here), and
the sum over a tile, signs at random, a few more.  The fixed point has to be as
good, so each result may be 32 u of the sum of its terms' sizes away.
"""
import numpy as np
import pytest

import oracle
from paper_0709_4552_gb300 import inputs
from _util import gpu_forces
from test_gpu_fp64_fixed import _sizes, _system

pytestmark = pytest.mark.gpu
BOUND = 32 * 2.0 ** -53
N = 1100


def _set(kind):
    m, x, v = inputs.plummer(N, 900, "equal")
    what, _, size = kind.partition(" ")
    t = float(size or 0)
    if what == "star":  # a tile of companions of 2^-t its mass, all about as far away
        m, x, v = np.full(61, 2.0 ** -t), x[:61], v[:61]
        x *= (np.linspace(0.6, 1.0, 61) / np.linalg.norm(x, axis=1))[:, None]
        m[7], x[7], v[7] = 1.0, 0.0, 0.0
    elif what in ("disc", "away"):
        x[:, 2] *= t
        v[:, 2] *= t
        if what == "away":
            x += [3.0, 4.0, 5.0]
    elif what == "needle":
        x[:, :2] *= t
        v[:, :2] *= t
    elif what == "cold":
        v[:, 2] *= t
    elif what == "sheet":  # no extent along z, little motion
        x[:, 2] = 0.0
        v[:, 2] *= t
    elif what == "moving":
        v[:, 0] += t
    elif what == "slow":  # but for a few of each tile
        v[np.arange(N) % 50 > 0] *= t
    elif what == "halo":  # a disc and a few particles far above it
        x[:, 2] *= t
        v[:, 2] *= t
        x[::50, 2] /= t
    return m, x, v, 1.0 / 1024


def _exact(m, x, v, eps, idx):
    """acc, jerk, pot of the particles idx and the sums of their terms' sizes, by component, in
    the widest floats there are."""
    L = np.longdouble
    m, x, v = m.astype(L), x.astype(L), v.astype(L)
    out = [np.zeros((len(idx), 3), L), np.zeros((len(idx), 3), L), np.zeros((len(idx), 1), L)]
    size = [np.zeros_like(q) for q in out]
    for k, i in enumerate(idx):
        j = np.arange(len(m)) != i
        d, w = x[j] - x[i], v[j] - v[i]
        s2 = (d * d).sum(1) + L(eps) * L(eps)
        p = m[j] / np.sqrt(s2)
        g, f = (p / s2)[:, None], (3 * (d * w).sum(1) / s2)[:, None]
        h = (3 * np.abs(d * w).sum(1) / s2)[:, None]
        for q, term, big in ((0, g * d, g * np.abs(d)), (1, g * (w - f * d), g * (np.abs(w) + h * np.abs(d))),
                             (2, -p[:, None], p[:, None])):
            out[q][k], size[q][k] = term.sum(0), big.sum(0)
    return out, size


def _noalloc(nbl, m, x, v, eps, idx):
    import torch
    m, x, v = (torch.as_tensor(q, device="cuda") for q in (m, x, v))
    out = [torch.empty(len(idx), 3, device="cuda", dtype=torch.float64) for _ in range(2)]
    out.append(torch.empty(len(idx), device="cuda", dtype=torch.float64))
    nbl.nb_forces_fp64_noalloc(m, x, v, eps, torch.as_tensor(idx, device="cuda", dtype=torch.int32), *out)
    torch.cuda.synchronize()
    return [q.cpu().numpy() for q in out]


@pytest.mark.parametrize("kind", ["plain", "star 6", "star 10", "star 14", "disc 0.3", "disc 0.05", "disc 0.01",
                                  "disc 1e-3", "disc 1e-4", "disc 1e-5", "disc 1e-6", "disc 1e-9", "away 0.1", "away 1e-3",
                                  "away 1e-6", "needle 1e-3", "cold 1e-3", "sheet 0", "sheet 1e-3", "halo 1e-3", "moving 7", "moving 30",
                                  "slow 0.02"])
def test_every_component(nbl, kind):
    m, x, v, eps = _set(kind)
    idx = np.unique(np.append(np.arange(0, len(m), max(1, len(m) // 161))[:160], 7)).astype(np.int32)  # (with the star)
    star = np.flatnonzero(idx == 7)
    ref, size = _exact(m, x, v, eps, idx)

    def check(got, rows, how):
        for q, g in enumerate((got[0], got[1], got[2][:, None])):
            off = np.abs(g - ref[q][rows])
            assert (off <= BOUND * size[q][rows]).all(), (kind, how, q, float((off / size[q][rows]).max() / 2.0 ** -53))

    for j_tile in (32, 64, 128):
        check(gpu_forces(nbl, nbl.NB_FP64, m, x, v, eps, idx, tuning=dict(j_tile=j_tile, n_split=3)), slice(None), j_tile)
    for n in (1, 16, 17, 33, 65, 161):  # every number of groups that share a tile
        rows = np.sort(np.concatenate([star, np.setdiff1d(np.arange(len(idx)), star)[:n - 1]]))
        check(gpu_forces(nbl, nbl.NB_FP64, m, x, v, eps, idx[rows]), rows, n)
        check(_noalloc(nbl, m, x, v, eps, idx[rows]), rows, f"noalloc {n}")


@pytest.mark.parametrize("kind", ["unsoftened", "close_pairs", "masses", "outliers", "large_softening", "big_units",
                                  "small_units", "planar"])
def test_groups_on_the_fixed_points_hard_cases(nbl, kind):
    # the sets and the bound of test_fixed_point_pairs (whose explicit splits take one group)
    m, x, v, eps = _system(kind, N)
    ar, jr, pr = oracle.forces(m, x, v, eps, compensated=True)
    for n in (1, 16, 17, 33, 65, 161):
        idx = inputs.sample_indices(N, n, n).astype(np.int32)
        A, J, P = _sizes(m, x, v, eps, idx)
        for a, j, p in (gpu_forces(nbl, nbl.NB_FP64, m, x, v, eps, idx), _noalloc(nbl, m, x, v, eps, idx)):
            for got, ref, size in ((a, ar[idx], A), (j, jr[idx], J), (p[:, None], pr[idx, None], P)):
                off = np.linalg.norm(got - ref, axis=1)
                assert (off <= 2.0 ** -48 * size).all(), (kind, n, (off / np.maximum(size, 1e-300)).max())


@pytest.mark.parametrize("kind", ["away", "moving"])
def test_systems_the_grid_does_not_resolve_cost_what_fp64_arithmetic_does(nbl, kind):
    # far from the origin, or with a common velocity, no pair is for the fixed point: the time is then
    # that of the 34 FP64 instructions a pair takes, 1.2 times what the unit's measured rate allows (the
    # start and end of a launch), not that of the attempts as well (1.34)
    import torch
    n_all, n = 20000, 2000
    m, x, v = inputs.plummer(n_all, 3, "salpeter")
    (x if kind == "away" else v)[:] += 1000.0
    stream = torch.cuda.current_stream()
    with nbl.NBody(n_all, nbl.NB_FP64, 0, stream=stream) as s:
        s.set_params(1.0 / 1024, 0.01, 2.0 ** -22, 2.0 ** -5)
        s.set_j_particles(0, m, x, v)
        s.predict(0.0)
        idx = torch.as_tensor(inputs.sample_indices(n_all, n, 5), device="cuda", dtype=torch.int32)
        out = [torch.empty(n, 3, device="cuda", dtype=torch.float64) for _ in range(2)]
        out.append(torch.empty(n, device="cuda", dtype=torch.float64))
        ms = []
        for _ in range(9):
            a, b = torch.cuda.Event(True), torch.cuda.Event(True)
            a.record(stream)
            s.compute_forces(idx, *out)
            b.record(stream)
            torch.cuda.synchronize()
            ms.append(a.elapsed_time(b))
        rate = s.measure_peaks()["fp64_tflops"] * 1e12 / 2
    assert min(ms) * 1e-3 <= 1.27 * 34 * n_all * n / rate, (min(ms), 34e3 * n_all * n / rate)


@pytest.mark.parametrize("n", [2, 33, 64, 100, 128])
def test_loops_agree_to_the_bit_with_close_pairs(nbl, n):
    # systems of at most two j-tiles, binaries that the fixed point leaves to FP64 arithmetic among
    # them: the host loop's groups, the persistent loop and the graph add up the same (the graph with
    # one tile: it may split two otherwise)
    m, x, v = inputs.plummer(n, 950 + n, "salpeter")
    k = n // 2
    rng = np.random.default_rng(n)
    x[k:2 * k] = x[:k] + 2.0 ** rng.uniform(-14, -8, (k, 1)) * rng.normal(size=(k, 3))
    runs = []
    for loop in [nbl.NB_LOOP_HOST, nbl.NB_LOOP_PERSISTENT] + ([nbl.NB_LOOP_GRAPH] if n <= 64 else []):
        with nbl.NBody(n, nbl.NB_FP64, 0) as s:
            s.set_params(2.0 ** -9, 0.01, 2.0 ** -22, 2.0 ** -6)
            s.set_j_particles(0, m, x, v)
            s.initial_forces_and_dt()
            s.integrate(2.0 ** -6, loop=loop)
            runs.append(s.get_particles(0, n))
    for r in runs[1:]:
        for key in ("x", "v", "a", "jerk", "pot", "t", "dt"):
            assert np.array_equal(runs[0][key], r[key]), key
