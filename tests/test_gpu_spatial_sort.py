"""Resident spatial order (mixed path): it depends on the positions alone, not
on the order in which the particles were given, at the sizes where the sort
changes its chunks and kernels (512 and 2048 rows a chunk, 64 chunks)."""
import numpy as np
import pytest

from paper_0709_4552_gb300 import inputs

pytestmark = pytest.mark.gpu


def _lattice(N, seed):
    # distinct cells of the 1024^3 grid, both corners among them, so that the
    # bounding box and the cells' boundaries are exact in FP64
    rng = np.random.default_rng(seed)
    cells = np.unique(rng.integers(0, 1 << 30, size=2 * N + 16))
    cells = np.concatenate([[0], rng.permutation(cells[1:])[:N - 2], [(1 << 30) - 1]])[:N]
    q = np.stack([cells & 1023, (cells >> 10) & 1023, cells >> 20], axis=1)
    x = q / 512.0 - 1.0
    v = rng.standard_normal((N, 3)) * 0.1
    return rng.uniform(0.5, 1.5, N) / N, x, v


@pytest.mark.parametrize("N", [2, 511, 512, 513, 2049, 32768, 32769, 131072, 131073, 262145])
def test_order_depends_on_positions_only(nbl, N):
    m, x, v = _lattice(N, 41)
    mix = np.random.default_rng(42).permutation(N)
    k = np.unique(np.linspace(0, N - 1, 300).astype(np.int32))  # particles in the first order
    at = np.empty(N, np.int64)
    at[mix] = np.arange(N)  # and where the second holds them
    got = []
    for order, idx in ((np.arange(N), k), (mix, np.sort(at[k]).astype(np.int32))):
        with nbl.NBody(N, nbl.NB_MIXED, 0) as s:
            s.set_params(1.0 / 256, 0.01, 2.0 ** -22, 2.0 ** -3)
            s.set_j_particles(0, m[order], x[order], v[order])
            s.predict(0.0)
            a, j, p = s.compute_forces(idx)
            st = s.get_particles(0, N)
            assert np.array_equal(st["x"], x[order]) and np.array_equal(st["m"], m[order])
            got.append((order[idx], a, j, p))
    (i0, *f0), (i1, *f1) = got
    back = np.argsort(i1)
    assert np.array_equal(i0, i1[back])
    for q0, q1 in zip(f0, f1):
        assert np.array_equal(q0, q1[back])  # same rows, same sums


def test_renewed_orders_compose(nbl):
    # several renewals of the order within one run
    N, t_end = 3000, 2.0 ** -5
    m, x, v = inputs.plummer(N, 43)
    mix = np.random.default_rng(44).permutation(N)
    out = []
    for order in (np.arange(N), mix):
        with nbl.NBody(N, nbl.NB_MIXED, 0) as s:
            s.set_params(1.0 / 256, 0.01, 2.0 ** -22, t_end)
            s.set_j_particles(0, m[order], x[order], v[order])
            s.initial_forces_and_dt()
            s.integrate(t_end, loop=nbl.NB_LOOP_PERSISTENT)
            assert s.get_counters()["block_steps"] > 128
            st = s.get_particles(0, N)
            assert np.array_equal(st["m"], m[order])
            out.append({q: np.asarray(u)[np.argsort(order)] for q, u in st.items()})
    for q in out[0]:
        assert np.array_equal(out[0][q], out[1][q])
