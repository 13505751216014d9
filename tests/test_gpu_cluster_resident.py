"""The cluster loop with its rows' state in shared memory (up to 256 rows per
CTA: N = 4096 with 16 CTAs) and without: the rows it leaves in global memory
are the rows it worked on."""
import numpy as np
import pytest

from paper_0709_4552_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [3, 100, 1025, 4095, 4096, 4097])
def test_two_launches_are_one(nbl, N):
    # a second launch reads what the first wrote back: stopping and going on
    # changes no bit
    m, x, v = inputs.plummer(N, 51, "salpeter")
    T = 2.0 ** -5
    out = []
    for stops in ((T,), (T / 4, T / 2, T)):
        with nbl.NBody(N, nbl.NB_MIXED, 0) as s:
            s.set_params(1.0 / 256, 0.01, 2.0 ** -22, T / 4)
            s.set_j_particles(0, m, x, v)
            s.initial_forces_and_dt()
            for t in stops:
                s.integrate(t, loop=nbl.NB_LOOP_CLUSTER)
            out.append(s.get_particles(0, N))
    for q in out[0]:
        assert np.array_equal(out[0][q], out[1][q]), q


@pytest.mark.parametrize("N", [4096, 4097])
def test_resident_rows_match_host_loop(nbl, N):
    m, x, v = inputs.plummer(N, 52, "salpeter")
    T = 2.0 ** -5
    out = []
    for loop in (nbl.NB_LOOP_HOST, nbl.NB_LOOP_CLUSTER):
        with nbl.NBody(N, nbl.NB_MIXED, 0) as s:
            s.set_params(1.0 / 256, 0.01, 2.0 ** -22, T)
            s.set_j_particles(0, m, x, v)
            s.initial_forces_and_dt()
            s.integrate(T, loop=loop)
            out.append(s.get_particles(0, N))
    a, b = out
    assert np.sum(a["dt"] != b["dt"]) <= 0.05 * N
    assert np.abs(a["x"] - b["x"]).max() < 1e-5
    assert np.abs(a["v"] - b["v"]).max() < 1e-4
