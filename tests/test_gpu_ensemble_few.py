"""Mixed ensembles on either side of the line between the two force kernels (a
step of few items, whose warps share each item's j-tiles, and one of many), with
cluster sizes about the i-tile of 32 and the j-tile of 128."""
import numpy as np
import pytest

import oracle
from paper_0709_4552_gb300 import inputs
from _util import rel_scalar, rel_vec

pytestmark = pytest.mark.gpu

SIZES = [2, 31, 32, 33, 127, 128, 129, 300, 1000]


# every particle active: 9 small clusters are 300 items; 24 clusters of 1500 more
# are 13000, past four per resident CTA of any GPU this runs on
@pytest.mark.parametrize("more", [0, 24])
def test_first_forces_of_every_cluster(nbl, more):
    sizes = SIZES + [1500] * more
    ics = [inputs.plummer(n, 70 + q, "salpeter") for q, n in enumerate(sizes)]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    m, x, v = (np.concatenate([c[k] for c in ics]) for k in range(3))
    eps = np.full(len(sizes), 1.0 / 256)
    with nbl.Ensemble(off, eps, nbl.NB_MIXED, 0) as e:
        e.set_params(0.01, 0.01, 2.0 ** -22, 2.0 ** -6)
        e.set_j_particles(0, m, x, v)
        e.initial_forces_and_dt()
        st = e.get_particles(0, len(m))
    for q, (mc, xc, vc) in enumerate(ics[:len(SIZES) + 1]):
        s = slice(off[q], off[q + 1])
        ar, jr, pr = oracle.forces(mc, xc, vc, eps[q], compensated=True)
        for err in (rel_vec(st["a"][s], ar), rel_vec(st["jerk"][s], jr), rel_scalar(st["pot"][s], pr)):
            assert np.median(err) <= 1e-6 and err.max() <= 1e-5  # the mixed path's bounds


@pytest.mark.parametrize("more", [0, 24])
def test_steps_match_the_per_cluster_loop(nbl, more):
    sizes = SIZES[4:] + [1500] * more
    ics = [inputs.plummer(n, 80 + q, "salpeter") for q, n in enumerate(sizes)]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    m, x, v = (np.concatenate([c[k] for c in ics]) for k in range(3))
    t_end = 2.0 ** -6
    out = []
    for mode in (nbl.NB_ENSEMBLE_PERSISTENT, nbl.NB_ENSEMBLE_PER_CLUSTER):
        with nbl.Ensemble(off, np.full(len(sizes), 1.0 / 256), nbl.NB_MIXED, 0) as e:
            e.set_params(0.01, 0.01, 2.0 ** -22, t_end)
            e.set_j_particles(0, m, x, v)
            e.initial_forces_and_dt()
            nbl.nb_ensemble_integrate(e.ctx, t_end, mode)
            out.append(e.get_particles(0, len(m)))
    a, b = out
    assert np.all(a["t"] == t_end) and np.all(b["t"] == t_end)
    assert np.mean(a["dt"] == b["dt"]) > 0.95  # sums group differently
    assert np.abs(a["x"] - b["x"]).max() < 1e-5
