"""Small blocks (mixed path): groups of threads share the j of a tile, at the
block sizes where the number of groups changes and one either side, on systems
that fill a tile, leave a ragged one and hold fewer tiles than groups."""
import numpy as np
import pytest

import oracle
from paper_0709_4552_gb300 import inputs
from _util import rel_scalar, rel_vec

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [128, 300, 20000])
@pytest.mark.parametrize("n", [1, 15, 16, 17, 32, 33, 64, 65, 96, 128, 160, 161, 192, 300])
@pytest.mark.parametrize("at", [False, True])
def test_small_block_parity(nbl, N, n, at):
    if n > N:
        pytest.skip("a block holds at most every particle")
    eps = 1.0 / 256
    m, x, v = inputs.plummer(N, 61, "salpeter")
    idx = inputs.sample_indices(N, n, 62)
    with nbl.NBody(N, nbl.NB_MIXED, 0) as s:
        s.set_params(eps, 0.01, 2.0 ** -22, 2.0 ** -3)
        s.set_j_particles(0, m, x, v)
        if at:
            a, j, p = s.compute_forces_at(0.0, idx.astype(np.int32))
        else:
            s.predict(0.0)
            a, j, p = s.compute_forces(idx.astype(np.int32))
        code, _ = s.check_device_status()
        assert code == nbl.NB_OK
    ar, jr, pr = oracle.forces(m, x, v, eps, idx=idx, compensated=True)
    for e in (rel_vec(a, ar), rel_vec(j, jr), rel_scalar(p, pr)):
        assert np.median(e) <= 1e-6 and e.max() <= 1e-5  # the mixed path's bounds
