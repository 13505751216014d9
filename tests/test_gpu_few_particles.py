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


@pytest.mark.parametrize("N", [130, 299, 300, 20000])
@pytest.mark.parametrize("n", [1, 15, 16, 17, 31, 32, 33, 64, 65, 96, 97, 129, 160, 161])
@pytest.mark.parametrize("noalloc", [False, True])
def test_small_fp64_block_parity(nbl, N, n, noalloc):
    # FP64: every pair is at least as accurate as in FP64 arithmetic, so the sum
    # is good to a few units of the sum of the terms' magnitudes
    if n > N:
        pytest.skip("a block holds at most every particle")
    torch = pytest.importorskip("torch")
    eps = 1.0 / 256
    m, x, v = inputs.plummer(N, 63, "salpeter")
    x[7] = x[N // 2] + 1e-9  # a pair closer than the tiles' grid resolves
    idx = inputs.sample_indices(N, n, 64)
    if noalloc:
        dev = lambda q: torch.from_numpy(np.ascontiguousarray(q)).cuda()
        out = [torch.empty((n, 3), dtype=torch.float64, device="cuda") for _ in range(2)]
        out.append(torch.empty(n, dtype=torch.float64, device="cuda"))
        nbl.nb_forces_fp64_noalloc(dev(m), dev(x), dev(v), eps, dev(idx.astype(np.int32)), *out)
        torch.cuda.synchronize()
        a, j, p = (q.cpu().numpy() for q in out)
    else:
        with nbl.NBody(N, nbl.NB_FP64, 0) as s:
            s.set_params(eps, 0.01, 2.0 ** -22, 2.0 ** -3)
            s.set_j_particles(0, m, x, v)
            s.predict(0.0)
            a, j, p = s.compute_forces(idx.astype(np.int32))
    ar, jr, pr = oracle.forces(m, x, v, eps, idx=idx, compensated=True)
    for e in (rel_vec(a, ar), rel_vec(j, jr), rel_scalar(p, pr)):
        assert e.max() <= 1e-12  # the FP64 path's bound
