"""Caller lists visited in spatial order (mixed path): the order found by
counting slots, at the sizes where it could go wrong (chunks of 1024 slots, one
list entry below and above the line, nearly every particle, every particle)."""
import numpy as np
import pytest

import oracle
from paper_0709_4552_gb300 import inputs
from _util import rel_scalar, rel_vec

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [32768, 1 << 19])
@pytest.mark.parametrize("pick", ["line_below", "line", "all_but_one", "all", "one_chunk"])
@pytest.mark.parametrize("at", [False, True])
def test_ordered_list_parity(nbl, N, pick, at):
    n = {"line_below": max(1024, (1 << 29) // N) - 1, "line": max(1024, (1 << 29) // N), "all_but_one": N - 1, "all": N,
         "one_chunk": max(1024, (1 << 29) // N)}[pick]
    if N > 1 << 18 and n > 1 << 14:
        pytest.skip("the small system covers whole lists")
    eps = 1.0 / 1024
    m, x, v = inputs.plummer(N, 31)
    # one_chunk: n consecutive particles; the others seeded subsets
    idx = np.arange(N // 3, N // 3 + n) if pick == "one_chunk" else inputs.sample_indices(N, n, 32)
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
    k = np.unique(np.linspace(0, n - 1, 400).astype(int))
    ar, jr, pr = oracle.forces(m, x, v, eps, idx=idx[k], compensated=True)
    for e in (rel_vec(a[k], ar), rel_vec(j[k], jr), rel_scalar(p[k], pr)):
        assert np.median(e) <= 1e-6 and e.max() <= 1e-5  # the mixed path's bounds


def test_repeated_entries_are_reported(nbl):
    # a device list with repeats: reported as before, and no access out of bounds
    torch = pytest.importorskip("torch")
    N = 1 << 19
    m, x, v = inputs.plummer(N, 33)
    dev = lambda q: torch.from_numpy(np.ascontiguousarray(q)).cuda()
    with nbl.NBody(N, nbl.NB_MIXED, 0, stream=torch.cuda.current_stream()) as s:
        s.set_j_particles(0, dev(m), dev(x), dev(v))
        s.predict(0.0)
        idx = torch.arange(2048, device="cuda", dtype=torch.int32) // 2
        out = [torch.empty((2048, 3), dtype=torch.float64, device="cuda") for _ in range(2)]
        s.compute_forces(idx, out[0], out[1], None)
        code, _ = s.check_device_status()
        assert code == nbl.NB_EINVAL
        s.clear_error()
