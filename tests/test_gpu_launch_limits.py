"""Launches at the limits of shared memory."""
import numpy as np
import pytest

import vqe_inputs as vi
from test_launch_host import _one_wide_group

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_terms", [2245, 2251])
def test_sweep_tables_just_below_48_kib(n_terms):
    """FP64 sums of n_terms terms of size <= 1 in two orders."""
    import paper_2402_11878_gb300 as pkg
    n, depth = 18, 2
    p = vi.ansatz_params(3, n, depth)
    x, z, c = _one_wide_group(n, n_terms)
    out = []
    for mode in (2, 0):
        eng = pkg.Engine(n, depth, "c128")
        eng.set_hamiltonian(x, z, c)
        assert eng.set_apply_mode(mode) == mode
        out.append(eng.gradient(p))
    (g, e), (g0, e0) = out
    assert abs(e - e0) <= 1e-13 * c.sum()
    assert np.max(np.abs(g - g0)) <= 1e-13 * c.sum()
