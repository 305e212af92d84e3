"""FP64 ansatz passes in block fixed point, where they can go wrong: single
threads and partial warps, tile edges, angles at the boundaries of the
coefficient forms, extreme scales of lambda, and non-finite parameters.

Tolerances: amplitudes 1e-12 and gradients 1e-10 as everywhere in FP64.  The
norm: every gate and table entry is unitary to 2^-57, and the rounding to
doubles after each pass is unbiased, so 1e-15 per pass bounds its drift.
"""
import numpy as np
import pytest

import oracle
import vqe_inputs as vi

pytestmark = pytest.mark.gpu


def engine(n, depth):
    import paper_2402_11878_gb300 as pkg
    return pkg.Engine(n, depth, "c128")


def boundary_params(n, depth, seed):
    """theta at multiples of pi/8 (where the coefficient forms meet), moved by
    rounding-size and tiny steps, zeros and large angles."""
    r = np.random.RandomState(seed)
    count = 2 * n * depth
    p = r.randint(-16, 17, count) * np.pi / 8
    kind = r.randint(0, 6, count)
    p[kind == 1] *= 1 + 1e-15
    p[kind == 2] += r.uniform(-1, 1, (kind == 2).sum()) * 10.0 ** r.uniform(-14, -1, (kind == 2).sum())
    p[kind == 3] = 0.0
    p[kind == 4] = r.uniform(-1e6, 1e6, (kind == 4).sum())
    return p


@pytest.mark.parametrize("n,depth,tile_bits", [(3, 5, 0), (4, 3, 0), (7, 4, 0), (8, 7, 0), (9, 2, 0),
                                               (10, 3, 0), (11, 6, 0), (12, 3, 0), (13, 4, 12),
                                               (13, 3, 9), (17, 2, 0), (12, 42, 12)])
@pytest.mark.parametrize("kind", ["uniform", "boundary", "zero"])
def test_state_and_gradient(n, depth, tile_bits, kind):
    if kind == "uniform":
        p = vi.ansatz_params(5, n, depth)
    else:
        p = boundary_params(n, depth, 7) if kind == "boundary" else np.zeros(2 * n * depth)
    H = vi.random_pauli_sum(n, 2 * n + 3, 3)
    eng = engine(n, depth)
    if tile_bits:
        eng.set_plan_options(tile_bits, 2, 3)
    eng.set_hamiltonian(H.x, H.z, H.c)
    eng.apply_ansatz(p)
    psi = eng.get_state()
    _, norm = eng.energy()
    ref = oracle.ansatz_state(n, depth, p)
    assert np.max(np.abs(psi - ref)) <= 1e-12
    passes = eng.stats()["ansatz_passes"]
    assert abs(norm - 1.0) <= 1e-15 * (passes + 1)
    g, e = eng.gradient(p)
    g_ref, e_ref = oracle.gradient_adjoint(n, depth, p, H.x, H.z, H.c)
    assert abs(e - e_ref) <= 1e-11 * H.sum_abs()
    assert np.max(np.abs(g - g_ref)) <= 1e-10 * max(1.0, np.max(np.abs(g_ref)))


@pytest.mark.parametrize("power", [-900, -40, 40, 900])
def test_gradient_scales_exactly(power):
    """A power of two on H only changes lambda's exponents: the same integers."""
    n, depth = 13, 3
    H = vi.random_pauli_sum(n, 20, 9)
    p = vi.ansatz_params(11, n, depth)
    eng = engine(n, depth)
    eng.set_hamiltonian(H.x, H.z, H.c)
    g, _ = eng.gradient(p)
    eng.set_hamiltonian(H.x, H.z, np.ldexp(H.c, power))
    gs, _ = eng.gradient(p)
    assert np.array_equal(np.ldexp(g, power), gs)


@pytest.mark.parametrize("n", [9, 13])
def test_non_finite_parameter_stays_in_its_state(n):
    import torch
    depth = 3
    H = vi.hubbard_1d(n // 2, 1.0, 4.0)
    P = np.stack([vi.ansatz_params(s, n, depth) for s in range(3)])
    eng = engine(n, depth)
    eng.set_hamiltonian(H.x, H.z, H.c)
    clean = torch.tensor(P, device="cuda")
    e0 = torch.empty(3, dtype=torch.float64, device="cuda")
    g0 = torch.empty_like(clean)
    eng.gradient_batch_dev(clean, g0, e0)
    P[1, n + 3] = np.nan
    bad = torch.tensor(P, device="cuda")
    e1, g1 = torch.empty_like(e0), torch.empty_like(g0)
    eng.gradient_batch_dev(bad, g1, e1)
    torch.cuda.synchronize()
    assert torch.isnan(e1[1]) and torch.isnan(g1[1]).any()
    for k in (0, 2):
        assert e1[k] == e0[k] and torch.equal(g1[k], g0[k])
