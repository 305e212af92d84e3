"""The excitation passes hold only the amplitudes of the n_elec sector that a
pass's gates pair: fillings from empty to full, excitations without a pair in
the sector, Hamiltonians that leave the sector, the block widths (a grid of more
than 608 blocks takes a narrower one, FP64 forward again from 2048) and an angle that is not a number.

Tolerances as in test_gpu_pc.py; the block widths add the same terms in
another order: FP64 1e-13 of the gradient's largest entry, complex64
(compensated FP32 partials, 2^-46 of the sum of the terms' magnitudes) 1e-9.
"""
import numpy as np
import pytest

import vqe_inputs as vi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg(lib_built):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    import paper_2402_11878_gb300 as p
    return p


def _any_excitations(n, count, seed):
    """Excitations between arbitrary modes, singles and doubles mixed."""
    rng = np.random.default_rng(seed)
    out = []
    for j in range(count):
        m = rng.permutation(n)[:4]
        out.append([m[0], -1, m[1], -1] if j % 3 == 0 else list(m))
    return np.array(out, dtype=np.int32)


def _random_hamiltonian(n, terms, seed):
    rng = np.random.default_rng(seed)
    return vi.PauliSum(n, rng.integers(0, 1 << n, terms), rng.integers(0, 1 << n, terms),
                       rng.uniform(-1, 1, terms))


@pytest.mark.parametrize("prec", ["c128", "c64"])
@pytest.mark.parametrize("n,ne", [(4, 0), (5, 5), (11, 3), (12, 1), (12, 6), (13, 0), (13, 12), (14, 14), (15, 4)])
def test_fillings(pkg, oracle_mod, prec, n, ne):
    exc, H = _any_excitations(n, 40, n + ne), _random_hamiltonian(n, 30, n)
    th = np.random.default_rng(ne).uniform(-3, 3, len(exc))
    eng = pkg.Engine.particle_conserving(n, ne, exc, prec)
    eng.set_hamiltonian(H.x, H.z, H.c)
    eng.apply_ansatz(th)
    ref = oracle_mod.pc_ansatz_state(n, ne, exc, th)
    assert np.max(np.abs(eng.get_state() - ref)) <= (1e-12 if prec == "c128" else 2e-6)
    g, E = eng.gradient(th)
    g_ref, E_ref = oracle_mod.pc_gradient_adjoint(n, ne, exc, th, H.x, H.z, H.c)
    assert abs(E - E_ref) <= (1e-11 if prec == "c128" else 1e-5) * H.sum_abs()
    scale = max(1.0, float(np.max(np.abs(g_ref))))
    assert np.max(np.abs(g - g_ref)) <= (1e-10 if prec == "c128" else 1e-4) * scale
    eng.close()


@pytest.mark.parametrize("prec", ["c128", "c64"])
@pytest.mark.parametrize("order", ["alternating", "halves"])
@pytest.mark.parametrize("n,ne", [(8, 3), (13, 7), (14, 2), (15, 8)])
def test_spins_kept_apart(pkg, oracle_mod, prec, order, n, ne):
    """Excitations that keep each spin's electrons, under both mode orders;
    the Hamiltonian keeps neither."""
    rng = np.random.default_rng(17 * n + ne)
    up = np.arange(0, n, 2) if order == "alternating" else np.arange(n // 2)
    down = np.setdiff1d(np.arange(n), up)
    exc = []
    for j in range(36):
        a, b = rng.permutation(up), rng.permutation(down)
        exc.append([[a[0], -1, a[1], -1], [b[0], -1, b[1], -1], [a[0], b[0], a[1], b[1]],
                    [a[0], b[0], b[1], a[1]], [*a[:4]] if len(a) > 3 else [a[0], -1, a[2], -1]][j % 5])
    exc, H = np.array(exc, dtype=np.int32), _random_hamiltonian(n, 30, n)
    th = rng.uniform(-3, 3, len(exc))
    eng = pkg.Engine.particle_conserving(n, ne, exc, prec)
    eng.set_hamiltonian(H.x, H.z, H.c)
    g, E = eng.gradient(th)
    g_ref, E_ref = oracle_mod.pc_gradient_adjoint(n, ne, exc, th, H.x, H.z, H.c)
    assert abs(E - E_ref) <= (1e-11 if prec == "c128" else 1e-5) * H.sum_abs()
    scale = max(1.0, float(np.max(np.abs(g_ref))))
    assert np.max(np.abs(g - g_ref)) <= (1e-10 if prec == "c128" else 1e-4) * scale
    eng.apply_ansatz(th)
    ref = oracle_mod.pc_ansatz_state(n, ne, exc, th)
    assert np.max(np.abs(eng.get_state() - ref)) <= (1e-12 if prec == "c128" else 2e-6)
    eng.close()


@pytest.mark.parametrize("prec", ["c128", "c64"])
@pytest.mark.parametrize("n,ne,batch", [(11, 4, 1), (12, 0, 1), (12, 6, 3), (13, 12, 1), (14, 7, 1), (15, 15, 2), (16, 5, 1)])
def test_sweep_over_the_sector(pkg, oracle_mod, prec, n, ne, batch):
    """lambda = H psi by sweeps over the sector's states (chunks of 2^12
    counter values: one that is not full, one, several)."""
    exc, H = _any_excitations(n, 30, 3 * n + ne), _random_hamiltonian(n, 30, 7 * n)
    P = np.random.default_rng(n).uniform(-3, 3, (batch, len(exc)))
    eng = pkg.Engine.particle_conserving(n, ne, exc, prec)
    eng.set_hamiltonian(H.x, H.z, H.c)
    assert eng.set_apply_mode(2) == 2
    G, E = eng.gradient_batch(P)
    for b in range(batch):
        g_ref, E_ref = oracle_mod.pc_gradient_adjoint(n, ne, exc, P[b], H.x, H.z, H.c)
        assert abs(E[b] - E_ref) <= (1e-11 if prec == "c128" else 1e-5) * H.sum_abs()
        scale = max(1.0, float(np.max(np.abs(g_ref))))
        assert np.max(np.abs(G[b] - g_ref)) <= (1e-10 if prec == "c128" else 1e-4) * scale
    eng.close()


@pytest.mark.parametrize("prec,batch", [("c128", 160), ("c128", 300), ("c64", 300)])
def test_block_widths(pkg, prec, batch):
    n = 14
    exc, H = vi.excitations(n, 6, 8, 24, seed=2), vi.hubbard_1d(7, 1.0, 4.0)
    P = np.random.default_rng(5).uniform(-2, 2, (batch, len(exc)))
    eng = pkg.Engine.particle_conserving(n, 6, exc, prec)
    eng.set_hamiltonian(H.x, H.z, H.c)
    G, E = eng.gradient_batch(P)
    for b in (0, 1, batch // 2, batch - 1):
        g, e = eng.gradient(P[b])
        tol = (1e-13 if prec == "c128" else 1e-9) * max(1.0, float(np.max(np.abs(g))))
        assert np.max(np.abs(G[b] - g)) <= tol
        assert abs(E[b] - e) <= (1e-13 if prec == "c128" else 1e-9) * H.sum_abs()
    eng.close()


@pytest.mark.parametrize("prec", ["c128", "c64"])
def test_an_angle_that_is_not_a_number_shows(pkg, prec):
    import torch
    # one electron: the double has no pair
    H = vi.hubbard_1d(6, 1.0, 4.0)
    eng = pkg.Engine.particle_conserving(12, 1, [[3, -1, 0, -1], [4, 5, 1, 2]], prec)
    eng.set_hamiltonian(H.x, H.z, H.c)
    P = torch.tensor([[np.nan, 0.1], [0.1, np.nan], [np.inf, 0.0], [0.1, 0.2]], dtype=torch.float64, device="cuda")
    G, E = torch.empty_like(P), torch.empty(4, dtype=torch.float64, device="cuda")
    eng.gradient_batch_dev(P, G, E)   # host parameters are refused, device ones are not looked at
    assert torch.isnan(E).tolist() == [True, True, True, False]
    eng.close()
