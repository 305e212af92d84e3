"""Amplitudes far below their tile's norm: FP64 layered circuits of small angles.

Against the same circuit in long double.  Tolerance per amplitude: FP64 gates err
by a few units of the last place of the terms they add, so with M the circuit of
the gates' absolute values applied to |0...0>, |error_i| <= 8 n D 2^-53 M_i (per
qubit and layer: 3 units for tangent and butterfly, 2 for the scale, 3 for the
phase).  Where a tile's amplitudes spread over less than 2^8 the passes may run in
block fixed point: each operation adds at most 1.5 units of 2^-61 of the tile's norm
to each of its 2^k amplitudes, two operations per qubit and layer, and the gates
keep the 2-norm of what was added: 3 n D 2^(k/2 - 61) more.
"""
import functools

import numpy as np
import pytest

import vqe_inputs as vi

pytestmark = pytest.mark.gpu
LD = np.longdouble


def circuit(n, depth, params):
    """(re, im, M) in long double."""
    p = np.asarray(params).astype(LD).reshape(depth, n, 2) / 2
    c, s = np.cos(p), np.sin(p)
    re, im, big = (np.zeros(1 << n, LD) for _ in range(3))
    re[0] = big[0] = 1
    i = np.arange(1 << n, dtype=np.uint64)
    cz = np.where(np.bitwise_count(i & (i >> np.uint64(1))) & 1, LD(-1), LD(1))

    def halves(v, q):
        v = v.reshape(-1, 2, 1 << q)
        return v[:, 0], v[:, 1]

    for d in range(depth):
        for q in range(n):
            (ct, cp), (st, sp) = c[d, q], s[d, q]
            for v, sign in ((re, -1), (im, -1), (big, 1)):
                x, y = halves(v, q)
                a, b = (abs(ct), abs(st)) if sign > 0 else (ct, st)
                new = a * x + sign * b * y, b * x + a * y
                x[:], y[:] = new
            (r0, r1), (i0, i1) = halves(re, q), halves(im, q)
            new = r0 * cp + i0 * sp, i0 * cp - r0 * sp, r1 * cp - i1 * sp, i1 * cp + r1 * sp
            r0[:], i0[:], r1[:], i1[:] = new
        re *= cz
        im *= cz
    return re, im, big


def angles(kind, n, depth, seed=3):
    r = np.random.RandomState(seed)
    if kind == "uniform":
        return vi.ansatz_params(seed, n, depth)
    if kind == "near":      # steps from multiples of pi
        return r.randint(-2, 3, 2 * n * depth) * np.pi + r.normal(size=2 * n * depth) * 1e-3
    if kind == "one layer":     # a single layer turns the qubits, by little
        p = np.zeros((depth, n, 2))
        p[depth // 2] = r.normal(size=(n, 2)) * 1e-4
        return p.ravel()
    return r.normal(size=2 * n * depth) * kind


reference = functools.lru_cache(maxsize=None)(lambda kind, n, depth: circuit(n, depth, angles(kind, n, depth)))


def tolerance(n, depth, big, fixed_point, tile_bits):
    tol = 8 * n * depth * 2.0**-53 * big
    return tol + 3 * n * depth * 2.0 ** (min(n, tile_bits) / 2 - 61) if fixed_point else tol


@pytest.mark.parametrize("n,depth,tile_bits", [(4, 3, 0), (7, 2, 0), (9, 4, 0), (11, 1, 0), (12, 3, 0), (13, 2, 0),
                                               (13, 3, 9), (13, 3, 12), (11, 12, 0)])
@pytest.mark.parametrize("kind", [1e-2, 1e-3, 1e-6, 1e-12, "near", "one layer", 0.1])
def test_every_amplitude_of_small_angles(n, depth, tile_bits, kind):
    import paper_2402_11878_gb300 as pkg
    re, im, big = reference(kind, n, depth)
    eng = pkg.Engine(n, depth, "c128")
    if tile_bits:
        eng.set_plan_options(tile_bits, 2, 3)
    eng.apply_ansatz(angles(kind, n, depth))
    psi = eng.get_state()
    err = np.hypot(psi.real.astype(LD) - re, psi.imag.astype(LD) - im)
    assert np.all(err <= tolerance(n, depth, big, False, 0))


@pytest.mark.parametrize("n,depth", [(3, 8), (9, 10), (12, 12), (13, 10)])
def test_every_amplitude_of_generic_angles(n, depth):
    import paper_2402_11878_gb300 as pkg
    re, im, big = reference("uniform", n, depth)
    eng = pkg.Engine(n, depth, "c128")
    eng.apply_ansatz(angles("uniform", n, depth))
    psi = eng.get_state()
    err = np.hypot(psi.real.astype(LD) - re, psi.imag.astype(LD) - im)
    assert np.all(err <= tolerance(n, depth, big, True, 11))
    assert np.sqrt((err**2).sum()) <= 2e-15      # rounding errors of 4 10^3 operations at 2^-61 of the norm and the store


@pytest.mark.parametrize("n", [9, 13])
def test_states_of_one_batch_choose_for_themselves(n):
    import torch
    import paper_2402_11878_gb300 as pkg
    depth = 6
    H = vi.random_pauli_sum(n, 3 * n, 5)
    P = np.stack([angles(k, n, depth, seed=s) for s, k in enumerate(["uniform", 1e-2, "uniform", "near", 0.1])])
    eng = pkg.Engine(n, depth, "c128")
    eng.set_hamiltonian(H.x, H.z, H.c)
    p = torch.tensor(P, device="cuda")
    g, e = torch.empty_like(p), torch.empty(len(P), dtype=torch.float64, device="cuda")
    eng.gradient_batch_dev(p, g, e)
    torch.cuda.synchronize()
    for k in range(len(P)):
        g1, e1 = eng.gradient(P[k])
        # blocks of the energy share the states of a batch differently: rounding of the sums
        assert abs(e1 - float(e[k])) <= 1e-13 * H.sum_abs()
        assert np.max(np.abs(g1 - g[k].cpu().numpy())) <= 1e-12 * max(1.0, np.max(np.abs(g1)))


@pytest.mark.parametrize("n,depth", [(5, 2), (9, 3), (13, 3), (17, 2)])
@pytest.mark.parametrize("kind", [1e-3, "near"])
def test_gradient_of_small_angles_against_floating_point_plans(n, depth, kind):
    """reg_bits 2 always runs in FP64: the same sums, in another order."""
    import paper_2402_11878_gb300 as pkg
    H = vi.random_pauli_sum(n, 3 * n, 5)
    p = angles(kind, n, depth)
    out = []
    for reg_bits in (3, 2):
        eng = pkg.Engine(n, depth, "c128")
        eng.set_plan_options(0, 0, reg_bits)
        eng.set_hamiltonian(H.x, H.z, H.c)
        out.append(eng.gradient(p))
    (g, e), (g2, e2) = out
    assert abs(e - e2) <= 1e-13 * H.sum_abs()
    assert np.max(np.abs(g - g2)) <= 1e-13 * H.sum_abs()
