"""Performance cases of the library: what users run, from the smallest calls to the largest.

A case is a dict of plain values that names an ansatz, a Hamiltonian, a
precision and the call that is made.  ``listed()`` are the standing cases,
``draw()`` further ones of the same ranges; ``prepare()`` makes what a user's
program holds before the call, ``run()`` makes one call, ``work()`` counts
what it cannot do without, and ``exact()`` gives the same results from plain
torch in 64 bits.

Fields of a case:
  call       state | gradient | gradients | energies | loss | batch
  ansatz     hea (RY, RZ, CZ chain) | pc (excitation gates on the Hartree-Fock state)
  ham        chain | ring | lattice | molecular | random
  n, depth   qubits and layers (hea); excitations instead of depth (pc)
  precision  c64 | c128
  starts     parameter vectors per call (energies, gradients)
  threshold  Hamiltonian cutoff (0: every term)
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2402_11878_gb300 as vqe
import vqe_inputs as vi

BATCH_SEED = 7      # the uneven batch's sizes; parameters and U come from the case's seed


def listed():
    return [
        # One look at a small circuit: 4-site open Hubbard chain, state and energy to the host.
        # All latency: a handful of launches and copies.
        {"name": "state_8q_c128", "call": "state", "ansatz": "hea", "ham": "chain", "n": 8, "depth": 4,
         "precision": "c128", "threshold": 0.0},
        # One optimiser iteration on a general Pauli sum with an odd qubit count, host buffers.
        {"name": "gradient_13q_c128", "call": "gradient", "ansatz": "hea", "ham": "random", "n": 13,
         "depth": 6, "precision": "c128", "threshold": 0.0},
        # One optimiser iteration of the particle-conserving ansatz at a size people converge.
        {"name": "pc_gradient_14q_c128", "call": "gradient", "ansatz": "pc", "ham": "chain", "n": 14,
         "n_exc": 60, "precision": "c128", "threshold": 0.0},
        # Many starts advanced together (a step of the batched optimiser), device buffers.
        {"name": "gradients_16q_c128", "call": "gradients", "ansatz": "hea", "ham": "ring", "n": 16,
         "depth": 8, "precision": "c128", "starts": 24, "threshold": 0.0},
        # Energies of many parameter vectors, 10-site periodic chain in FP64.
        {"name": "energies_20q_c128", "call": "energies", "ansatz": "hea", "ham": "ring", "n": 20,
         "depth": 10, "precision": "c128", "starts": 64, "threshold": 0.0},
        # 512 uneven instances (12 to 18 qubits) in one graph launch.
        {"name": "batch_512_c64", "call": "batch", "count": 512, "n_min": 12, "n_max": 18,
         "precision": "c64"},
        # Molecular Hamiltonian (29,737 strings) slimmed at 1e-4: energy and gradient in complex64.
        {"name": "molecular_24q_c64", "call": "gradients", "ansatz": "hea", "ham": "molecular", "n": 24,
         "depth": 12, "precision": "c64", "starts": 1, "threshold": 1e-4},
        # FP64 reference energy of a large ring.
        {"name": "energy_26q_c128", "call": "energies", "ansatz": "hea", "ham": "ring", "n": 26,
         "depth": 8, "precision": "c128", "starts": 1, "threshold": 0.0},
        # Excitation ansatz with 118 parameters at a large size, FP64.
        {"name": "pc_gradient_28q_c128", "call": "gradients", "ansatz": "pc", "ham": "lattice", "n": 28,
         "n_exc": 118, "precision": "c128", "starts": 1, "threshold": 0.0},
        # The same ansatz in complex64, one qubit idle in the Hamiltonian.
        {"name": "pc_gradient_27q_c64", "call": "loss", "ansatz": "pc", "ham": "ring", "n": 27,
         "n_exc": 118, "precision": "c64", "threshold": 0.0},
        # Loss and gradient inside a torch program (float32 parameters), 5x3 lattice, complex64.
        {"name": "loss_30q_c64", "call": "loss", "ansatz": "hea", "ham": "lattice", "n": 30, "depth": 8,
         "precision": "c64", "threshold": 0.0},
        # The largest: FP64 energy and gradient of a 7x2 lattice.
        {"name": "gradient_28q_c128", "call": "gradients", "ansatz": "hea", "ham": "lattice", "n": 28,
         "depth": 8, "precision": "c128", "starts": 1, "threshold": 0.0},
    ]


LATTICES = {20: (5, 2), 24: (4, 3), 28: (7, 2), 30: (5, 3)}


def _starts(rng, n, top):
    """Starts per call: up to `top` amplitudes (log2) in all, at most 128."""
    most = max(1, min(128, 1 << max(0, top - n)))
    return int(round(math.exp(rng.uniform(0.0, math.log(most)))))


def draw(rng):
    kind = rng.choice(["state", "host", "pc_host", "gradients", "energies", "batch", "molecular",
                       "energy", "pc", "loss", "large"])
    if kind == "state":
        return {"call": "state", "ansatz": "hea", "ham": rng.choice(["chain", "random"]),
                "n": rng.randint(4, 16), "depth": rng.randint(1, 8),
                "precision": rng.choice(["c128", "c64"]), "threshold": 0.0}
    if kind == "host":
        return {"call": "gradient", "ansatz": "hea", "ham": rng.choice(["chain", "ring", "random"]),
                "n": rng.randint(6, 18), "depth": rng.randint(2, 10),
                "precision": rng.choice(["c128", "c128", "c64"]), "threshold": 0.0}
    if kind == "pc_host":
        return {"call": "gradient", "ansatz": "pc", "ham": "chain", "n": rng.randint(8, 18),
                "n_exc": rng.randint(10, 118), "precision": rng.choice(["c128", "c64"]),
                "threshold": 0.0}
    if kind == "gradients":
        n = rng.randint(10, 20)
        return {"call": "gradients", "ansatz": "hea", "ham": rng.choice(["chain", "ring"]), "n": n,
                "depth": rng.randint(3, 10), "precision": rng.choice(["c128", "c64"]),
                "starts": _starts(rng, n, 22), "threshold": 0.0}
    if kind == "energies":
        n = rng.randint(14, 22)
        return {"call": "energies", "ansatz": "hea", "ham": rng.choice(["chain", "ring"]), "n": n,
                "depth": rng.randint(4, 12), "precision": rng.choice(["c128", "c64"]),
                "starts": _starts(rng, n, 26), "threshold": 0.0}
    if kind == "batch":
        lo = rng.randint(6, 14)
        return {"call": "batch", "count": int(round(math.exp(rng.uniform(math.log(24), math.log(512))))),
                "n_min": lo, "n_max": rng.randint(lo, 18), "precision": rng.choice(["c64", "c128"])}
    if kind == "molecular":
        return {"call": rng.choice(["gradients", "energies"]), "ansatz": "hea", "ham": "molecular",
                "n": 2 * rng.randint(5, 12), "depth": rng.randint(4, 12), "precision": "c64", "starts": 1,
                "threshold": rng.choice([0.0, 1e-6, 1e-4, 1e-3])}
    if kind == "energy":
        return {"call": "energies", "ansatz": "hea", "ham": "ring", "n": rng.randint(21, 27),
                "depth": rng.randint(4, 8), "precision": "c128", "starts": 1,
                "threshold": rng.choice([0.0, 0.6])}
    if kind == "pc":
        return {"call": "gradients", "ansatz": "pc", "ham": "ring", "n": rng.randint(20, 28),
                "n_exc": rng.randint(30, 118), "precision": rng.choice(["c128", "c64"]), "starts": 1,
                "threshold": 0.0}
    n = rng.randint(20, 27)
    if kind == "loss":
        return {"call": "loss", "ansatz": rng.choice(["hea", "pc"]), "ham": "ring", "n": n,
                "depth": rng.randint(3, 8), "n_exc": rng.randint(30, 118), "precision": "c64",
                "threshold": 0.0}
    return {"call": "gradients", "ansatz": "hea", "ham": "lattice" if n in LATTICES else "ring", "n": n,
            "depth": rng.randint(3, 8), "precision": "c128", "starts": 1, "threshold": 0.0}


# ------------------------------------------------------------------ inputs

def _uniform(seed, low, high):
    return low + (high - low) * float(vi.uniform01(seed, 1, stream=71)[0])


@functools.lru_cache(maxsize=4)
def _molecule(n_spatial, seed):
    return vi.synthetic_molecular(n_spatial, seed)


def _hamiltonian(case, seed):
    """The Pauli sum of a case.  A qubit count that no lattice fills leaves
    the top qubit out of the Hamiltonian."""
    n, ham, U = case["n"], case["ham"], _uniform(seed, 2.5, 8.0)
    if ham == "molecular":
        return _molecule(n // 2, 2024 + seed % 2)
    if ham == "random":
        return vi.random_pauli_sum(n, 5 * n, seed)
    if ham == "lattice":
        return vi.hubbard_2d_snake(*LATTICES[n], 1.0, U, periodic=True)
    return vi.hubbard_1d(n // 2, 1.0, U, periodic=ham == "ring")


def _excitations(case):
    n = case["n"]
    n_singles = max(1, case["n_exc"] // 7)
    return vi.excitations(n, n // 2, n_singles, case["n_exc"] - n_singles, seed=1)


def _n_params(case):
    return len(_excitations(case)) if case["ansatz"] == "pc" else 2 * case["n"] * case["depth"]


def _params(case, seed):
    """Parameter vectors, starts x n_params."""
    def one(s):
        if case["ansatz"] == "pc":
            return vi.excitation_params(s, _n_params(case))
        return vi.ansatz_params(s, case["n"], case["depth"])
    p = np.stack([one(1000 * seed + k) for k in range(case.get("starts", 1))])
    return p.astype(np.float32) if case["call"] == "loss" else p


def _instances(case, seed):
    """Uneven instances: the sizes belong to the case, parameters and U to the seed."""
    sizes = vi.batched_instances(case["count"], BATCH_SEED, case["n_min"], case["n_max"])
    out = []
    for k, ins in enumerate(sizes):
        n, depth = ins["n"], ins["depth"]
        out.append({"n": n, "depth": depth, "U": _uniform(1000 * seed + k, 1.0, 8.0),
                    "params": vi.ansatz_params(1000 * seed + k, n, depth)})
    return out


# ------------------------------------------------------------------ the calls

def prepare(case, seed):
    if case["call"] == "batch":
        ins = _instances(case, seed)
        b = vqe.Batch([i["n"] for i in ins], [i["depth"] for i in ins], precision=case["precision"])
        for k, i in enumerate(ins):
            h = vi.hubbard_1d(i["n"] // 2, 1.0, i["U"])
            b.set_hamiltonian(k, h.x, h.z, h.c)
        p = torch.tensor(np.concatenate([i["params"] for i in ins]), device="cuda")
        return {"call": "batch", "batch": b, "params": p, "grads": torch.empty_like(p),
                "energies": torch.empty(len(ins), dtype=torch.float64, device="cuda")}
    if case["ansatz"] == "pc":
        eng = vqe.Engine.particle_conserving(case["n"], case["n"] // 2, _excitations(case),
                                             case["precision"])
    else:
        eng = vqe.Engine(case["n"], case["depth"], case["precision"])
    h = _hamiltonian(case, seed)
    eng.set_hamiltonian(h.x, h.z, h.c)
    if case["threshold"]:
        eng.slim(case["threshold"])
    p = _params(case, seed)
    s = {"call": case["call"], "engine": eng}
    if case["call"] in ("state", "gradient"):
        s["params"] = p[0]
    elif case["call"] == "loss":
        s["params"] = torch.tensor(p[0], device="cuda", requires_grad=True)
    else:
        s["params"] = torch.tensor(p, device="cuda")
        s["energies"] = torch.empty(len(p), dtype=torch.float64, device="cuda")
        if case["call"] == "energies":
            s["norms"] = torch.empty_like(s["energies"])
        else:
            s["grads"] = torch.empty_like(s["params"])
    return s


def run(s):
    call = s["call"]
    if call == "batch":
        s["batch"].run_dev(s["params"], s["energies"], s["grads"])
        return {"energies": s["energies"], "grads": s["grads"]}
    eng = s["engine"]
    if call == "state":
        eng.apply_ansatz(s["params"])
        energy, norm = eng.energy()
        return {"energy": energy, "norm": norm, "state": eng.get_state()}
    if call == "gradient":
        grad, energy = eng.gradient(s["params"])
        return {"energy": energy, "grad": grad}
    if call == "energies":
        eng.energy_batch_dev(s["params"], s["energies"], s["norms"])
        return {"energies": s["energies"], "norms": s["norms"]}
    if call == "gradients":
        eng.gradient_batch_dev(s["params"], s["grads"], s["energies"])
        return {"energies": s["energies"], "grads": s["grads"]}
    s["params"].grad = None
    loss = vqe.energy_and_grad(s["params"], eng)
    loss.backward()
    return {"loss": loss.detach(), "grad": s["params"].grad}


# ------------------------------------------------------------------ work

L2_BYTES = 129e6    # states up to this size need not touch memory


def _work_one(n, depth, exc, groups, n_terms, amp_bytes, gradient):
    """One evaluation: flops of the gates at one multiply-add per output
    component (a rotation up to its scale), the diagonal once a layer, one
    complex multiply-add per pair and X mask of H; the adjoint's two
    un-applied states and one overlap per parameter.  A state larger than L2
    is written by the circuit and read by the expectation; the gradient writes
    and reads lambda beside it."""
    N = 2.0 ** n
    if exc is None:
        forward = depth * (4.0 * n + 6.0) * N
        backward = depth * (12.0 * n + 16.0) * N
        n_params = 2 * n * depth
    else:
        touched = sum(N / (8.0 if row[1] >= 0 else 2.0) for row in exc)    # amplitudes a gate moves
        forward, backward, n_params = 6.0 * touched, 16.0 * touched, len(exc)
    expect = 4.0 * groups * N
    flops = forward + expect + (backward + expect if gradient else 0.0)
    bytes_ = 8.0 * n_params * (2 if gradient else 1) + 24.0 * n_terms + 16
    if N * amp_bytes > L2_BYTES:
        bytes_ += N * amp_bytes * (4 if gradient else 2)
    return bytes_, flops


def work(case):
    amp = 8 if case["precision"] == "c64" else 16
    if case["call"] == "batch":
        b = f = 0.0
        for ins in vi.batched_instances(case["count"], BATCH_SEED, case["n_min"], case["n_max"]):
            h = ins["H"]
            x, y = _work_one(ins["n"], ins["depth"], None, h.n_groups, len(h), amp, True)
            b, f = b + x, f + y
        return {"bytes": b, "flops": f}
    h = _hamiltonian(case, 0)
    keep = np.abs(h.c) >= case["threshold"]
    exc = _excitations(case) if case["ansatz"] == "pc" else None
    x, y = _work_one(case["n"], case.get("depth", 0), exc, len(np.unique(h.x[keep])), int(keep.sum()), amp,
                     case["call"] in ("gradient", "gradients", "loss"))
    if case["call"] == "state":
        x += 2.0 ** case["n"] * amp
    k = case.get("starts", 1)
    return {"bytes": k * x, "flops": k * y}


# ------------------------------------------------------------------ exact results

def _parity(v):
    for s in (32, 16, 8, 4, 2, 1):
        v = v ^ (v >> s)
    return v & 1


def _sign_rows(z, bits, device):
    """(-1)^popcount(z & i) for i < 2^bits, one row per mask."""
    i = torch.arange(1 << bits, device=device)
    return 1.0 - 2.0 * _parity(z[:, None] & i[None, :]).double()


def _apply_h(psi, h, n):
    """H psi for a batch of states: per X mask one gather times the sum of its
    terms' signs, which is a product of a high and a low half."""
    lo = n // 2
    hi = n - lo
    dev = psi.device
    view = psi.view(-1, 1 << hi, 1 << lo)
    out = torch.zeros_like(view)
    xs, zs, cs = np.asarray(h.x).astype(np.int64), np.asarray(h.z).astype(np.int64), np.asarray(h.c)
    order = np.argsort(xs, kind="stable")
    xs, zs, cs = xs[order], zs[order], cs[order]
    edges = np.flatnonzero(np.r_[True, xs[1:] != xs[:-1]]).tolist() + [len(xs)]
    ih = torch.arange(1 << hi, device=dev)
    il = torch.arange(1 << lo, device=dev)
    for a, b in zip(edges[:-1], edges[1:]):
        x = int(xs[a])
        phase = np.bitwise_count((xs[a:b] & zs[a:b]).astype(np.uint64)) & 3     # (-i)^phase
        moved = view[:, ih ^ (x >> lo)][:, :, il ^ (x & ((1 << lo) - 1))] if x else view
        for odd in (0, 1):
            use = np.flatnonzero((phase & 1) == odd)
            if not len(use):
                continue
            z = torch.tensor(zs[a:b][use], device=dev)
            c = torch.tensor(cs[a:b][use] * np.where(phase[use] >= 2, -1.0, 1.0), device=dev)
            f = (_sign_rows(z >> lo, hi, dev) * c[:, None]).T @ _sign_rows(z & ((1 << lo) - 1), lo, dev)
            if odd:
                out += moved * (f * -1j)
            else:
                out += moved * f
    return out.view(psi.shape)


def _rotate(psi, q, c, s, ph):
    """RY then RZ on qubit q of a batch of states; c, s real and ph complex per state."""
    v = psi.view(psi.shape[0], -1, 2, 1 << q)
    a, b = v[:, :, 0], v[:, :, 1]
    c, s, ph = (t.view(-1, 1, 1) for t in (c, s, ph))
    x = (c * a - s * b) * ph
    y = (s * a + c * b) * ph.conj()
    v[:, :, 0], v[:, :, 1] = x, y


def _unrotate(psi, q, c, s, ph):
    v = psi.view(psi.shape[0], -1, 2, 1 << q)
    c, s, ph = (t.view(-1, 1, 1) for t in (c, s, ph))
    a, b = v[:, :, 0] * ph.conj(), v[:, :, 1] * ph
    x = c * a + s * b
    y = c * b - s * a
    v[:, :, 0], v[:, :, 1] = x, y


def _cz_chain(psi, n):
    for q in range(n - 1):
        psi.view(psi.shape[0], -1, 2, 2, 1 << q)[:, :, 1, 1] *= -1


def _dot(a, b):
    return (a.reshape(a.shape[0], -1).conj() * b.reshape(b.shape[0], -1)).sum(1)


def _exact_hea(n, depth, params, apply_h, gradient):
    """(energies, norms, grads, states) of a batch of parameter vectors."""
    dev = params.device
    B = params.shape[0]
    t = params.view(B, depth, n, 2)
    c, s = torch.cos(t[..., 0] / 2), torch.sin(t[..., 0] / 2)
    ph = torch.polar(torch.ones_like(t[..., 1]), -t[..., 1] / 2)
    psi = torch.zeros(B, 1 << n, dtype=torch.complex128, device=dev)
    psi[:, 0] = 1
    for d in range(depth):
        for q in range(n):
            _rotate(psi, q, c[:, d, q], s[:, d, q], ph[:, d, q])
        _cz_chain(psi, n)
    lam = apply_h(psi)
    norm = _dot(psi, psi).real
    energy = _dot(psi, lam).real / norm
    if not gradient:
        return energy, norm, None, psi
    g = torch.zeros_like(t)
    for d in reversed(range(depth)):
        _cz_chain(psi, n)
        _cz_chain(lam, n)
        for q in reversed(range(n)):
            def halves(v):
                v = v.view(B, -1, 2, 1 << q)
                return v[:, :, 0], v[:, :, 1]
            (p0, p1), (l0, l1) = halves(psi), halves(lam)
            g[:, d, q, 1] = (_dot(l0, p0) - _dot(l1, p1)).imag              # Im <l|Z|p>
            a = (c[:, d, q], s[:, d, q], ph[:, d, q])
            _unrotate(psi, q, *a)
            _unrotate(lam, q, *a)
            (p0, p1), (l0, l1) = halves(psi), halves(lam)
            g[:, d, q, 0] = (_dot(l1, p0) - _dot(l0, p1)).real              # Im <l|Y|p>
    return energy, norm, g.view(B, -1), None


def _exact_pc(n, exc, params, apply_h, gradient):
    dev = params.device
    psi = torch.zeros(1, 1 << n, dtype=torch.complex128, device=dev)
    psi[0, (1 << (n // 2)) - 1] = 1

    def pairs(row):
        """Basis states the excitation acts on, their partners and T's sign."""
        p, q, r, s = (int(v) for v in row)
        gone, made = ([r, s], [p, q]) if q >= 0 else ([r], [p])
        free = [m for m in range(n) if m not in gone + made]
        i = torch.zeros(1, dtype=torch.int64, device=dev)
        for m in free:
            i = torch.cat([i, i | (1 << m)])
        i = i | sum(1 << m for m in gone)
        j, par = i, torch.zeros_like(i)
        for m in reversed(gone):                    # rightmost ladder operator first
            par ^= _parity(j & ((1 << m) - 1))
            j = j ^ (1 << m)
        for m in reversed(made):
            par ^= _parity(j & ((1 << m) - 1))
            j = j ^ (1 << m)
        return i, j, 1.0 - 2.0 * par.double()

    def turn(v, i, j, sg, angle):
        a, b = v[0, i], v[0, j]
        c, s = torch.cos(angle), torch.sin(angle) * sg
        v[0, i] = c * a - s * b
        v[0, j] = c * b + s * a

    for k, row in enumerate(exc):
        turn(psi, *pairs(row), params[0, k])
    lam = apply_h(psi)
    norm = _dot(psi, psi).real
    energy = _dot(psi, lam).real / norm
    if not gradient:
        return energy, norm, None, psi
    g = torch.zeros_like(params)
    for k in reversed(range(len(exc))):
        i, j, sg = pairs(exc[k])
        g[0, k] = 2.0 * (sg * (lam[0, j].conj() * psi[0, i] - lam[0, i].conj() * psi[0, j])).real.sum()
        turn(psi, i, j, sg, -params[0, k])
        turn(lam, i, j, sg, -params[0, k])
    return energy, norm, g, None


def _exact_batch(case, seed):
    """Instances of one size have the same circuit and H = hopping + U * onsite."""
    ins = _instances(case, seed)
    energies, grads = [None] * len(ins), [None] * len(ins)
    for n in sorted({i["n"] for i in ins}):
        L = n // 2
        hop, onsite = vi.hubbard_1d(L, 1.0, 0.0), vi.hubbard_1d(L, 0.0, 1.0)
        where = [k for k, i in enumerate(ins) if i["n"] == n]
        for a in range(0, len(where), 32):
            part = where[a:a + 32]
            p = torch.tensor(np.stack([ins[k]["params"] for k in part]), device="cuda")
            U = torch.tensor([ins[k]["U"] for k in part], dtype=torch.float64, device="cuda")
            e, _, g, _ = _exact_hea(n, ins[part[0]]["depth"], p,
                                    lambda v: _apply_h(v, hop, n) + U[:, None] * _apply_h(v, onsite, n), True)
            for k, x, y in zip(part, e, g):
                energies[k], grads[k] = x, y
    return {"energies": torch.stack(energies), "grads": torch.cat(grads)}


def exact(case, seed):
    call = case["call"]
    if call == "batch":
        return _exact_batch(case, seed)
    n = case["n"]
    if n > 28:              # tens of seconds and of GiB in plain torch
        return None
    h = _hamiltonian(case, seed)
    keep = np.abs(h.c) >= case["threshold"]
    h = vi.PauliSum(n, h.x[keep], h.z[keep], h.c[keep])
    params = torch.tensor(_params(case, seed), device="cuda").double()
    gradient = call in ("gradient", "gradients", "loss")
    got = []
    step = max(1, 1 << max(0, 24 - n))
    for a in range(0, len(params), step):
        p = params[a:a + step]
        if case["ansatz"] == "pc":
            got.append(_exact_pc(n, _excitations(case), p, lambda v: _apply_h(v, h, n), gradient))
        else:
            got.append(_exact_hea(n, case["depth"], p, lambda v: _apply_h(v, h, n), gradient))
    e = torch.cat([r[0] for r in got])
    nn = torch.cat([r[1] for r in got])
    g = torch.cat([r[2] for r in got]) if gradient else None
    if call == "state":
        return {"energy": float(e[0]), "norm": float(nn[0]), "state": got[0][3][0].cpu().numpy()}
    if call == "gradient":
        return {"energy": float(e[0]), "grad": g[0].cpu().numpy()}
    if call == "energies":
        return {"energies": e, "norms": nn}
    if call == "gradients":
        return {"energies": e, "grads": g}
    return {"loss": e[0], "grad": g[0]}
