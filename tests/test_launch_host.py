"""What the host queues, seen through a CUDA runtime that records it (fake_cudart.cpp)."""
import ctypes
import glob
import os
import subprocess

import numpy as np
import pytest

import vqe_inputs as vi

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fake_lib(tmp_path_factory):
    from paper_2402_11878_gb300 import build
    objs = sorted(glob.glob(os.path.join(build.OBJ_DIR, "*.cu.o")))
    built = build.build(force=len(objs) != len(build.sources()))
    objs = [os.path.join(build.OBJ_DIR, os.path.basename(s) + ".o") for s in build.sources()]
    out = str(tmp_path_factory.mktemp("fake") / "libvqe_fake.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-std=c++17", "-Wl,-Bsymbolic", "-I", cuda, "-o", out,
                    os.path.join(HERE, "fake_cudart.cpp")] + objs, check=True)
    assert built
    return out


@pytest.fixture
def runtime(fake_lib, monkeypatch):
    from paper_2402_11878_gb300 import binding
    monkeypatch.setattr(binding, "LIB_PATH", fake_lib)
    monkeypatch.setattr(binding, "_lib", None)
    lib = ctypes.CDLL(fake_lib)
    lib.fake_record.restype = ctypes.c_char_p

    class Runtime:
        engine = binding.Engine

        def reset(self, static_bytes=1024):
            lib.fake_reset(static_bytes)

        def events(self, kind):
            rows = [line.split() for line in lib.fake_record().decode().splitlines()]
            return [r[1:] for r in rows if r[0] == kind]

    r = Runtime()
    r.reset()
    return r


@pytest.mark.parametrize("n", [8, 13, 22])
@pytest.mark.parametrize("ansatz", ["hea", "pc"])
@pytest.mark.parametrize("precision", ["c64", "c128"])
@pytest.mark.parametrize("ham", ["chain", "random"])
def test_the_first_kernel_of_a_call_is_launched_plainly(runtime, n, ansatz, precision, ham):
    if ansatz == "pc":
        eng = runtime.engine.particle_conserving(n, n // 2, vi.excitations(n, n // 2, 2, 6, seed=1), precision)
    else:
        eng = runtime.engine(n, 2, precision)
    h = vi.hubbard_1d(n // 2, 1.0, 4.0) if ham == "chain" else vi.random_pauli_sum(n, 2 * n, 3)
    eng.set_hamiltonian(h.x, h.z, h.c)
    p = np.zeros(eng.n_params)
    eng.apply_ansatz(p)
    calls = [lambda: eng.apply_ansatz(p), eng.energy, lambda: eng.gradient(p), lambda: eng.energy_batch(p)]
    for call in calls:
        runtime.reset()
        call()
        kinds = [e[2] for e in runtime.events("launch")]
        assert kinds[0] == "plain" and len(kinds) >= 2


def _one_wide_group(n, n_terms):
    """One X mask of six bits, which the sweeps keep term by term: 20 bytes of
    tables per FP64 term and 4132 beside them."""
    z = np.arange(n_terms, dtype=np.uint64) << np.uint64(6)     # no Y: every term real
    return np.full(n_terms, 0b111111, dtype=np.uint64), z, np.linspace(0.1, 1.0, n_terms)


@pytest.mark.parametrize("n_terms", [2244, 2245, 2251, 2252])
def test_sweep_tables_about_48_kib(runtime, n_terms):
    """48 KiB hold the tables and the kernel's static 136 bytes, not the tables alone."""
    eng = runtime.engine(18, 1, "c128")
    eng.set_hamiltonian(*_one_wide_group(18, n_terms))
    assert eng.set_apply_mode(2) == 2
    runtime.reset(static_bytes=136)
    eng.gradient(np.zeros(eng.n_params))
    sizes = [int(e[1]) for e in runtime.events("launch") if "k_apply_h_sweep" in e[0]]
    assert sizes == [4132 + 20 * n_terms]


def test_a_smaller_launch_never_lowers_a_kernels_limit(runtime):
    """The limit belongs to the process: a thread that lowers it to its own launch's
    size refuses the larger launch another thread is about to make."""
    def pc(n, count, precision):
        return runtime.engine.particle_conserving(n, n // 2, vi.excitations(n, n // 2, count // 7, count, seed=1),
                                                  precision)

    def hea(n, depth, precision, *options):
        eng = runtime.engine(n, depth, precision)
        if options:
            eng.set_plan_options(*options)
        return eng

    runtime.reset()
    for make in (lambda: hea(14, 24, "c128"), lambda: hea(14, 2, "c128"), lambda: hea(14, 3, "c64", 13, 3, 4),
                 lambda: hea(14, 3, "c64", 12, 3, 3), lambda: hea(14, 3, "c64"), lambda: hea(14, 2, "c128", 12, 2, 4),
                 lambda: hea(14, 2, "c128", 11, 2, 2), lambda: hea(14, 12, "c128", 12, 2, 3),
                 lambda: hea(14, 2, "c128", 12, 2, 3), lambda: pc(14, 60, "c128"), lambda: pc(16, 8, "c128"),
                 lambda: pc(14, 60, "c64"), lambda: pc(16, 8, "c64")):
        eng = make()
        h = vi.hubbard_1d(eng.n // 2, 1.0, 4.0)
        eng.set_hamiltonian(h.x, h.z, h.c)
        eng.gradient(np.zeros(eng.n_params))
    limits = {}
    for name, value in runtime.events("limit"):
        limits.setdefault(name, set()).add(int(value))
    assert len(limits) >= 6
    assert {n: v for n, v in limits.items() if len(v) > 1} == {}


@pytest.mark.parametrize("n,kind", [(14, "early"), (15, "plain"), (16, "plain"), (17, "plain"), (18, "early")])
def test_passes_do_not_start_beside_a_grid_that_leaves_some_sms(runtime, n, kind):
    """apply-H of a general Pauli sum has 2^(n - 9) blocks (152 SMs): the passes behind
    its energy reduction may start early only beside a grid of up to 38 blocks, or one
    that fills the chip."""
    eng = runtime.engine(n, 2, "c128")
    h = vi.random_pauli_sum(n, 5 * n, 1)
    eng.set_hamiltonian(h.x, h.z, h.c)
    assert eng.set_apply_mode(0) == 0
    runtime.reset()
    eng.gradient(np.zeros(eng.n_params))
    rows = runtime.events("launch")
    at = [i for i, r in enumerate(rows) if "k_apply_h" in r[0]][0]
    assert "k_energy_finish" in rows[at + 1][0] and rows[at + 1][2] == kind
