"""What the benchmark counts beside its times."""
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))


def test_the_first_excitation_pass_writes_the_whole_state():
    import bench
    # 4 qubits, 2 electrons: 2 x 2 amplitudes with one electron of either spin
    fwd, bwd = bench.excitation_pass_bytes(4, 2, 3, 16.0)
    assert fwd == 16 * (2**4 + 2 * 2 * 4)      # a whole write, then two passes of read + write
    assert bwd == 16 * 3 * 4 * 4               # psi and lambda, read + write
