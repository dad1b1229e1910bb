"""Half B in half A's memory: so many bitstrings that both halves stay, and few, give the same
amplitudes bit for bit."""
import numpy as np
import pytest

from paper_1804_04797_gb300 import inputs, sv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize('rows,cols,depth,half_a,full', [
    (4, 4, 9, 0xFF, False), (4, 4, 9, 0xFF, True), (3, 5, 10, 0x1F, False), (3, 5, 8, 0x3FF, False),
    (2, 7, 7, 0x1, False)])
def test_number_of_bitstrings_changes_no_amplitude(rows, cols, depth, half_a, full):
    lat = inputs.lattice_for(rows, cols, depth, seed=21)
    n = lat.n_qubits
    every = np.arange(1 << n, dtype=np.uint64)
    kw = dict(full_decomposition=full)
    want = sv.sv_branch_amplitudes(lat, half_a, every, **kw)  # 2^n bitstrings: two halves
    assert abs(np.sum(np.abs(want) ** 2) - 1) < 1e-5
    for some in (every[:1], every[5:12], every[::max(1, (1 << n) // 9)], every[-3:]):
        got = sv.sv_branch_amplitudes(lat, half_a, some, **kw)
        assert np.array_equal(got, want[some.astype(np.int64)])
