"""Last passes on the tiles of the wanted amplitudes alone: one, few and every bitstring give the
same amplitudes bit for bit, with summed branch bits among the tile's qubits and outside them."""
import numpy as np
import pytest

from oracle import circuit as oc
from oracle import csim
from paper_1804_04797_gb300 import inputs, sv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize('rows,cols,depth,half_a,tile_bits', [
    (4, 5, 9, 0x3FF, 10), (4, 5, 9, 0xFFFF, 10), (3, 6, 9, 0x3FFFF >> 4, 11), (2, 9, 11, 0x1FF, 10), (3, 6, 9, 0x7, 12)])
@pytest.mark.parametrize('full', [False, True])
def test_few_bitstrings_match_every_bitstring(rows, cols, depth, half_a, tile_bits, full):
    lat = inputs.lattice_for(rows, cols, depth, seed=41)
    n = lat.n_qubits
    opts = sv.options(jit=1, tile_bits=tile_bits)
    every = np.arange(1 << n, dtype=np.uint64)
    want = sv.sv_branch_amplitudes(lat, half_a, every, opts, full_decomposition=full)
    assert abs(np.sum(np.abs(want) ** 2) - 1) < 1e-5
    for some in ([0], [(1 << n) - 1], inputs.bitstrings(n, 5, seed=2), inputs.bitstrings(n, 70, seed=3)):
        got = sv.sv_branch_amplitudes(lat, half_a, some, opts, full_decomposition=full)
        assert np.array_equal(got, want[np.array(some, dtype=np.int64)])


@pytest.mark.parametrize('precision', [sv.SV_PREC_PLAIN, sv.SV_PREC_TF32X3, sv.SV_PREC_F16X3])
@pytest.mark.parametrize('rows,cols,depth,half_a,full', [
    (4, 6, 8, 0xFFF, False), (4, 6, 7, 0xFFF, True), (4, 6, 9, 0x3FFFF, False), (3, 8, 9, 0xFFFF, False)])
def test_matrix_stages_fork_and_list_as_the_plain_passes(rows, cols, depth, half_a, full, precision):
    """Halves of 12-qubit tiles with branch bits above them, on each arithmetic: against the
    oracle, and one bitstring against many (whole last passes)."""
    lat = inputs.lattice_for(rows, cols, depth, seed=43)
    n, gates = oc.generate(lat.rows, lat.cols, lat.removed_mask, lat.depth, lat.seed)
    want = csim.run(n, gates)
    opts = sv.options(jit=1, precision=precision)
    many = inputs.bitstrings(n, 6000, seed=7)
    got = sv.sv_branch_amplitudes(lat, half_a, many, opts, full_decomposition=full)
    sel = want[np.array(many, dtype=np.int64)]
    assert np.linalg.norm(got - sel) <= 1e-5 * np.linalg.norm(sel)
    for a, b in ((0, 1), (5, 9), (4000, 4040)):
        assert np.array_equal(sv.sv_branch_amplitudes(lat, half_a, many[a:b], opts, full_decomposition=full), got[a:b])
