"""Branch trees whose forks are read by the next segment's first pass: tiles of every pipelined
size, one and several branch bits a fork, halves of one slice and of many."""
import numpy as np
import pytest

from oracle import circuit as oc
from oracle import csim
from paper_1804_04797_gb300 import inputs, sv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize('rows,cols,depth,half_a,tile_bits', [
    (4, 5, 9, 0x3FF, 10), (4, 5, 9, 0x1F, 10), (5, 4, 10, 0xFFF, 11), (3, 7, 9, 0x3FFF, 12), (2, 9, 12, 0x1FF, 10),
    (4, 6, 8, 0xFFF, 0), (4, 5, 9, 0x7FFF, 13)])
@pytest.mark.parametrize('full', [False, True])
def test_amplitudes_match_the_oracle(rows, cols, depth, half_a, tile_bits, full):
    lat = inputs.lattice_for(rows, cols, depth, seed=31)
    n, gates = oc.generate(lat.rows, lat.cols, lat.removed_mask, lat.depth, lat.seed)
    want = csim.run(n, gates)
    bits = [0, (1 << n) - 1] + inputs.bitstrings(n, 30, seed=5)
    got = sv.sv_branch_amplitudes(lat, half_a, bits, sv.options(jit=1, tile_bits=tile_bits), full_decomposition=full)
    sel = want[np.array(bits, dtype=np.int64)]
    assert np.linalg.norm(sel) > 0
    assert np.linalg.norm(got - sel) <= 1e-5 * np.linalg.norm(sel)
