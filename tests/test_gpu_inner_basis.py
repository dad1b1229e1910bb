"""Backward states from basis states on plan kernels that skip what is still zero: states of one
tile and of many, supports that reach every qubit in the last pass or before it, tile sizes of
the pipelined kernels, bitstrings with every and no bit set."""
import numpy as np
import pytest

from oracle import circuit as oc
from oracle import csim
from paper_1804_04797_gb300 import inputs, sv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize('rows,cols,depth,split,tile_bits', [
    (3, 4, 14, 6, 0), (3, 4, 14, 6, 10), (1, 13, 18, 5, 12), (3, 5, 14, 2, 11), (4, 4, 16, 8, 13), (4, 5, 16, 3, 10),
    (4, 5, 16, 8, 0), (4, 5, 16, 14, 0), (3, 7, 15, 7, 12)])
def test_amplitudes_match_the_oracle(rows, cols, depth, split, tile_bits):
    lat = inputs.lattice_for(rows, cols, depth, seed=11)
    n, gates = oc.generate(lat.rows, lat.cols, lat.removed_mask, lat.depth, lat.seed)
    want = csim.run(n, gates)
    bits = [0, (1 << n) - 1] + inputs.bitstrings(n, 14, seed=5)
    got = sv.sv_amplitudes_by_inner_product(lat, split, bits, sv.options(jit=1, tile_bits=tile_bits))
    sel = want[np.array(bits, dtype=np.int64)]
    assert np.linalg.norm(sel) > 0
    assert np.linalg.norm(got - sel) <= 1e-5 * np.linalg.norm(sel)
