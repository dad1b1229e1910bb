"""Batches of circuits of every size the persistent launch takes in one CTA size (tiles of 10 to
12 qubits share 128 threads) and below it (smaller CTAs beside it), at every tile size."""
import numpy as np
import pytest

from oracle import circuit as oc
from oracle import csim
from paper_1804_04797_gb300 import inputs, sv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize('tile_bits', [0, 10, 11, 12, 13])
@pytest.mark.parametrize('sizes', [(14, 9, 13, 10, 11, 12, 17), (8, 9), (16, 13, 8, 12, 9, 10, 8, 11), (10,)],
                         ids=lambda s: '-'.join(map(str, s)))
def test_sizes_match_the_oracle(sizes, tile_bits):
    lats = [inputs.batch_lattice(n, 8 + i, 40 + i) for i, n in enumerate(sizes)]
    try:
        stats = sv.sv_apply_batch(lats, sv.options(tile_bits=tile_bits))
        for i, lat in enumerate(lats):
            n, gates = oc.generate(lat.rows, lat.cols, lat.removed_mask, lat.depth, lat.seed)
            want = csim.run(n, gates)
            bits = inputs.bitstrings(n, 32, seed=3)
            got = sv.sv_batch_amplitudes(i, bits)
            sel = want[np.array(bits, dtype=np.int64)]
            assert np.linalg.norm(got - sel) <= 1e-5 * max(np.linalg.norm(sel), 2.0 ** (-n / 2))
            assert stats[i][2] == n and abs(stats[i][0] - 1) <= 1e-6
        assert np.array_equal(stats, sv.sv_apply_batch(lats, sv.options(tile_bits=tile_bits)))
    finally:
        sv.sv_batch_free()
