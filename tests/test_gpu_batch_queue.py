"""Large batches take their tiles in runs, and amplitudes come back in groups: the values of a
circuit in any batch, and of an amplitude in any request, are bit for bit those of it alone."""
import numpy as np
import pytest

from paper_1804_04797_gb300 import inputs, sv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize('sizes', [(22,) * 14 + (13, 10, 17), (18,) * 40 + (22,) * 20 + (11, 19), (22,) * 76 + (12, 16, 10)],
                         ids=['runs of 2', 'runs of 4', 'runs of 16'])
def test_runs_of_tiles_change_no_value(sizes):
    opts = sv.options(jit=-1, tile_bits=10)
    lats = [inputs.batch_lattice(n, 6 + i % 5, 70 + i) for i, n in enumerate(sizes)]
    try:
        stats = sv.sv_apply_batch(lats, opts)
        picks = list(range(0, len(sizes), max(1, len(sizes) // 6))) + [len(sizes) - 2, len(sizes) - 1]
        bits = {i: inputs.bitstrings(sizes[i], 300, seed=i) for i in picks}
        amps = {i: sv.sv_batch_amplitudes(i, bits[i]) for i in picks}
        for i in picks:
            alone = sv.sv_apply_batch([lats[i]], opts)
            assert np.array_equal(alone[0], stats[i])
            assert np.array_equal(sv.sv_batch_amplitudes(0, bits[i]), amps[i])
    finally:
        sv.sv_batch_free()


def test_amplitudes_do_not_depend_on_the_request():
    lat = inputs.batch_lattice(12, 9, 3)
    try:
        sv.sv_apply_batch([inputs.batch_lattice(10, 5, 1), lat])
        bits = np.array(inputs.bitstrings(12, 600, seed=5), np.uint64)
        one = np.concatenate([sv.sv_batch_amplitudes(1, bits[i:i + 1]) for i in range(600)])
        for m in (0, 2, 31, 33, 255, 256, 257, 512, 600):
            assert np.array_equal(sv.sv_batch_amplitudes(1, bits[:m]), one[:m])
        with pytest.raises(sv.SvError):
            sv.sv_batch_amplitudes(1, [0, 1 << 12])
    finally:
        sv.sv_batch_free()
