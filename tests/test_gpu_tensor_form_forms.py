"""The forms of the tensor-core product: every expanded CZ summed over (neither signs nor a scale with
a lo part), signs alone, and branches fixed by output bits, on halves of one tile and of several."""
import numpy as np
import pytest

from oracle import circuit as oc
from oracle import csim
from paper_1804_04797_gb300 import inputs, sv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize('rows,cols,cut,depth,whole', [
    (2, 7, 1, 10, True), (4, 4, 2, 8, True), (4, 5, 2, 9, True),
    (2, 7, 1, 6, False), (2, 7, 1, 10, False),
    (4, 5, 2, 7, False), (4, 5, 2, 8, False), (4, 6, 2, 9, False),
])
def test_each_form_matches_the_oracle(rows, cols, cut, depth, whole):
    lat = inputs.lattice_for(rows, cols, depth, seed=11)
    n, gates = oc.generate(lat.rows, lat.cols, lat.removed_mask, lat.depth, lat.seed)
    want = csim.run(n, gates)
    h = sv.sv_create(n)
    try:
        sv.sv_branch_full_state(lat, (1 << (cut * cols)) - 1, h, sv.options(precision=sv.SV_PREC_TF32X3),
                                full_decomposition=whole)
        got = sv.sv_copy_state(h, n).astype(np.complex128)
    finally:
        sv.sv_destroy(h)
    assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)
