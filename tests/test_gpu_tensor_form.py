"""The tensor form's products at the edges of their tiles: halves smaller than a tile's rows or
columns, halves of exactly one tile, few and many branches (a step's remainder), and absorbed
CZs, whose signs the product applies."""
import numpy as np
import pytest

from oracle import circuit as oc
from oracle import csim
from paper_1804_04797_gb300 import inputs, sv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize('precision', [sv.SV_PREC_PLAIN, sv.SV_PREC_TF32X3], ids=['cuda_cores', 'tensor_cores'])
@pytest.mark.parametrize('rows,cols,cut,depth', [(2, 3, 1, 6), (3, 4, 1, 6), (3, 4, 2, 8), (2, 7, 1, 6), (2, 7, 1, 10),
                                                 (3, 7, 2, 8), (2, 9, 1, 6)])
def test_small_halves_and_signs_match_the_oracle(rows, cols, cut, depth, precision):
    lat = inputs.lattice_for(rows, cols, depth, seed=3)
    half_a = (1 << (cut * cols)) - 1
    assert sv.sv_branch_counts(lat, half_a)[1] > 0  # signs
    n, gates = oc.generate(lat.rows, lat.cols, lat.removed_mask, lat.depth, lat.seed)
    want = csim.run(n, gates)
    h = sv.sv_create(n)
    try:
        sv.sv_branch_full_state(lat, half_a, h, sv.options(precision=precision))
        got = sv.sv_copy_state(h, n).astype(np.complex128)
    finally:
        sv.sv_destroy(h)
    assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)
