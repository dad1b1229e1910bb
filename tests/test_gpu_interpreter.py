"""The interpreting tile kernels on the sizes where their shapes change: every register width
(2 slots up to 11 and at 13..15 qubits, else 4; stage widths 1..4), tiles of 6 to 13 qubits,
one tile and many, passes whose program stays in shared memory and passes whose program
does not (long gate lists), from |0..0> and from a loaded state, with projectors."""
import numpy as np
import pytest

from oracle import circuit as oc
from oracle import statevec as ov
from paper_1804_04797_gb300 import sv

pytestmark = pytest.mark.gpu

CODE = dict(oc.KIND_CODE, P0=5, P1=6, Z=7, TDG=8, SXDG=9, SYDG=10)
KINDS = ['H', 'T', 'SX', 'SY', 'CZ', 'CZ', 'Z', 'TDG', 'SXDG', 'SYDG']


def gate_list(n, count, seed, projectors):
    rng = np.random.default_rng(seed)
    out = []
    for i in range(count):
        k = ('P0', 'P1')[i & 1] if projectors and i % 40 == 17 else KINDS[rng.integers(len(KINDS))]
        a = int(rng.integers(n))
        out.append((k, a, (a + 1 + int(rng.integers(n - 1))) % n if k == 'CZ' else 0))
    return out


def apply(n, gates, psi):
    psi = np.array(psi, dtype=np.complex128)
    for k, a, b in gates:
        if k == 'CZ':
            ov.apply_cz(psi, a, b)
        elif k in ('P0', 'P1'):
            psi.reshape(-1, 2, 1 << a)[:, 1 if k == 'P0' else 0] = 0
        elif k == 'Z':
            psi.reshape(-1, 2, 1 << a)[:, 1] *= -1
        else:
            m = ov.gate_matrix(k[:-2]).conj().T if k.endswith('DG') else ov.gate_matrix(k)
            ov.apply_1q(psi, m, a)
    return psi


@pytest.mark.parametrize('n,count,kw', [
    (6, 90, {}), (7, 90, {}), (11, 150, {}), (12, 150, {}), (13, 150, {}), (15, 150, {}), (16, 150, {}),
    (19, 150, {}), (20, 150, {}), (10, 120, dict(tile_bits=6, low_bits=3)), (14, 120, dict(tile_bits=7, low_bits=2)),
    (13, 120, dict(tile_bits=13)), (15, 120, dict(tile_bits=10, low_bits=4, fuse_k=1)),
    (15, 120, dict(tile_bits=9, low_bits=5, fuse_k=2)), (14, 120, dict(tile_bits=12, low_bits=2, fuse_k=4)),
    (6, 2500, {}), (12, 2500, {}), (14, 2500, dict(tile_bits=8, low_bits=4))])
def test_random_gates_match_the_oracle(n, count, kw):
    # three fp32 roundings of an amplitude a gate at most, each 2^-24 relative
    tol = 3 * count * 2.0 ** -24
    rng = np.random.default_rng(n)
    start = (rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)).astype(np.complex64)
    start /= np.linalg.norm(start)
    for loaded in (False, True):
        # (projectors on a loaded state: on |0..0> they may leave nothing)
        gates = gate_list(n, count, 7 * n + loaded, projectors=loaded and count < 200)
        want = apply(n, gates, start if loaded else ov.zero_state(n))
        h = sv.sv_create(n, sv.options(jit=-1, **kw))
        try:
            if loaded:
                sv.sv_load_state(h, start)
            sv.sv_apply_circuit(h, sv.gates_from_tuples([(CODE[k], a, b, 1) for k, a, b in gates]))
            got = sv.sv_copy_state(h, n).astype(np.complex128)
        finally:
            sv.sv_destroy(h)
        assert np.linalg.norm(got - want) <= tol * max(np.linalg.norm(want), 1e-3)
