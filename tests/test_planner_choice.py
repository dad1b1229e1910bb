"""The planner's greedy choices -- a pass's tile qubits, a stage's register qubits -- follow all
candidates of a round together; here each candidate is tried by itself, and the execution order
and the tiles have to be the same."""
import numpy as np
import pytest

from oracle import circuit as oc
from paper_1804_04797_gb300 import sv

DIAG = {oc.KIND_CODE[k] for k in ('T', 'CZ', 'Z')}
CZ = oc.KIND_CODE['CZ']


def _qubits(g):
    return (g[1], g[2]) if g[0] == CZ else (g[1],)


def _walk(gates, rem, fits):
    """The gates of rem that run before a gate that does not fit blocks them, in order."""
    waits, waits_nd, taken = set(), set(), []
    for i in rem:
        qs, diag = _qubits(gates[i]), gates[i][0] in DIAG
        if not (waits_nd if diag else waits) & set(qs) and (diag or fits(qs[0])):
            taken.append(i)
        else:
            waits |= set(qs)
            if not diag:
                waits_nd |= set(qs)
    return taken


def _score(gates, taken):
    return sum(gates[i][0] not in DIAG for i in taken), len(taken)


def _plan(n, gates, m, c, r):
    order, tiles, rem = [], [], list(range(len(gates)))
    while rem:
        tile = set(range(min(c, n)))
        first = {}
        for k, i in enumerate(rem):
            if gates[i][0] not in DIAG:
                first.setdefault(gates[i][1], k)
        while len(tile) < min(m, n):
            best = max((q for q in range(n) if q not in tile),
                       key=lambda q: (_score(gates, _walk(gates, rem, lambda x: x in tile or x == q)),
                                      -first.get(q, 1 << 19), -q))
            tile.add(best)
        left = _walk(gates, rem, lambda x: x in tile)
        rem = [i for i in rem if i not in set(left)]
        while left:
            regs = {0}
            cur = _score(gates, _walk(gates, left, lambda x: x in regs))
            for _ in range(r):
                best = None
                for q in sorted(tile - regs):
                    sc = _score(gates, _walk(gates, left, lambda x: x in regs or x == q))
                    if sc > cur:
                        cur, best = sc, q
                if best is None:
                    break
                regs.add(best)
            now = _walk(gates, left, lambda x: x in regs)
            order += now
            left = [i for i in left if i not in set(now)]
        tiles.append(tile)
    return order, tiles


def _random_gates(n, count, seed):
    rng = np.random.default_rng(seed)
    out = []
    for layer in range(count):
        k = ['H', 'T', 'SX', 'SY', 'CZ', 'Z', 'CZ'][rng.integers(7)]
        a = int(rng.integers(n))
        b = int((a + 1 + rng.integers(n - 1)) % n)
        out.append((oc.KIND_CODE[k], a, b if k == 'CZ' else 0, layer))
    return out


@pytest.mark.parametrize('n,gates,m', [
    (13, _random_gates(13, 1, 0), 12),
    (13, _random_gates(13, 7, 1), 10),
    (14, _random_gates(14, 8, 2), 10),       # one full group of counted masks
    (18, _random_gates(18, 9, 3), 13),
    (16, _random_gates(16, 600, 4), 12),
    (34, _random_gates(34, 300, 5), 13),
    (12, _random_gates(12, 150, 6), 12),     # one tile
    (28, oc.to_codes(oc.generate(4, 7, 0, 16, 3)[1]), 12),
])
def test_candidates_followed_together_choose_as_one_by_one(n, gates, m):
    opts = sv.options(jit=1, pipeline=-1, tile_bits=m, fuse_k=4)
    summ, order, pass_of, tiles = sv.sv_plan(n, sv.gates_from_tuples(gates), opts, fresh_state=False)
    want, sets = _plan(n, gates, m, 4, 4)
    assert order.tolist() == want
    assert [set(t[t >= 0].tolist()) for t in tiles] == sets
