"""The simulator's measured work: what a user has it do, from the smallest calls to the largest.

Every case goes through the public binding (paper_1804_04797_gb300.sv).  The seed picks the
circuit (the generator's one-qubit gates), the loaded amplitudes and the bitstrings.
Lattices are rows x cols with the last `drop` sites left out.  Kinds:

  apply   one circuit on a caller's device buffer (sv_create_from_ptr): from |0..0>
          (loaded = 0) or on the amplitudes the buffer holds (loaded = 1: every pass evolves
          them further); returns the state.  precision: plain fp32, or the tensor cores
          with F16x3 or TF32x3 products.
  report  one circuit from |0..0> on a state the library owns, then its norm and sum p^2
          and a copy of the amplitudes into the caller's buffer.
  batch   many uneven circuits in one call (4-row lattices of n_min..n_max qubits, depths
          10..24), their statistics, and two amplitudes of each circuit.
  branch  amplitudes of a circuit too large to store, by cutting its lattice between rows.
  inner   amplitudes by the inner product of a forward and a backward state.
  full    the full state from the two halves of a cut lattice (tensor form).
"""
import math

import numpy as np
import torch

from paper_1804_04797_gb300 import inputs, sv

_PRECISION = {'plain': sv.SV_PREC_PLAIN, 'f16x3': sv.SV_PREC_F16X3, 'tf32x3': sv.SV_PREC_TF32X3}


def listed():
    return [
        # a circuit of a parameter sweep or a test: all latency and launches
        _apply('apply 12q', 3, 4, 0, 16),
        # the 4x4 depth-10 circuit of the parity tests, from |0..0>
        _apply('apply 16q', 4, 4, 0, 10),
        # a prepared state evolved in place
        _apply('apply 20q loaded', 4, 5, 0, 14, loaded=1),
        # an odd lattice just below the size from which plans are compiled
        _apply('apply 23q', 4, 6, 1, 20),
        # compiled plan, the statistics of the run (Porter-Thomas) and the amplitudes out
        dict(name='report 27q', kind='report', rows=4, cols=7, drop=1, depth=16),
        # the 5x6 depth-20 circuit: the largest full state that fits the card three times over
        # with room for its 64-bit check
        _apply('apply 30q', 5, 6, 0, 20),
        # tensor-core products, both formats
        _apply('apply 28q f16x3', 4, 7, 0, 20, precision='f16x3'),
        _apply('apply 25q tf32x3 loaded', 5, 5, 0, 12, loaded=1, precision='tf32x3'),
        # a batch of uneven circuits, each list new to the library
        dict(name='batch 64', kind='batch', count=64, n_min=10, n_max=22),
        # the amplitude task: 6x7 depth 10 cut between rows 2 and 3, 64 bitstrings
        dict(name='branch 42q', kind='branch', rows=6, cols=7, drop=0, depth=10, cut=3, m=64, precision='plain'),
        # the amplitude task by inner products: 4x7 depth 16, the forward and the backward
        # state half the layers each
        dict(name='inner 28q', kind='inner', rows=4, cols=7, drop=0, depth=16, split=8, m=4),
        # the tensor form: 4x7 depth 10 cut between rows 1 and 2
        dict(name='full 28q', kind='full', rows=4, cols=7, drop=0, depth=10, cut=2, precision='plain'),
    ]


def _apply(name, rows, cols, drop, depth, loaded=0, precision='plain'):
    return dict(name=name, kind='apply', rows=rows, cols=cols, drop=drop, depth=depth, loaded=loaded, precision=precision)


def draw(rng):
    kind = rng.choice(['apply', 'apply', 'apply', 'report', 'batch', 'branch', 'inner', 'full'])
    if kind in ('apply', 'report'):
        precision = rng.choice(['plain', 'plain', 'plain', 'f16x3', 'tf32x3']) if kind == 'apply' else 'plain'
        n = rng.randint(8, 29) if precision == 'plain' else rng.randint(14, 27)
        rows, cols, drop = _shape(rng, n)
        case = dict(kind=kind, rows=rows, cols=cols, drop=drop, depth=rng.randint(6, 24 if n < 28 else 14))
        if kind == 'apply':
            case.update(loaded=rng.randint(0, 1), precision=precision)
        return case
    if kind == 'batch':
        n_min = rng.randint(8, 14)
        return dict(kind='batch', count=rng.randint(8, 96), n_min=n_min, n_max=n_min + rng.randint(2, 8))
    precision = rng.choice(['plain', 'f16x3', 'tf32x3'])
    if kind == 'branch':
        rows, cols = rng.choice([(4, 5), (4, 6), (4, 7), (5, 6), (6, 5), (6, 6), (6, 7)])
        return dict(kind='branch', rows=rows, cols=cols, drop=rng.randint(0, 2), depth=rng.randint(6, 10),
                    cut=rows // 2, m=rng.randint(1, 200), precision=precision)
    if kind == 'inner':
        rows, cols, drop = _shape(rng, rng.randint(14, 28))
        depth = rng.randint(10, 16)
        return dict(kind='inner', rows=rows, cols=cols, drop=drop, depth=depth, split=rng.randint(3, depth - 2),
                    m=rng.randint(1, 4))
    rows, cols = rng.choice([(4, 4), (4, 5), (4, 6), (4, 7), (5, 5)])
    return dict(kind='full', rows=rows, cols=cols, drop=rng.randint(0, 1), depth=rng.randint(6, 10), cut=rows // 2,
                precision=precision)


def _shape(rng, n):
    rows = rng.choice([r for r in (2, 3, 4, 5) if -(-n // r) * r - n < -(-n // r)])
    cols = -(-n // rows)
    return rows, cols, rows * cols - n


# ---- what a user's program holds, and its call -------------------------------------------

class _State:
    """A handle and the buffers that go with it; the handle goes when the state does."""

    def __init__(self, handle=None, **held):
        self.handle = handle
        self.__dict__.update(held)

    def __del__(self):
        if self.handle is not None:
            sv.sv_destroy(self.handle)
            self.handle = None


def _lattice(case, seed):
    sites = case['rows'] * case['cols']
    mask = ((1 << case['drop']) - 1) << (sites - case['drop'])
    return inputs.Lattice(case['rows'], case['cols'], mask, case['depth'], seed)


def prepare(case, seed):
    kind = case['kind']
    if kind == 'batch':
        lats = inputs.batch(case['count'], seed, case['n_min'], case['n_max'])
        bits = [np.array(inputs.bitstrings(l.n_qubits, 2, seed + i), np.uint64) for i, l in enumerate(lats)]
        return _State(kind=kind, lats=[sv.lattice(l) for l in lats], bits=bits)
    lat = _lattice(case, seed)
    n = lat.n_qubits
    if kind == 'apply':
        if case['loaded']:
            psi = _amplitudes(n, seed)
        else:
            psi = torch.empty(1 << n, dtype=torch.complex64, device='cuda')
        h = sv.sv_create_from_ptr(n, psi.data_ptr())
        sv.sv_set_options(h, sv.options(precision=_PRECISION[case['precision']]))
        return _State(h, kind=kind, psi=psi, loaded=case['loaded'], gates=sv.sv_generate_circuit(lat))
    if kind == 'report':
        psi = torch.empty(1 << n, dtype=torch.complex64, device='cuda')
        return _State(sv.sv_create(n), kind=kind, n=n, psi=psi, gates=sv.sv_generate_circuit(lat))
    opts = sv.options(precision=_PRECISION[case.get('precision', 'plain')])
    if kind == 'full':
        psi = torch.empty(1 << n, dtype=torch.complex64, device='cuda')
        h = sv.sv_create_from_ptr(n, psi.data_ptr())
        return _State(h, kind=kind, psi=psi, lat=lat, opts=opts, half_a=(1 << (case['cut'] * case['cols'])) - 1)
    bits = np.array(inputs.bitstrings(n, case['m'], seed), np.uint64)
    if kind == 'branch':
        return _State(kind=kind, lat=lat, bits=bits, opts=opts, half_a=(1 << (case['cut'] * case['cols'])) - 1)
    return _State(kind=kind, lat=lat, bits=bits, split=case['split'])


def run(state):
    if state.kind == 'apply':
        if not state.loaded:
            sv.sv_reset(state.handle)
        sv.sv_apply_circuit(state.handle, state.gates)
        return state.psi
    if state.kind == 'report':
        sv.sv_reset(state.handle)
        sv.sv_apply_circuit(state.handle, state.gates)
        norm2, sum_p2 = sv.sv_norm(state.handle)
        sv.sv_copy_state(state.handle, state.n, state.psi.data_ptr())
        return {'state': state.psi, 'norm2': norm2, 'sum_p2': sum_p2}
    if state.kind == 'batch':
        stats = sv.sv_apply_batch(state.lats)
        return {'stats': stats, 'amplitudes': np.concatenate([sv.sv_batch_amplitudes(i, b)
                                                              for i, b in enumerate(state.bits)])}
    if state.kind == 'branch':
        return sv.sv_branch_amplitudes(state.lat, state.half_a, state.bits, state.opts)
    if state.kind == 'inner':
        return sv.sv_amplitudes_by_inner_product(state.lat, state.split, state.bits)
    sv.sv_branch_full_state(state.lat, state.half_a, state.handle, state.opts)
    return state.psi


# ---- what a pass cannot do without ----------------------------------------------------------

_FLOPS = {'H': 4, 'SX': 2, 'SY': 2, 'T': 2, 'CZ': 0}  # real operations per amplitude


def _flops(gates):
    return sum(_FLOPS[k] for k, _, _, layer in gates if layer > 0)


def work(case):
    kind = case['kind']
    if kind == 'batch':
        lats = inputs.batch(case['count'], 0, case['n_min'], case['n_max'])
        return {'bytes': sum(8 << l.n_qubits for l in lats) + 56 * len(lats),
                'flops': sum(_flops(_circuit(l)) << l.n_qubits for l in lats)}
    lat = _lattice(case, 0)
    n, gates = lat.n_qubits, _circuit(lat)
    if kind in ('apply', 'report', 'full'):
        states = 2 if case.get('loaded') or kind == 'report' else 1
        if kind == 'full':  # one complex product per amplitude and branch, and the write
            _, _, summed = _branch_bits(case, gates, implicit=False)
            return {'bytes': 8 << n, 'flops': 8 << (n + summed)}
        return {'bytes': 8 * states << n, 'flops': _flops(gates) << n}
    if kind == 'inner':  # the forward state written, read for each bitstring; the gates on both
        back = [g for g in gates if g[3] > case['split']]
        forth = [g for g in gates if g[3] <= case['split']]
        return {'bytes': (8 << n) * (1 + case['m']), 'flops': (_flops(forth) + case['m'] * _flops(back)) << n}
    # both halves over their branches, each written once
    na = case['cut'] * case['cols']
    bits_a, bits_b, _ = _branch_bits(case, gates, implicit=True)
    return {'bytes': (8 << (na + bits_a)) + (8 << (n - na + bits_b)) + 24 * case['m'],
            'flops': (_flops([g for g in gates if g[1] < na]) << (na + bits_a)) +
                     (_flops([g for g in gates if g[1] >= na]) << (n - na + bits_b))}


def _branch_bits(case, gates, implicit):
    """Branch bits of the two halves and the summed ones: a crossing CZ after which no gate
    other than a diagonal one meets a qubit needs none for the half that holds it."""
    na = case['cut'] * case['cols']
    last = {a: i for i, (k, a, _, _) in enumerate(gates) if k in ('H', 'SX', 'SY')}
    in_a = in_b = both = 0
    for i, (k, a, b, _) in enumerate(gates):
        if k == 'CZ' and (a < na) != (b < na):
            qa, qb = (a, b) if a < na else (b, a)
            quiet_a, quiet_b = last[qa] < i, last[qb] < i
            if quiet_a and quiet_b:
                continue
            if not implicit or not (quiet_a or quiet_b):
                both += 1
            elif quiet_a:
                in_b += 1
            else:
                in_a += 1
    return in_a + both, in_b + both, both


# ---- the same results in 64 bits, in plain torch ---------------------------------------------

def _splitmix(seed):
    m64 = (1 << 64) - 1
    s = seed & m64
    while True:
        s = (s + 0x9E3779B97F4A7C15) & m64
        z = s
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & m64
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m64
        yield z ^ (z >> 31)


def _circuit(lat):
    """[(kind, q0, q1, layer)] of a lattice: H on every qubit, then per layer the one-qubit
    gates of the qubits a CZ has just left and the layer's pattern of neighbouring CZs."""
    number = {}
    for r in range(lat.rows):
        for c in range(lat.cols):
            if not (lat.removed_mask >> (r * lat.cols + c)) & 1:
                number[r, c] = len(number)
    n = len(number)
    gates = [('H', q, q, 0) for q in range(n)]
    rng, before, previous = _splitmix(lat.seed), set(), {}
    for layer in range(1, lat.depth + 1):
        vertical, shift = (layer - 1) % 2, ((layer - 1) % 8) // 2
        bonds = []
        for (r, c), q in number.items():
            other = number.get((r + 1, c) if vertical else (r, c + 1))
            where = (r + 2 * (c % 2)) if vertical else (c + 2 * (r % 2))
            if other is not None and where % 4 == shift:
                bonds.append((min(q, other), max(q, other)))
        now = {q for b in bonds for q in b}
        for q in sorted(before - now):
            choice = [k for k in ('T', 'SX', 'SY') if k != previous.get(q)]
            previous[q] = choice[next(rng) % len(choice)]
            gates.append((previous[q], q, q, layer))
        gates += [('CZ', a, b, layer) for a, b in sorted(bonds)]
        before = now
    return gates


_R = math.sqrt(0.5)
_MATRIX = {'H': ((_R, _R), (_R, -_R)),
           'SX': (((1 + 1j) / 2, (1 - 1j) / 2), ((1 - 1j) / 2, (1 + 1j) / 2)),
           'SY': (((1 + 1j) / 2, (-1 - 1j) / 2), ((1 + 1j) / 2, (1 + 1j) / 2))}


def _evolve(psi, gates):
    """gates on psi[..., 2^n] (complex128), in place."""
    for k, a, b, _ in gates:
        v = psi.view(-1, 2, 1 << a)
        if k == 'T':
            v[:, 1].mul_(complex(_R, _R))
        elif k == 'CZ':
            psi.view(-1, 2, 1 << (b - a - 1), 2, 1 << a)[:, 1, :, 1].neg_()
        else:
            (m00, m01), (m10, m11) = _MATRIX[k]
            x, y = v[:, 0], v[:, 1]
            z = x * m10
            z.add_(y, alpha=m11)
            x.mul_(m00).add_(y, alpha=m01)
            y.copy_(z)
    return psi


def _device():
    return 'cuda' if torch.cuda.is_available() else 'cpu'


def _amplitudes(n, seed):
    g = torch.Generator(_device()).manual_seed(seed)
    psi = torch.randn(1 << n, 2, generator=g, device=_device())
    psi.mul_(1.0 / math.sqrt(2.0 * 2.0 ** n))  # norm 1 on the whole, to its spread
    return torch.view_as_complex(psi)


def _final(lat, psi=None):
    n, gates = lat.n_qubits, _circuit(lat)
    if psi is None:  # the H layer on |0..0>
        psi = torch.full((1 << n,), 2.0 ** (-0.5 * n), dtype=torch.complex128, device=_device())
        gates = gates[n:]
    return _evolve(psi, gates)


def _sums(psi):
    p = torch.view_as_real(psi).square().sum(-1)
    return float(p.sum()), float(p.square().sum())


def exact(case, seed):
    kind = case['kind']
    if kind == 'batch':
        lats = inputs.batch(case['count'], seed, case['n_min'], case['n_max'])
        stats, amplitudes = [], []
        for i, lat in enumerate(lats):
            psi = _final(lat)
            stats.append((*_sums(psi), float(lat.n_qubits)))
            amplitudes.append(_pick(psi, inputs.bitstrings(lat.n_qubits, 2, seed + i)))
        return {'stats': np.array(stats), 'amplitudes': np.concatenate(amplitudes)}
    lat = _lattice(case, seed)
    n = lat.n_qubits
    if kind == 'branch':
        return _cut_amplitudes(lat, case['cut'] * case['cols'], inputs.bitstrings(n, case['m'], seed))
    psi = _final(lat, _amplitudes(n, seed).to(torch.complex128) if case.get('loaded') else None)
    if kind == 'inner':
        return _pick(psi, inputs.bitstrings(n, case['m'], seed))
    if kind == 'report':
        norm2, sum_p2 = _sums(psi)
        return {'state': psi, 'norm2': norm2, 'sum_p2': sum_p2}
    return psi


def _pick(psi, bits):
    return psi[torch.tensor(bits, device=psi.device)].cpu().numpy()


def _cut_amplitudes(lat, na, bits):
    """Sum over the branches of the CZs that cross the cut: |l><l| on the one half, Z^l on
    the other."""
    n, gates = lat.n_qubits, _circuit(lat)
    sides = [[], []]
    crossing = 0
    for g in gates:
        k, a, b, layer = g
        if layer == 0:
            continue
        if k == 'CZ' and a < na <= b:
            sides[0].append(('P', a, crossing, layer))
            sides[1].append(('Z', b - na, crossing, layer))
            crossing += 1
        else:
            s = int(a >= na)
            sides[s].append((k, a - s * na, b - s * na, layer))
    if crossing > 12:
        return None
    x = torch.tensor(bits, device=_device())
    index = (x & ((1 << na) - 1), x >> na)
    total = torch.zeros(len(bits), dtype=torch.complex128, device=_device())
    at_once = 1 << max(0, min(crossing, 27 - max(na, n - na)))
    for first in range(0, 1 << crossing, at_once):
        branch = torch.arange(first, first + at_once, device=_device())
        found = []
        for s, size in enumerate((na, n - na)):
            psi = torch.full((at_once, 1 << size), 2.0 ** (-0.5 * size), dtype=torch.complex128, device=_device())
            for g in sides[s]:
                if g[0] not in 'PZ':
                    _evolve(psi, [g])
                    continue
                bit = ((branch >> g[2]) & 1).to(torch.float64).view(-1, 1, 1)
                v = psi.view(at_once, -1, 2, 1 << g[1])
                if g[0] == 'P':
                    v[:, :, 0].mul_(1 - bit)
                    v[:, :, 1].mul_(bit)
                else:
                    v[:, :, 1].mul_(1 - 2 * bit)
            found.append(psi[:, index[s]])
        total += (found[0] * found[1]).sum(0)
    return total.cpu().numpy()
