"""The programs of a batch's passes lie one after the other, and those of many deep circuits take
more than 4 GiB: 141208 circuits of 4x4 qubits and depth 200, with 74 GB of states, do."""
import pytest

import host_cpp


def test_programs_past_four_gib_keep_their_offsets(tmp_path):
    free = next(int(line.split()[1]) for line in open('/proc/meminfo') if line.startswith('MemAvailable'))
    if free < 6 << 20:
        pytest.skip('takes 4 GiB of host memory')
    r = host_cpp.run(host_cpp.build(tmp_path, 'interp_offsets', ['plan.cpp', 'interp.cpp']))
    assert r.returncode == 0, r.stdout
