"""Kernels compiled at run time are kept on disk; those of a library whose device headers have changed
since are not taken for the new ones."""
import os

import host_cpp
from paper_1804_04797_gb300 import build


def test_a_changed_header_is_another_kernel(tmp_path):
    text = build._jit_headers_source()
    cache = tmp_path / 'cache'
    cache.mkdir()
    more = ['-L', os.path.join(host_cpp.CUDA, 'lib64'), '-lcudart_static', '-lrt']
    exes = []
    for name, headers in (('before', text), ('after', text.replace(')svjit"', '\n// changed\n)svjit"'))):
        here = tmp_path / name
        here.mkdir()
        (here / 'headers.cpp').write_text(headers)
        exes.append(host_cpp.build(here, 'kernel_cache', ['jit.cpp', 'plan.cpp'], [str(here / 'headers.cpp')] + more))
    kept = []
    for exe in (exes[0], exes[1], exes[0]):
        r = host_cpp.run(exe, cache)
        assert r.returncode == 0, r.stdout + r.stderr
        kept.append(len(os.listdir(cache)))
    assert kept == [1, 2, 2]
