"""Small C++ programs that run the library's host code without a device."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, 'paper_1804_04797_gb300', 'csrc')
CUDA = os.environ.get('CUDA_HOME', '/usr/local/cuda')


def build(out_dir, program, sources, more=()):
    """tests/<program>.cpp with library sources, as an executable in out_dir (more: further files and
    flags)."""
    exe = os.path.join(str(out_dir), program)
    cmd = ['g++', '-std=c++17', '-O1', '-I', CSRC, '-I', os.path.join(CUDA, 'include'), '-o', exe,
           os.path.join(ROOT, 'tests', program + '.cpp')] + [os.path.join(CSRC, s) for s in sources] + list(more) + ['-ldl', '-lpthread']
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


def run(exe, *args, env=None):
    return subprocess.run([exe] + [str(a) for a in args], capture_output=True, text=True, timeout=300,
                          env=dict(os.environ, **(env or {})))
