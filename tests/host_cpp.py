"""Small C++ programs that run the library's host code without a device."""
import concurrent.futures as cf
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, 'paper_1804_04797_gb300', 'csrc')
CUDA = os.environ.get('CUDA_HOME', '/usr/local/cuda')


def build(out_dir, program, sources, more=()):
    """tests/<program>.cpp with library sources, as an executable in out_dir (more: further files and
    flags)."""
    exe = os.path.join(str(out_dir), program)
    files = [os.path.join(ROOT, 'tests', program + '.cpp')] + [os.path.join(CSRC, s) for s in sources]
    files += [f for f in more if f.endswith('.cpp')]
    flags = [f for f in more if not f.endswith('.cpp')]

    def one(f):
        obj = os.path.join(str(out_dir), os.path.basename(f) + '.o')
        _done(['g++', '-std=c++17', '-O1', '-I', CSRC, '-I', os.path.join(CUDA, 'include')] +
              [x for x in flags if x.startswith('-D')] + ['-c', f, '-o', obj])
        return obj

    with cf.ThreadPoolExecutor(len(files)) as pool:
        objs = list(pool.map(one, files))
    _done(['g++', '-o', exe] + objs + [x for x in flags if not x.startswith('-D')] + ['-ldl', '-lpthread'])
    return exe


def _done(cmd):
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr


def run(exe, *args, env=None):
    return subprocess.run([exe] + [str(a) for a in args], capture_output=True, text=True, timeout=300,
                          env=dict(os.environ, **(env or {})))
