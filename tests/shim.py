"""Runs a Python program in a child process with tests/cuda_shim.c preloaded."""
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def build(tmp):
    so = os.path.join(str(tmp), "cuda_shim.so")
    subprocess.check_call(["gcc", "-O1", "-shared", "-fPIC", "-o", so, os.path.join(HERE, "cuda_shim.c"),
                           "-ldl", "-lpthread"])
    return so


def run(so, program, timeout=300, **env):
    """The program's standard output; it finds the shim's own calls in `shim`."""
    head = f"import ctypes, sys\nsys.path.insert(0, {ROOT!r})\nshim = ctypes.CDLL({so!r})\n"
    head += ("shim.shim_set_budget.argtypes = [ctypes.c_longlong]\n"
             "shim.shim_used.restype = shim.shim_refused.restype = ctypes.c_longlong\n")
    p = subprocess.run([sys.executable, "-c", head + program], cwd=ROOT, capture_output=True, text=True,
                       timeout=timeout, env=dict(os.environ, LD_PRELOAD=so, **{k: str(v) for k, v in env.items()}))
    assert p.returncode == 0, p.stdout[-2000:] + p.stderr[-4000:]
    return p.stdout
