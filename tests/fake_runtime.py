"""Builds tests/fake_cudart.c and runs a snippet with it preloaded."""
import os
import subprocess
import sys

from paper_1602_05806_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def run(code, folder, **env):
    """Output of `code` in a process of its own; the stand-in is at $FAKE."""
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc())))
    so = os.path.join(folder, "fake_cudart.so")
    libs = os.path.join(cuda, "lib64")
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-I", os.path.join(cuda, "include"), "-o", so,
                    os.path.join(HERE, "fake_cudart.c"), "-L", libs, "-Wl,--no-as-needed", "-lcudart", f"-Wl,-rpath,{libs}",
                    "-ldl"], check=True)
    r = subprocess.run([sys.executable, "-c", code], cwd=os.path.dirname(HERE), capture_output=True, text=True,
                       env=dict(os.environ, LD_PRELOAD=so, FAKE=so, **env), timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return r.stdout.split("\n")
