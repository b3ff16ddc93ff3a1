"""Small C++ programs against the library's internal header (its host-callable rules), built with the
host compiler.  For CPU tests of rules that no entry point shows: addresses, plans, states."""
import os
import shutil
import subprocess

from paper_2009_09501_gb300 import build as B


def build(folder, body):
    """Compiles `body` and returns a function that runs it with some arguments and returns what it printed."""
    src, exe = folder / "probe.cpp", folder / "probe"
    src.write_text(body)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc())))
    cmd = [shutil.which("g++") or "c++", "-std=c++17", "-O1", "-I" + B.INCLUDE, "-I" + B.CSRC,
           "-I" + os.path.join(cuda, "include"), str(src), "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]

    def run(*args):
        r = subprocess.run([str(exe)] + [str(a) for a in args], capture_output=True, text=True, timeout=120)
        assert r.returncode == 0, (args, r.returncode, r.stdout[-2000:], r.stderr[-2000:])
        return r.stdout

    return run
