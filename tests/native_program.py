"""Builds and runs a small C++/CUDA program against the library's own headers and
libsim.so, for parts that the C API does not reach by themselves."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def run(tmp_path, source, *args):
    """Compiles `source` (CUDA C++), runs it and returns what it printed."""
    from paper_2006_16117_gb300 import build as b

    b.build()
    lib = os.path.dirname(b.LIB)
    src, exe = os.path.join(str(tmp_path), "prog.cu"), os.path.join(str(tmp_path), "prog")
    with open(src, "w") as f:
        f.write(source)
    cmd = [b.nvcc(), *b.ARCH, *b.FLAGS, src, "-o", exe, "-L", lib, "-l:libsim.so", "-Xlinker", "-rpath," + lib,
           "-Xlinker", "-rpath,/usr/local/cuda/lib64"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([exe, *map(str, args)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout
