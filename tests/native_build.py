"""Small shared libraries built by the tests out of the library's internal
headers and object files, for rules and kernels that no entry point shows."""
import ctypes
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def load(name: str, out_dir, objects: bool = False) -> ctypes.CDLL:
    """tests/native/<name>.cu as a shared library (objects: linked with the
    library's own object files)."""
    from paper_1901_10475_gb300 import build as b
    b.build()
    out = os.path.join(str(out_dir), f"lib{name}.so")
    objs = []
    if objects:
        d = os.path.join(b.OUT_DIR, "obj")
        objs = [os.path.join(d, os.path.basename(s)[:-3] + ".o") for s in b.sources()]
        if not all(os.path.exists(o) for o in objs):
            b.build(force=True)
    cmd = [b.nvcc(), *b.ARCH, "-O1", "-std=c++17", "-Xcompiler", "-fPIC",
           "--expt-relaxed-constexpr", "-I", b.CSRC, "-shared",
           os.path.join(HERE, "native", name + ".cu"), *objs, "-o", out]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return ctypes.CDLL(out)
