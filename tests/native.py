"""Builds and runs a small C++/CUDA program against the library's internal headers."""

import os
import subprocess

from paper_2606_04864_gb300 import _build


def build_native(tmp_path, source):
    """Compile `source` (the text of a .cu file) with the library's flags and link it to libams.so; the program's path."""
    lib = _build.build()
    src, exe = os.path.join(tmp_path, "main.cu"), os.path.join(tmp_path, "main")
    with open(src, "w") as f:
        f.write(source)
    d = os.path.dirname(lib)
    cmd = [_build._nvcc(), *_build.ARCH, *_build.FLAGS, "-I", _build.CSRC, src, "-o", exe, "-L", d, "-l:libams.so",
           "-Xlinker", "-rpath", "-Xlinker", d]
    p = subprocess.run(cmd, capture_output=True, text=True)
    assert p.returncode == 0, p.stdout + p.stderr
    return exe


def run_native(exe, *args):
    """Run the program and return what it printed, one line per list entry."""
    p = subprocess.run([exe, *map(str, args)], capture_output=True, text=True, timeout=120)
    assert p.returncode == 0, p.stdout + p.stderr
    return p.stdout.split("\n")[:-1]
