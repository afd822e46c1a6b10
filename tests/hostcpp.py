"""Compiles a C++ snippet against the library's internal headers and runs it on the CPU."""
import os
import subprocess

from paper_2306_16493_gb300 import build


def run(tmp_path, source, stdin=""):
    """The standard output of `source`, a translation unit with a main(), given `stdin`."""
    src, exe = os.path.join(str(tmp_path), "t.cu"), os.path.join(str(tmp_path), "t")
    with open(src, "w") as f:
        f.write(source)
    r = subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-I" + os.path.join(build.ROOT, "include"),
                        "-I" + build.CSRC, src, "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], input=stdin, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return r.stdout
