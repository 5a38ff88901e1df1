"""Calls of the library's internal host functions, for tests that need no GPU: a
small C++ program, compiled against the library's own header and linked with
libwtheta.so, prints what they return."""
import os
import subprocess

PKG = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_1208_3658_gb300")


def run(tmp_path, body, args=()):
    """Compiles main(argc, argv) with the given body and returns its output's
    lines, split into words."""
    from paper_1208_3658_gb300 import build
    lib = build.build()
    src, exe = str(tmp_path / "calls.cpp"), str(tmp_path / "calls")
    with open(src, "w") as f:
        f.write('#include <cstdio>\n#include <cstdlib>\n#include <vector>\n'
                '#include "wtheta_internal.h"\nusing namespace wtheta;\n'
                "int main(int argc, char** argv) {\n" + body + "\nreturn 0; }\n")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    cmd = ["g++", "-std=c++17", "-I" + os.path.join(cuda, "include"), "-I" + build.CSRC,
           "-I" + build.INCLUDE, src, "-o", exe, lib, "-Wl,-rpath," + os.path.dirname(lib)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([exe] + [str(a) for a in args], capture_output=True, text=True)
    assert out.returncode == 0, out.stderr
    return [line.split() for line in out.stdout.splitlines()]
