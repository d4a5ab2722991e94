"""Compiles host code against the library's internal headers and runs it here, so
that rules of the launch code are checked without a GPU."""
import os
import subprocess
import textwrap

from paper_2303_17679_gb300 import build

PROLOGUE = """
#include <algorithm>
#include <cassert>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <thread>
#include <vector>
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\\n", __LINE__, #x); std::exit(1); } } while (0)
"""


def run(tmp_path, includes, body, link=()):
    """Compiles and runs `body` (with its main) after the headers in `includes`."""
    src, exe = tmp_path / "host.cu", tmp_path / "host"
    text = PROLOGUE + "".join(f'#include "{name}"\n' for name in includes)
    src.write_text(text + textwrap.dedent(body))
    r = subprocess.run([build.nvcc(), *build.ARCH, "-O1", "-std=c++17", "--expt-relaxed-constexpr",
                        "-I", build.CSRC, "-I", build.INCLUDE, str(src), *link, "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout
