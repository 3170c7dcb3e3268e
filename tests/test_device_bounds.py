"""The kernels' range tests (csrc/bounds.cuh), compiled as plain C++ and checked at
the edges of their ranges on the CPU."""
import os
import subprocess

import paper_2009_12457_gb300 as bb

CSRC = os.path.join(os.path.dirname(bb.__file__), "csrc")


def run(tmp_path, body):
    src = tmp_path / "bounds.cpp"
    src.write_text('#include <stdio.h>\n#include "bounds.cuh"\nusing namespace bbtc;\n'
                   "int main() {\n" + body + "\nreturn 0;\n}\n")
    exe = str(tmp_path / "bounds")
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-x", "c++", "-I", CSRC, str(src),
                    "-o", exe], check=True)
    return subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()


def test_span_inside(tmp_path):
    cases = [(0, 0, 0, 1), (0, 1, 0, 0), (0, 8, 8, 1), (1, 8, 8, 0), (8, 0, 8, 1), (9, 0, 8, 0),
             # a span that starts below the array, although its end lies inside
             (-1, 8, 100, 0), (-5, 8, 100, 0), (-1, 1, 100, 0), (-(1 << 63) + 1, 8, 100, 0),
             (99, 1, 100, 1), (99, 2, 100, 0), ((1 << 63) - 1, 8, 100, 0),
             (1 << 33, 4_000_000_000, (1 << 33) + 4_000_000_000, 1)]
    body = "\n".join(f'printf("%d\\n", (int)span_inside({a}ll, {c}u, {s}ll));'
                     for a, c, s, _ in cases)
    assert run(tmp_path, body) == [str(w) for *_, w in cases]


def test_window_holds(tmp_path):
    top = (1 << 32) - 1
    cases = [(0, 0, 0, 0), (0, 31, 32, 1), (0, 32, 32, 0), (100, 0, 100, 0), (100, 5, 106, 1),
             # windows at the last positions of the largest graph: base + i passes 2^32
             (top - 16, 15, top, 1), (top - 16, 16, top, 0), (top - 16, 17, top, 0),
             (top - 16, 31, top, 0), (top - 40, 32, top, 1), (top - 40, 63, top, 0),
             (top, 1, top, 0)]
    body = "\n".join(f'printf("%d\\n", (int)window_holds({b}u, {i}u, {e}u));'
                     for b, i, e, _ in cases)
    assert run(tmp_path, body) == [str(w) for *_, w in cases]
