"""Which launches of the solver's chain overlap the one before (csrc/chain_rule.h, compiled here with
the host C++ compiler, no GPU): the launch sizes at which both sides were timed on 152 SMs, with the
side that was faster.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1611_00298_gb300", "csrc")

CASES = [
    # kind, blocks, one wave, chained is faster
    ("CHAIN_F64", 4, True, True),        # 4^4 x 8
    ("CHAIN_F64", 72, True, True),       # 6^2 x 8^2 x 8
    ("CHAIN_F64", 81, True, False),      # 6^4 x 12
    ("CHAIN_F64", 128, True, False),     # 8^4 x 8
    ("CHAIN_F64", 256, True, False),     # 8^3 x 16 x 9
    ("CHAIN_F64", 450, True, False),     # 10^2 x 12^2 x 5
    ("CHAIN_F64", 900, True, False),     # 10^2 x 12^2 x 12
    ("CHAIN_ONE", 128, True, True),      # 8^4 x 9
    ("CHAIN_ONE", 256, True, False),     # 8^3 x 16 x 9
    ("CHAIN_ONE", 300, True, False),     # 8 x 10^2 x 12 x 9
    ("CHAIN_ONE", 324, True, True),      # 12^4 x 7
    ("CHAIN_PAIR", 86, True, True),      # 8^4 x 8
    ("CHAIN_PAIR", 171, True, True),     # 8^3 x 16 x 8
    ("CHAIN_PAIR", 264, True, False),    # 10^4 x 10
    ("CHAIN_PAIR", 300, True, False),    # 8 x 10^2 x 12 x 12
    ("CHAIN_PAIR", 512, True, True),     # 8^3 x 16 x 24
    ("CHAIN_PAIR", 608, False, False),   # 16^4 x 16: more than one wave
    ("CHAIN_STREAM", 253, True, True),
    ("CHAIN_STREAM", 1216, False, False),
]


def test_rule_takes_the_faster_side(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    body = "\n".join(f'    std::printf("%d\\n", chain_pays({k}, {n}, {str(w).lower()}, 152));' for k, n, w, _ in CASES)
    src.write_text('#include <cstdio>\n#include "chain_rule.h"\nint main() {\n' + body + "\n    return 0;\n}\n")
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    for case, got in zip(CASES, out):
        assert (got == "1") == case[3], case
