"""Host logic of the 5D-local blocks (csrc/op5.h, compiled here with the host C++ compiler, no GPU):
the constants that op_finalize derives always belong to the block's present coefficients.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1611_00298_gb300", "csrc")

PRELUDE = r"""
#include <cstddef>
#include <cstdio>
#include <cstring>
#include "op5.h"
static Op5 block() {  // the form of G'^-1 = D-tilde M^-1
    Op5 op;
    std::memset(&op, 0, sizeof op);
    for (int h = 0; h < 2; h++) {
        op.inv[h] = op.fwd[h] = 1;
        op.p1[h] = 4.3, op.q1[h] = -1.9, op.p2[h] = 1.5, op.q2[h] = 0.5;
        op.dir1[h] = op.dir2[h] = h;
    }
    op.mass = 0.04;
    op.a_out = 1.0;
    return op;
}
"""


def _run(tmp_path, body):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PRELUDE + "int main() {\n" + body + "\n    return 0;\n}\n")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()


EDITS = ["p1[1] = 3.1", "q1[0] = -0.7", "p2[0] = 0.0", "q2[1] = 2.0", "mass = 0.6", "sigma[1] = 0.3", "dir2[0] = 1",
         "inv[0] = 0", "fwd[1] = 0"]


@pytest.mark.parametrize("edit", EDITS)
def test_constants_follow_an_edit_of_a_finalised_block(tmp_path, edit):
    same, changed = _run(tmp_path, f"""
    Op5 fresh = block();
    fresh.{edit};
    Op5 done = op_finalize(block(), 12), old = done;
    done.{edit};
    fresh = op_finalize(fresh, 12), done = op_finalize(done, 12);
    std::printf("%d %d", !std::memcmp(&fresh, &done, sizeof fresh), !!std::memcmp(&old.mr, &done.mr, sizeof(Op5) - offsetof(Op5, mr)));
""")
    assert same == "1" and changed == "1"


def test_constants_of_another_extent(tmp_path):
    assert _run(tmp_path, """
    Op5 a = op_finalize(op_finalize(block(), 8), 3), b = op_finalize(block(), 3);
    std::printf("%d", !std::memcmp(&a, &b, sizeof a));
""") == ["1"]
