"""Which 5D-local blocks the two-slice kernels take (csrc/pair_op.h, compiled here with the host C++
compiler, no GPU), and the constants they get: the block applied to pairs of slices with them, written
out here, against the dense matrices of the definition.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1611_00298_gb300", "csrc")

PRELUDE = r"""
#include <cstdio>
#include <cstring>
#include "pair_op.h"
static Op5 block(int dag) {
    Op5 op;
    std::memset(&op, 0, sizeof op);
    for (int h = 0; h < 2; h++) {
        op.inv[h] = op.fwd[h] = 1;
        op.p1[h] = 3.2, op.q1[h] = -0.9, op.p2[h] = 1.5, op.q2[h] = 0.5;
        op.dir1[h] = op.dir2[h] = h ^ dag;
    }
    op.mass = 0.3;
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


@pytest.mark.parametrize("edit,taken", [
    ("", True), ("op.sigma[0] = 0.2;", True), ("op.sigma[1] = -0.2;", True), ("op.fwd[0] = op.fwd[1] = 0;", True),
    ("op.fwd[1] = 0;", True),
    ("op.sigma[0] = 0.2; op.sigma[1] = -0.2;", False),  # rank-one terms on both chiralities
    ("op.inv[1] = 0;", False), ("op.dir2[0] = 1;", False), ("op.dir1[0] = op.dir2[0] = 1;", False)])
def test_forms_taken(tmp_path, edit, taken):
    got = _run(tmp_path, f"""
    Op5 op = block(0);
    {edit}
    dsl::PairOp o;
    std::printf("%d", dsl::pair_op_of(op_finalize(op, 8), 8, true, 1.0, o));
""")
    assert got == [str(int(taken))]


@pytest.mark.parametrize("Ls", [2, 6, 12])
@pytest.mark.parametrize("dag", [0, 1])
def test_constants_give_the_block(tmp_path, Ls, dag):
    out = _run(tmp_path, f"""
    dsl::PairOp o;
    if (!dsl::pair_op_of(op_finalize(block({dag}), {Ls}), {Ls}, {str(not dag).lower()}, -0.5, o)) return 1;
    for (int h = 0; h < 2; h++)
        std::printf("%.9g %.9g %.9g %.9g %.9g %.9g ", o.mr[h], o.m2[h], o.c1[h], o.k0[h], o.k1[h], o.cor[h]);
""")
    c = np.array(out, dtype=float).reshape(2, 6)
    for h in range(2):
        mr, m2, c1, k0, k1, cor = c[h]
        up = (h ^ dag) == 0
        L = np.diag(np.ones(Ls - 1), -1)
        L[0, Ls - 1] = -0.3
        L = L if up else L.T
        want = -0.5 * (1.5 * np.eye(Ls) + 0.5 * L) @ np.linalg.inv(3.2 * np.eye(Ls) - 0.9 * L)
        got = np.empty((Ls, Ls))
        for col in range(Ls):
            x = np.zeros(Ls)
            x[col] = 1.0
            x = x if up else x[::-1]
            P = 0.0
            for i in range(Ls // 2):  # end values of the pairs, then the corner
                P = x[2 * i + 1] + mr * x[2 * i] + m2 * P
            k, y = cor * P, np.empty(Ls)
            for i in range(Ls // 2):
                y[2 * i], y[2 * i + 1] = c1 * x[2 * i] + k0 * k, c1 * x[2 * i + 1] + k0 * x[2 * i] + k1 * k
                k = x[2 * i + 1] + mr * x[2 * i] + m2 * k
            got[:, col] = y if up else y[::-1]
        assert np.max(np.abs(got - want)) < 20 * 2.0 ** -24  # the constants are FP32; entries below 1
