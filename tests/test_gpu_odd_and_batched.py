"""Routes of the mixed-precision solves beside the unrolled two-slice kernels: odd Ls, alone (one-slice kernels,
their columns without a leading factor, all epilogues of both CG forms, the rank-one terms of both sides) and
in lock-step batches (the multi-system kernels), and batches at even Ls with and without an unrolled build.

A solve meets the FP64 true residual and follows the FP64 one in its iterations; a batch's solutions are put
through the oracle's operators.
"""
import numpy as np
import pytest

from oracle import dwf, eofa as oeofa
from paper_1611_00298_gb300 import inputs

pytestmark = pytest.mark.gpu

ALPHA, M5 = 2.0, 1.8


@pytest.fixture(scope="module")
def eofa():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1611_00298_gb300 import eofa as e
    e.load_library()
    return e


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("Ls", [5, 7, 13])
def test_odd_extents_follow_the_fp64_solve(eofa, Ls, form):
    dims = (4, 4, 4, 6)
    lat = eofa.Lattice(dims, Ls, bc_t=-1)
    lat.gauge_load(inputs.gauge_field(dims, 0.5, 61))
    b = inputs.fermion5d(dims, Ls, 62)
    for system, shift in ((eofa.SYS_EOFA_L, -0.4), (eofa.SYS_EOFA_R, -1.0), (eofa.SYS_DWF, 0.0)):
        kw = dict(system=system, alpha=ALPHA, M5=M5, mf=0.04, m1=0.1, m2=0.8, shift=shift, tol=1e-9)
        x64, i64 = lat.solve(b, precision=eofa.PREC_F64, **kw)
        for prec in (eofa.PREC_MIXED_F32, eofa.PREC_MIXED_F16):
            lat.set_cg_form(prec, form)
            x, inf = lat.solve(b, precision=prec, **kw)
            assert inf.true_resid <= 1e-9
            slack = 1.15 if prec == eofa.PREC_MIXED_F32 else 1.6
            assert inf.iters <= slack * i64.iters + 40, (system, prec, inf.iters, i64.iters)
            assert np.linalg.norm(x - x64) / np.linalg.norm(x64) < 1e-6
    lat.close()


@pytest.mark.parametrize("prec", ["PREC_MIXED_F32", "PREC_MIXED_F16"])
@pytest.mark.parametrize("Ls", [5, 7, 10, 12, 24])
def test_batches_solve_their_systems(eofa, Ls, prec):
    dims = (4, 4, 2, 4)
    U = inputs.gauge_field(dims, 0.5, 63)
    lat = eofa.Lattice(dims, Ls, bc_t=-1)
    lat.gauge_load(U)
    sys_ = [("L", eofa.SYS_EOFA_L, 0.1, 0.6, -0.3), ("R", eofa.SYS_EOFA_R, 0.2, 0.8, -1.0), ("R", eofa.SYS_EOFA_R, 0.1, 0.6, -0.5),
            (None, eofa.SYS_DWF, 0.2, 0.0, 0.0)]
    params = [lat.solve_params(system=s, alpha=ALPHA, M5=M5, mf=m1, m1=m1, m2=m2, shift=a, precision=getattr(eofa, prec), tol=1e-10)
              for _, s, m1, m2, a in sys_]
    bs = [inputs.fermion5d(dims, Ls, 64, stream=70 + k) for k in range(len(sys_))]
    xs = [np.zeros_like(b) for b in bs]
    info = eofa.solve_batched([lat] * len(sys_), params, bs, xs)
    for (side, _, m1, m2, a), b, x, inf in zip(sys_, bs, xs, info):
        Ax = dwf.dwf(U, x, ALPHA, M5, m1, -1) if side is None else oeofa.system_apply(U, x, ALPHA, M5, m1, m2, side, a, -1)
        assert inf.status == eofa.OK
        assert np.linalg.norm(b - Ax) / np.linalg.norm(b) <= 1.05e-10
    lat.close()


def test_force_of_16_byte_aligned_solutions(eofa):
    """Solutions that start 16 bytes past a 32-byte boundary take the narrow loads: the same products and sums."""
    import torch
    dims, Ls = (4, 2, 6, 4), 7
    lat = eofa.Lattice(dims, Ls, bc_t=-1)
    lat.gauge_load(inputs.gauge_field(dims, 0.5, 65))
    chi = [torch.from_numpy(inputs.fermion5d(dims, Ls, 66, stream=80 + k)).cuda() for k in range(2)]
    n = chi[0].numel()

    def force(call, offs):
        raw = [torch.empty(n + 2, dtype=torch.complex128, device="cuda") for _ in chi]
        c = [r[o:o + n] for r, o in zip(raw, offs)]
        for dst, src in zip(c, chi):
            assert (dst.data_ptr() % 32 == 16) == (dst is c[0] and offs[0] == 1 or dst is c[1] and offs[1] == 1)
            dst.copy_(src.reshape(-1))
        F = torch.empty(lat.shapeU, dtype=torch.complex128, device="cuda")
        call(0.9, c[0], c[1], F)
        return F.cpu().numpy()

    for call in (lat.force_from_chi_dev, lat.grad_from_chi_dev):
        want = force(call, (0, 0))
        for offs in ((1, 1), (1, 0), (0, 1)):
            assert np.max(np.abs(force(call, offs) - want)) <= 1e-15 * np.max(np.abs(want))
    lat.close()


def test_two_contexts_solve_at_once(eofa):
    """Two host threads, each with its own lattice and stream, on lattices small enough for chained launches:
    the solutions are those of the same solves one after the other."""
    import threading
    import torch
    prec = (eofa.PREC_MIXED_F32, eofa.PREC_MIXED_F16)
    lats, bs, want = [], [], []
    kw = dict(system=eofa.SYS_EOFA_R, alpha=ALPHA, M5=M5, m1=0.1, m2=0.8, shift=-1.0, tol=1e-10)
    for k, (dims, Ls) in enumerate((((4, 4, 4, 4), 8), ((4, 4, 4, 6), 7))):
        lat = eofa.Lattice(dims, Ls, bc_t=-1)
        lat.gauge_load(inputs.gauge_field(dims, 0.5, 67 + k))
        for p in prec:
            lat.set_cg_form(p, k)
        b = torch.from_numpy(inputs.fermion5d(dims, Ls, 69 + k)).cuda()
        lats.append(lat)
        bs.append(b)
        want.append([])
        for p in prec:
            x = torch.zeros_like(b)
            lat.solve_dev(b, x, precision=p, **kw)
            want[k].append(x)
    torch.cuda.synchronize()
    got, fail = [[], []], []

    def work(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for i in range(6):
                    x = torch.zeros_like(bs[k])
                    inf = lats[k].solve_dev(bs[k], x, precision=prec[i % 2], **kw)
                    assert inf.true_resid <= 1e-10
                    got[k].append(x)
                torch.cuda.current_stream().synchronize()
        except Exception as e:  # reported by the main thread
            fail.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not fail, fail
    for k in range(2):
        for i, x in enumerate(got[k]):
            assert torch.linalg.vector_norm(x - want[k][i % 2]) <= 1e-8 * torch.linalg.vector_norm(x)
    for lat in lats:
        lat.close()
