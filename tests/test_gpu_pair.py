"""The two-slices-per-thread dslash kernels (csrc/dslash_pair.cuh) at the edges of their range.

Every even Ls takes them: Ls = 2 (one pair a site), extents without an unrolled build, extents whose
threads do not fill a block, the largest Ls; lattices with a ragged last tile; fields that are only
16-byte aligned fall back to the one-slice kernel.  Reference: the FP64 oracle's hop and dense
5D-local blocks.  Tolerances are those of the storage precision (2^-24 and 2^-11 per value, some
hundred terms per output).
"""
import numpy as np
import pytest

from oracle import dwf
from paper_1611_00298_gb300 import inputs

pytestmark = pytest.mark.gpu

ALPHA, M5, MF = 2.0, 1.8, 0.04


@pytest.fixture(scope="module")
def eofa():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1611_00298_gb300 import eofa as e
    e.load_library()
    return e


def _blocks(Ls, alpha, mf):
    Pp, Pm = dwf.dperp_matrices(Ls, alpha, mf)
    one = np.eye(Ls)
    return np.linalg.inv((4 - M5) * one + Pp), np.linalg.inv((4 - M5) * one + Pm)


def _parity(dims):
    X, Y, Z, T = dims
    t, z, y, x = np.meshgrid(*[np.arange(n) for n in (T, Z, Y, X)], indexing="ij")
    return ((x + y + z + t) % 2)[None, :, :, :, :, None, None]


def _apply(lat, prec, psi, out_par, dag, schur, alpha, mf, offset=0):
    """The packed kernel on one output parity; offset: bytes by which the buffers miss 256-byte alignment."""
    import torch
    nb = lat.field_bytes(prec)
    raw = [torch.empty(nb + 64, dtype=torch.uint8, device="cuda") for _ in range(3)]
    ev, od, out = (r[offset:offset + nb] for r in raw)
    dev = torch.from_numpy(psi).cuda()
    lat.pack_dev(prec, dev, ev, od)
    src = ev if out_par else od
    if schur:
        lat.schur_hop_dev(prec, out_par, dag, src, out, alpha, M5, mf)
    else:
        lat.hop_dev(prec, out_par, dag, src, out)
    res = torch.empty_like(dev)
    lat.unpack_dev(prec, ev if out_par else out, out if out_par else od, res)
    torch.cuda.synchronize()
    return res.cpu().numpy()


@pytest.mark.parametrize("prec,tol", [(1, 2e-6), (2, 3e-3)])
@pytest.mark.parametrize("Ls,dims,alpha,mf", [
    (2, (4, 2, 6, 4), 2.0, 0.04), (4, (2, 2, 2, 2), 1.0, 0.3), (6, (6, 2, 2, 4), 3.0, 1.0), (10, (6, 4, 2, 10), 2.0, 0.04),
    (14, (2, 4, 6, 2), 2.0, 0.0), (20, (4, 4, 2, 6), 1.0, 0.04), (24, (4, 6, 2, 2), 2.0, 0.0362), (34, (2, 2, 4, 6), 2.0, 0.2),
    (64, (2, 4, 2, 2), 2.0, 0.04)])
def test_pair_kernels_match_oracle(eofa, Ls, dims, alpha, mf, prec, tol):
    U = inputs.gauge_field(dims, 0.5, 11)
    psi = inputs.fermion5d(dims, Ls, 12)
    lat = eofa.Lattice(dims, Ls, bc_t=-1)
    lat.gauge_load(U)
    par = _parity(dims)
    Gp, Gm = _blocks(Ls, alpha, mf)
    for dag in (0, 1):
        hop = dwf.wilson_hop(U, psi, -1, dagger=bool(dag))
        full = np.concatenate([np.einsum("st,t...->s...", G.T if dag else G, h)
                               for G, h in ((Gp, hop[..., :2, :]), (Gm, hop[..., 2:, :]))], axis=-2)
        for out_par in (0, 1):
            for schur, ref in ((False, hop), (True, full)):
                got = _apply(lat, prec, psi, out_par, dag, schur, alpha, mf)
                sel = np.broadcast_to(par == out_par, got.shape)
                rel = np.linalg.norm((got - ref)[sel]) / np.linalg.norm(ref[sel])
                assert rel < tol, (dag, out_par, schur, rel)
    lat.close()


@pytest.mark.parametrize("prec,tol", [(1, 1e-6), (2, 2e-3)])
def test_half_aligned_fields_give_the_same_result(eofa, prec, tol):
    dims, Ls = (4, 4, 2, 6), 8
    lat = eofa.Lattice(dims, Ls, bc_t=-1)
    lat.gauge_load(inputs.gauge_field(dims, 0.5, 13))
    psi = inputs.fermion5d(dims, Ls, 14)
    sel = np.broadcast_to(_parity(dims) == 0, psi.shape)
    a = _apply(lat, prec, psi, 0, 0, True, ALPHA, MF)[sel]
    b = _apply(lat, prec, psi, 0, 0, True, ALPHA, MF, offset=16)[sel]
    assert np.linalg.norm(a - b) / np.linalg.norm(a) < tol
    lat.close()


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("Ls", [2, 6, 10, 24])
def test_cg_launches_on_pairs_follow_the_fp64_solve(eofa, Ls, form):
    """All epilogues (both CG forms, with the rank-one terms of both systems): the FP32 solve takes the
    iterations of the FP64 one, and meets the FP64 true residual."""
    dims = (4, 4, 4, 6)
    lat = eofa.Lattice(dims, Ls, bc_t=-1)
    lat.gauge_load(inputs.gauge_field(dims, 0.5, 15))
    b = inputs.fermion5d(dims, Ls, 16)
    for system, shift in ((eofa.SYS_EOFA_L, -0.4), (eofa.SYS_EOFA_R, -1.0), (eofa.SYS_DWF, 0.0)):
        kw = dict(system=system, alpha=ALPHA, M5=M5, mf=MF, m1=0.1, m2=0.8, shift=shift, tol=1e-9)
        _, i64 = lat.solve(b, precision=eofa.PREC_F64, **kw)
        for prec in (eofa.PREC_MIXED_F32, eofa.PREC_MIXED_F16):
            lat.set_cg_form(prec, form)
            _, inf = lat.solve(b, precision=prec, **kw)
            assert inf.true_resid <= 1e-9
            slack = 1.15 if prec == eofa.PREC_MIXED_F32 else 1.6
            assert inf.iters <= slack * i64.iters + 40, (system, prec, inf.iters, i64.iters)
    lat.close()
