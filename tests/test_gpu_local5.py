"""FP64 5D-local passes and columns without their leading factor (csrc/local5d.cu, dslash_impl.cuh).

The forms that take a new route: D-tilde and M as a two-point stencil (with and without the axpy, Ls = 1
where the neighbour is the slice itself, Ls = 2), the inverse with and without the rank-one term at extents
with and without an unrolled build.  Reference: the FP64 oracle; 1e-12 is some thousand roundings.
"""
import numpy as np
import pytest

from oracle import dwf
from paper_1611_00298_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eofa():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1611_00298_gb300 import eofa as e
    e.load_library()
    return e


@pytest.mark.parametrize("Ls", [1, 2, 3, 7, 8, 13, 16, 24, 37, 64])
@pytest.mark.parametrize("alpha,mf", [(1.0, 0.0), (2.0, 0.04), (4.0, 1.0)])
def test_operators_over_ls(eofa, Ls, alpha, mf):
    dims = (2, 4, 2, 6)
    U = inputs.gauge_field(dims, 0.5, 21)
    psi = inputs.fermion5d(dims, Ls, 22)
    lat = eofa.Lattice(dims, Ls, bc_t=-1)
    lat.gauge_load(U)
    for got, ref in ((lat.dwf_apply(psi, alpha, 1.8, mf), dwf.dwf(U, psi, alpha, 1.8, mf, -1)),
                     (lat.dwf_apply(psi, alpha, 1.8, mf, dagger=True), dwf.dwf_dag(U, psi, alpha, 1.8, mf, -1)),
                     (lat.eofa_apply(psi, alpha, 1.8, mf), dwf.deofa(U, psi, alpha, 1.8, mf, -1))):
        assert np.linalg.norm(got - ref) / np.linalg.norm(ref) < 1e-12
    lat.close()


@pytest.mark.parametrize("Ls", [1, 5, 12])
def test_fp64_solves_with_rank_one_terms(eofa, Ls):
    """Columns with the rank-one sum, odd and unrolled Ls, and a warm start (D-tilde in place): the true
    residual is recomputed by the library from the unpreconditioned system."""
    dims = (4, 2, 4, 4)
    lat = eofa.Lattice(dims, Ls, bc_t=-1)
    lat.gauge_load(inputs.gauge_field(dims, 0.5, 23))
    b = inputs.fermion5d(dims, Ls, 24)
    for system, shift in ((eofa.SYS_EOFA_L, -0.5), (eofa.SYS_EOFA_R, -1.0), (eofa.SYS_DWF, 0.0)):
        kw = dict(system=system, alpha=2.0, M5=1.8, mf=0.1, m1=0.1, m2=0.8, shift=shift, precision=eofa.PREC_F64)
        x, inf = lat.solve(b, tol=1e-11, **kw)
        assert inf.true_resid <= 1e-11
        y, again = lat.solve(b, x0=x, tol=1e-10, **kw)
        assert again.iters <= 4 and np.linalg.norm(x - y) / np.linalg.norm(x) < 1e-8
    lat.close()
