"""Unpacking (csrc/pack.cu) at the edges of its blocks' split: fewer sites x components than threads with
several slices a thread and without, more than threads (Ls < 5, sixteen site pairs), slices that do not divide
by the threads' stride, a last block with fewer pairs, and FP16 storage.  A packed field comes back as its
storage holds it: unchanged in FP64, rounded to nearest in FP32; in FP16 as half x scale, the scale being the
largest component of the site and slice (within 2^-11 of it)."""
import numpy as np
import pytest

from paper_1611_00298_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,Ls", [((2, 2, 2, 2), 4), ((4, 4, 2, 2), 3), ((6, 4, 2, 6), 4), ((4, 2, 6, 2), 5), ((2, 6, 2, 6), 11),
                                     ((6, 2, 4, 6), 10), ((4, 6, 2, 2), 17), ((2, 2, 6, 4), 33)])
@pytest.mark.parametrize("prec", [0, 1, 2])
def test_round_trip(dims, Ls, prec):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1611_00298_gb300 import eofa
    lat = eofa.Lattice(dims, Ls, bc_t=-1)
    psi = inputs.fermion5d(dims, Ls, 41)
    dev = torch.from_numpy(psi).cuda()
    half = [torch.empty(lat.field_bytes(prec), dtype=torch.uint8, device="cuda") for _ in range(2)]
    back = torch.full_like(dev, np.nan)
    lat.pack_dev(prec, dev, *half)
    lat.unpack_dev(prec, *half, back)
    got = back.cpu().numpy()
    if prec < 2:
        assert np.array_equal(got, psi if prec == 0 else psi.astype(np.complex64).astype(np.complex128))
    else:
        scale = np.maximum(np.abs(psi.real), np.abs(psi.imag)).max(axis=(-2, -1), keepdims=True)
        err = np.maximum(np.abs((got - psi).real), np.abs((got - psi).imag))
        assert np.all(err <= 1.01 * 2.0 ** -11 * scale)
    lat.close()
