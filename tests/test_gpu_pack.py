"""Conversions of 5D fields (csrc/pack.cu), unpacking through shared memory: whole numbers of blocks and
remainders, from one site pair a block (the largest Ls) to sixteen.  A field packed and unpacked comes back as its
storage precision holds it: unchanged in FP64, rounded to nearest in FP32; and a packed FP64 field holds
site j of a parity, component c, slice s at [j][c][s]."""
import numpy as np
import pytest

from paper_1611_00298_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,Ls", [((2, 2, 2, 2), 1), ((4, 2, 6, 4), 5), ((6, 2, 2, 10), 8), ((2, 4, 2, 6), 24), ((6, 4, 2, 2), 63),
                                     ((2, 2, 4, 2), 64), ((10, 6, 2, 4), 2)])
def test_pack_layout_and_round_trip(dims, Ls):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1611_00298_gb300 import eofa
    lat = eofa.Lattice(dims, Ls, bc_t=-1)
    psi = inputs.fermion5d(dims, Ls, 31)
    dev = torch.from_numpy(psi).cuda()
    X, Y, Z, T = dims
    t, z, y, x = np.meshgrid(*[np.arange(n) for n in (T, Z, Y, X)], indexing="ij")
    par = ((x + y + z + t) % 2).reshape(-1)
    for prec in (0, 1):
        half = [torch.empty(lat.field_bytes(prec), dtype=torch.uint8, device="cuda") for _ in range(2)]
        lat.pack_dev(prec, dev, *half)
        back = torch.full_like(dev, np.nan)
        lat.unpack_dev(prec, *half, back)
        torch.cuda.synchronize()
        got = back.cpu().numpy()
        assert np.array_equal(got, psi if prec == 0 else psi.astype(np.complex64).astype(np.complex128))
        if prec == 0:
            for p in (0, 1):
                h = half[p].cpu().numpy().view(np.complex128).reshape(lat.V // 2, 12, Ls)
                assert np.array_equal(h, psi.reshape(Ls, lat.V, 12)[:, par == p].transpose(1, 2, 0))
    lat.close()
