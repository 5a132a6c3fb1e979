"""The launch profile counts every launch between start and stop, also beyond the event pairs that it holds."""
import pytest

from paper_1611_00298_gb300 import inputs

pytestmark = pytest.mark.gpu

HELD = 65536


@pytest.mark.parametrize("n", [3, HELD, HELD + 3001])
def test_every_launch_is_counted(n):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1611_00298_gb300 import eofa
    dims, Ls = (2, 2, 2, 2), 2
    lat = eofa.Lattice(dims, Ls, bc_t=-1)
    lat.gauge_load(inputs.gauge_field(dims, 0.5, 51))
    a, b = (torch.zeros(lat.field_bytes(eofa.PREC_F64), dtype=torch.uint8, device="cuda") for _ in range(2))
    for _ in range(2):  # a second profile starts from nothing
        lat.profile_start()
        for _ in range(n):
            lat.hop_dev(eofa.PREC_F64, 0, 0, a, b)
        launches, ms, nbytes = lat.profile_stop()
        assert launches == [n, 0, 0, 0, 0, 0]
        assert ms[0] > 0.0 and ms[1:] == [0.0] * 5
        assert nbytes[0] == n * (lat.V // 2 * Ls) * (384 + 1152 // Ls)
    lat.close()
