"""Rows and columns beyond the effective bond dimensions (csrc/absorb.cu): the sweep's tensors are
padded to their static bond dimensions, and the update and tensor-core Gram passes leave out what is
zero.  Cases whose cap is far above the kept ranks, against the exact transfer matrix (nothing is
truncated: the tolerances are those of the exact cases of the parity tests), at one, a few and many
shots -- which also changes how many jobs a gate side's rows are split into."""
import numpy as np
import pytest

from oracle import exact
from td_inputs import point_sector_3d, repetition_phenomenological, rotated_phenomenological, sample_shots

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = {
    "rotated": (lambda: rotated_phenomenological(3, 2, 0.05, 0.04), 16, 32),
    "rotated-13": (lambda: rotated_phenomenological(3, 2, 0.05, 0.04), 13, 32),   # ragged columns of a step
    "rotated-32": (lambda: rotated_phenomenological(3, 2, 0.05, 0.04), 32, 32),
    "point": (lambda: point_sector_3d(3, 0.05), 8, 64),
    "repetition": (lambda: repetition_phenomenological(6, 4, 0.06, 0.03), 32, 8),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("precision,tol", [(0, 1e-9), (2, 5e-6)])
def test_padding_does_not_enter(name, precision, tol):
    import paper_2310_10722_gb300 as td
    make, chi, chi_mps = CASES[name]
    dem = make()
    det, _ = sample_shots(dem, 67, seed=chi)
    net = td.Network.from_dem(dem, chi=chi, chi_mps=chi_mps, precision=precision)
    d = torch.from_numpy(det).cuda()
    full = net.coset_logprob(d).cpu().numpy()
    for first, count in ((5, 1), (20, 9)):
        part = net.coset_logprob(d[first:first + count].contiguous()).cpu().numpy()
        assert np.array_equal(part, full[first:first + count])
    net.check()
    net.close()
    assert np.abs(full - exact.transfer_matrix(dem, det)).max() < tol
