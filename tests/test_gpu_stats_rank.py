"""Statistics of cuts that truncate nothing but values below svd_cutoff (the rank path of csrc/cut.cuh): the
discarded fraction as include/td.h defines it, against the oracle's singular values.

The dropped values are some 5e-12 of the largest and known to FP64 rounding, 1e-16 of the largest: 2e-5 of
themselves, 4e-5 in their squares; the bound is 1e-2 for the sweep before them."""
import numpy as np
import pytest

from oracle import su
from td_inputs import point_sector_3d, sample_shots

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", [0, 2])
def test_discarded_fraction_of_rank_cuts(precision):
    import paper_2310_10722_gb300 as td
    dem = point_sector_3d(4, 5e-4)
    det, _ = sample_shots(dem, 6, seed=4)
    net = td.Network.from_dem(dem, chi=8, chi_mps=64, svd_cutoff=1e-11, precision=precision)
    _, st = net.coset_logprob_stats(torch.from_numpy(det).cuda())
    net.check()
    ref = su.su_truncation_stats(dem, det, 8, 64, cutoff=1e-11)
    assert (ref[:, 2] > 1e-24).all()
    np.testing.assert_allclose(st.cpu().numpy()[:, 2:], ref[:, 2:], rtol=1e-2)
