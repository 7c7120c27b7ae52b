"""Caps at which a cut's matrices are smaller than a warp's rows (csrc/finlayout.cuh): decodes and the gradient's
recorded forward against the oracle, for every block size of the final contraction.  Tolerance: the parity
tests' 1e-6 in log p."""
import numpy as np
import pytest

from oracle import su
from td_inputs import rotated_phenomenological, sample_shots

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _far(a, b):
    both = np.isneginf(a) & np.isneginf(b)      # a class, or a shot, that truncation leaves without weight
    return np.abs(np.where(both, 0.0, a) - np.where(both, 0.0, b)).max()


@pytest.mark.parametrize("threads", [256, 512, 1024])
@pytest.mark.parametrize("chi,chi_mps", [(4, 4), (8, 2), (2, 8), (8, 1), (9, 1), (11, 1), (6, 5), (15, 2)])
def test_small_caps(chi, chi_mps, threads):
    import paper_2310_10722_gb300 as td
    dem = rotated_phenomenological(5, 3, 0.04, 0.04)
    det, _ = sample_shots(dem, 12, seed=21)
    d = torch.from_numpy(det).cuda()
    ref = su.su_logprob(dem, det, chi, chi_mps)
    net = td.Network.from_dem(dem, chi=chi, chi_mps=chi_mps)
    net.set_schedule(threads, 2048)
    lp = net.coset_logprob(d).cpu().numpy()
    logP, _ = net.grad_logprob(d)
    net.check()
    assert _far(lp, ref) < 1e-6
    assert _far(logP.cpu().numpy(), np.logaddexp(ref[:, 0], ref[:, 1])) < 1e-6
