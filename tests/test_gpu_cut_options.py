"""svd_cutoff and multiplet_rtol in the final contraction (csrc/cut.cuh) against the oracle's keep rule:
values at which they, not chi_mps, decide cuts.

Tolerances are those of the parity tests (1e-6 in log p for the FP64 path, 1e-3 for the mixed ones); a cut
that follows built-in limits, or pivots of a QR, instead of the option is off by 2e-3 to 0.2 on these shots
(the oracle with such cuts)."""
import numpy as np
import pytest

from oracle import su
from td_inputs import point_sector_3d, rotated_phenomenological, sample_shots

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ROT5, ROT5_HIGH = rotated_phenomenological(5, 4, 0.04, 0.04), rotated_phenomenological(5, 4, 0.08, 0.08)
POINT4 = point_sector_3d(4, 0.1)
CASES = {   # DEM, chi, chi_mps, svd_cutoff, multiplet_rtol, seed of the shots
    "multiplet of rotated d5": (ROT5, 8, 8, 1e-12, 1e-2, 1),
    "multiplet of point d4": (POINT4, 8, 8, 1e-12, 1e-2, 2),
    "multiplet of rotated d5, high rate": (ROT5_HIGH, 8, 4, 1e-12, 1e-3, 1),
    "cutoff above the cap, rotated d5": (ROT5, 8, 4, 1e-2, 1e-8, 2),
    "cutoff above the cap, point d4": (POINT4, 4, 6, 1e-2, 1e-8, 2),
    "cutoff below the cap, rotated d5": (ROT5, 8, 16, 1e-3, 1e-8, 2),
    "cutoff below the cap, rotated d5, high rate": (ROT5_HIGH, 8, 16, 1e-2, 1e-8, 2),
    "cutoff below the cap, point d3": (point_sector_3d(3, 0.1), 8, 64, 3e-2, 1e-8, 2),
}


def _network(name, precision):
    import paper_2310_10722_gb300 as td
    dem, chi, chi_mps, cutoff, rtol, seed = CASES[name]
    det, _ = sample_shots(dem, 4, seed=seed)
    net = td.Network.from_dem(dem, chi=chi, chi_mps=chi_mps, precision=precision, svd_cutoff=cutoff, multiplet_rtol=rtol)
    return net, det, su.su_logprob(dem, det, chi, chi_mps, cutoff, rtol)


def _far(a, b):
    both = np.isneginf(a) & np.isneginf(b)
    return np.abs(np.where(both, 0.0, a) - np.where(both, 0.0, b)).max()


@pytest.mark.parametrize("precision,tol", [(0, 1e-6), (1, 1e-3), (2, 1e-3)])
@pytest.mark.parametrize("name", CASES)
def test_the_options_decide_the_cuts(name, precision, tol):
    net, det, ref = _network(name, precision)
    out = net.coset_logprob(torch.from_numpy(det).cuda()).cpu().numpy()
    net.check()
    assert _far(out, ref) < tol


@pytest.mark.parametrize("name", CASES)
def test_decode_and_gradient_see_one_network(name):
    """The gradient's recorded forward takes every cut by a plain Jacobi SVD: the same log P."""
    net, det, _ = _network(name, 0)
    d = torch.from_numpy(det).cuda()
    lp = net.coset_logprob(d)
    logP, _ = net.grad_logprob(d)
    assert (torch.logsumexp(lp, dim=1) - logP).abs().max().item() < 1e-6
