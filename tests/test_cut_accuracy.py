"""The cuts of a decode (csrc/cut.cuh) against the recorded cuts of the gradient's forward, a plain FP64
Jacobi SVD of each: on the FP64 path both contract the same final network, so their log P differ by the cuts
alone.  Near and below threshold.

Bound 1e-11: a cut is right to 6e-14 of its largest singular value (against numpy's SVD), and the networks have
up to 60.  A cut left at FP32 accuracy is seen: the oracle with the left vectors of its truncating cuts from an
FP32 SVD is off by more than ten times that."""
import numpy as np
import pytest

from oracle import su
from td_inputs import point_sector_3d, rotated_phenomenological, sample_shots

torch = pytest.importorskip("torch")
CASES = {   # DEM, chi, chi_mps
    "rotated d5": (rotated_phenomenological(5, 4, 0.04, 0.04), 8, 8),
    "rotated d7": (rotated_phenomenological(7, 5, 0.03, 0.03), 8, 8),
    "rotated d7 below threshold": (rotated_phenomenological(7, 5, 5e-3, 5e-3), 8, 8),
    "rotated d7 below threshold, small cap": (rotated_phenomenological(7, 5, 1e-2, 1e-2), 8, 4),
    "point d4 below threshold": (point_sector_3d(4, 2e-2), 8, 6),
}
TOL = 1e-11


def _case(name):
    dem, chi, chi_mps = CASES[name]
    return dem, chi, chi_mps, sample_shots(dem, 6, seed=31)[0]


@pytest.mark.parametrize("name", CASES)
def test_cuts_at_fp32_accuracy_would_be_seen(name, monkeypatch):
    dem, chi, chi_mps, det = _case(name)
    ref = su.su_logprob(dem, det, chi, chi_mps)
    svd = np.linalg.svd

    def fp32_cut(M, **kw):
        if kw.get("full_matrices", True) or min(M.shape) <= chi_mps:
            return svd(M, **kw)
        U = svd((M / np.abs(M).max()).astype(np.float32), full_matrices=False)[0]
        U = np.linalg.qr(U.astype(np.float64))[0]
        C = U.T @ M
        s = np.linalg.norm(C, axis=1)
        return U, s, C / s[:, None]

    monkeypatch.setattr(su.np.linalg, "svd", fp32_cut)
    out = su.su_logprob(dem, det, chi, chi_mps)
    assert np.abs(np.logaddexp(*out.T) - np.logaddexp(*ref.T)).max() > 10 * TOL


def _apart(dem, det, chi, chi_mps, schedule=(256, 2048), **kw):
    import paper_2310_10722_gb300 as td
    net = td.Network.from_dem(dem, chi=chi, chi_mps=chi_mps, **kw)
    net.set_schedule(*schedule)
    d = torch.from_numpy(det).cuda()
    lp = net.coset_logprob(d)
    logP, _ = net.grad_logprob(d)
    net.check()
    return (torch.logsumexp(lp, dim=1) - logP).abs().max().item()


@pytest.mark.gpu
@pytest.mark.parametrize("name", CASES)
def test_cuts_to_fp64_accuracy(name):
    dem, chi, chi_mps, det = _case(name)
    assert _apart(dem, det, chi, chi_mps) < TOL


@pytest.mark.gpu
@pytest.mark.parametrize("p,q,chi,rtol,shots,seed", [(0.00418, 0.03563, 9, 1e-6, 1, 3244), (0.02076, 0.00709, 7, 1e-2, 3, 3328)])
def test_values_next_to_the_cutoff(p, q, chi, rtol, shots, seed):
    """Cuts that drop only values below svd_cutoff, with some next to it, on unlikely syndromes: which ones go is
    seen in log P (1.4e-9 and 4e-10 where the pivots of a QR decide it)."""
    dem = rotated_phenomenological(7, 4, p, q)
    assert _apart(dem, sample_shots(dem, shots, seed=seed)[0], chi, 32, multiplet_rtol=rtol) < TOL


@pytest.mark.gpu
def test_cut_next_to_a_multiplet():
    """A gap just above the multiplet rule's: the residual has to fall below its usual bound by the gap (8.9e-10
    where it does not)."""
    dem = rotated_phenomenological(7, 4, 0.03234, 0.00364)
    det = sample_shots(dem, 3, seed=2278)[0]
    assert _apart(dem, det, 16, 2, (512, 4096, False), multiplet_rtol=1e-4) < TOL
