"""Zip-up cuts of the final contraction (csrc/cut.cuh): the leading-vector path, the rank path
and the full Jacobi path they leave to, at the sizes where the choice between them turns --
odd caps, chi_mps below and above the bond, cuts with fewer columns than rows, rank-limited
cuts -- against the same-caps oracle.

Tolerance 1e-6 in log p, the parity bound of the FP64 path: the cuts themselves differ from
numpy's SVD by ~1e-14 of the largest singular value, so it is the bound of the sweep before them.
"""
import numpy as np
import pytest

from oracle import su
from td_inputs import point_sector_3d, repetition_phenomenological, rotated_phenomenological, sample_shots

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _decode(dem, det, schedule=None, **kw):
    import paper_2310_10722_gb300 as td
    net = td.Network.from_dem(dem, **kw)
    if schedule:
        net.set_schedule(*schedule)
    out = net.coset_logprob(torch.from_numpy(det).cuda()).cpu().numpy()
    net.check()
    net.close()
    return out


def _far(a, b):
    both = np.isneginf(a) & np.isneginf(b)
    return np.abs(np.where(both, 0.0, a) - np.where(both, 0.0, b)).max()


@pytest.mark.parametrize("chi,chi_mps", [(2, 3), (3, 2), (4, 5), (5, 7), (8, 1), (8, 3), (8, 13), (13, 4), (16, 2)])
@pytest.mark.parametrize("precision", [0, 2])
def test_cuts_match_the_oracle(chi, chi_mps, precision):
    dem = rotated_phenomenological(5, 4, 0.04, 0.04)
    det, _ = sample_shots(dem, 5, seed=90 + chi)
    ref = su.su_logprob(dem, det, chi=chi, chi_mps=chi_mps)
    assert _far(_decode(dem, det, chi=chi, chi_mps=chi_mps, precision=precision), ref) < 1e-6


@pytest.mark.parametrize("dem,chi,chi_mps", [
    (point_sector_3d(4, 0.1), 16, 6),              # wide first row (n < m), 96-column cuts
    (point_sector_3d(3, 0.02), 6, 9),              # low rate: steep spectra, rank-limited cuts
    (rotated_phenomenological(3, 2, 2e-3, 2e-3), 8, 4),    # kept values far below the largest
    (repetition_phenomenological(7, 3, 0.05, 0.05), 8, 2),  # one row: no cut at all
])
def test_cut_shapes_match_the_oracle(dem, chi, chi_mps):
    det, _ = sample_shots(dem, 6, seed=33)
    ref = su.su_logprob(dem, det, chi=chi, chi_mps=chi_mps)
    assert _far(_decode(dem, det, chi=chi, chi_mps=chi_mps), ref) < 1e-6


@pytest.mark.parametrize("schedule", [(256, 2048, True), (256, 2048, False), (512, 2048, False), (1024, 2048, False)])
def test_cut_scratch_placement(schedule):
    """Lanes per pair, shared or global FP32 scratch: the same cuts (1e-9: an FP64 result from
    FP32 starts that round differently)."""
    dem = point_sector_3d(4, 0.08)
    det, _ = sample_shots(dem, 160, seed=5)        # more shots than SMs: two blocks share one
    ref = _decode(dem, det, chi=8, chi_mps=16)
    assert _far(_decode(dem, det, schedule, chi=8, chi_mps=16), ref) < 1e-9


def test_symmetric_syndrome_cuts_a_multiplet():
    """All-zero syndromes of the symmetric lattice have exactly degenerate singular values: cuts
    inside a multiplet, which the full Jacobi path decides."""
    dem = point_sector_3d(4, 0.1)
    det = np.zeros((2, dem.n_det), dtype=np.uint8)
    for chi_mps in (2, 3, 4, 6):
        ref = su.su_logprob(dem, det, chi=8, chi_mps=chi_mps)
        assert _far(_decode(dem, det, chi=8, chi_mps=chi_mps), ref) < 1e-6
