"""A shot that meets a non-finite intermediate reads NaN and is reported (TD_ERR_NUMERIC), also where the
overflow is followed by zeros that the kernels leave out.  With both cutoffs (next to) off and low rates the
sweep keeps directions at rounding level, whose transforms leave the range of FP32 storage; the sampled
syndromes are likely ones, so any number below -100, or above 0, would be wrong."""
import numpy as np
import pytest

from td_inputs import point_sector_3d, repetition_phenomenological, rotated_phenomenological, sample_shots

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dem,gram_cutoff", [
    (rotated_phenomenological(5, 5, 1e-4, 1e-4), 0.0),
    (repetition_phenomenological(7, 6, 1e-6, 1e-6), 1e-30),
    (point_sector_3d(4, 1e-4), 1e-30),
])
def test_overflow_reads_nan_and_is_reported(dem, gram_cutoff):
    import paper_2310_10722_gb300 as td
    det, _ = sample_shots(dem, 3, seed=5)
    d = torch.from_numpy(det).cuda()
    net = td.Network.from_dem(dem, chi=8, chi_mps=8, precision=td.TD_FP32, svd_cutoff=0.0, gram_cutoff=gram_cutoff)
    out = net.coset_logprob(d).cpu().numpy()
    with pytest.raises(td.TDError, match="TD_ERR_NUMERIC"):
        net.check()
    assert np.isnan(out).all()
    # the same shots at the default cutoffs
    net = td.Network.from_dem(dem, chi=8, chi_mps=8, precision=td.TD_FP32)
    out = net.coset_logprob(d).cpu().numpy()
    net.check()
    assert (out.max(axis=1) > -100).all() and (out < 1e-3).all()
