"""The reverse sweep at odd and even sizes of its kernels: bond caps below, at and above a warp's
columns, boundary caps with odd and even numbers of columns in the recorded cuts (csrc/cut.cuh,
csrc/adjoint.cu) -- against the oracle's reverse sweep, at log-uniform rates (no multiplets), with the
tolerances of the full-size comparison."""
import numpy as np
import pytest

from oracle import reverse
from td_inputs import log_uniform_rates, rotated_phenomenological, sample_shots

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("chi,chi_mps", [(2, 3), (3, 5), (5, 8), (6, 4), (8, 7)])
def test_against_the_oracle(chi, chi_mps):
    import paper_2310_10722_gb300 as td
    dem = log_uniform_rates(rotated_phenomenological(3, 3, 0.01, 0.01), seed=31)
    det, _ = sample_shots(dem, 2, seed=32 + chi)
    net = td.Network.from_dem(dem, chi=chi, chi_mps=chi_mps)
    jac = reverse.object_jacobian(dem)
    for b in range(2):
        logP, g = net.grad_logprob(torch.from_numpy(det[b:b + 1]).cuda())
        lp_ref, g_ref = reverse.reverse_grad_total_logprob(dem, det[b:b + 1], chi, chi_mps, jac=jac)
        assert abs(logP.item() - lp_ref[0]) < 1e-6
        g = g.cpu().numpy()
        assert np.abs(g - g_ref[0]).max() / max(1.0, np.abs(g_ref[0]).max()) < 1e-5
    net.close()
