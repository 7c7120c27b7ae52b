"""The truncation cores' grouped Jacobi sweeps (csrc/core.cu): the number of items that share a
block follows the batch (one, two or four), and every grouping does the same operations in the
same order -- so a shot's bits do not depend on the batch it came in."""
import numpy as np
import pytest

from td_inputs import rotated_phenomenological, sample_shots

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("chi", [3, 8, 11, 16, 20])   # one-, two- and four-warp teams, odd sizes
@pytest.mark.parametrize("precision", [0, 2])
def test_bits_do_not_depend_on_the_batch(chi, precision):
    import paper_2310_10722_gb300 as td
    dem = rotated_phenomenological(5, 3, 0.03, 0.03)
    det, _ = sample_shots(dem, 421, seed=60 + chi)
    d = torch.from_numpy(det).cuda()
    net = td.Network.from_dem(dem, chi=chi, chi_mps=4, precision=precision)
    n = net.info()["n_gates"]
    full_w, full_s, _ = net.debug_sweep(d, n)
    full = net.coset_logprob(d)
    for first, count in ((0, 1), (3, 2), (7, 38), (100, 150)):
        part = d[first:first + count].contiguous()
        w, s, _ = net.debug_sweep(part, n)
        assert torch.equal(w, full_w[first:first + count])
        assert torch.equal(s, full_s[first:first + count])
        assert np.array_equal(net.coset_logprob(part).cpu().numpy(), full[first:first + count].cpu().numpy())
    net.check()
    net.close()
