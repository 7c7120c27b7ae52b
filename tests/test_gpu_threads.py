"""One network per thread and stream, decoding at the same time: each gets what it gets alone.  The launches of
small and large batches ask for different amounts of shared memory."""
import threading

import numpy as np
import pytest

from td_inputs import rotated_phenomenological, sample_shots

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", [0, 2])
def test_concurrent_networks(precision):
    import paper_2310_10722_gb300 as td
    dem = rotated_phenomenological(5, 4, 0.03, 0.03)
    batches, passes = (1, 700, 2, 400), 60
    nets, dets, alone = [], [], []
    for B in batches:
        nets.append(td.Network.from_dem(dem, chi=8, chi_mps=8, precision=precision, max_wave=B))
        dets.append(torch.from_numpy(sample_shots(dem, B, seed=B)[0]).cuda())
        alone.append(nets[-1].coset_logprob(dets[-1]).cpu().numpy())
    results, errors = [None] * len(batches), []

    def work(i):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                for _ in range(passes):
                    out = nets[i].coset_logprob(dets[i])
                results[i] = out.cpu().numpy()
            nets[i].check(stream)
        except Exception as e:   # an assertion in a thread would be lost
            errors.append((batches[i], str(e)))

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(batches))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for got, want in zip(results, alone):
        np.testing.assert_array_equal(got, want)
