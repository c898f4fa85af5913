"""The quadratic form on either side of the size up to which clusters share a tile, and of the largest
workspace that is kept; and calls that overlap, more of them than workspaces are kept, each from its own
thread on its own stream: the same bits as one call alone."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2207_10701_gb300 as P  # noqa: E402
from oracle.reciprocal import qform_fft  # noqa: E402


def _inputs(n):
    rng = np.random.default_rng(n)
    return rng.standard_normal(n) + 1j * rng.standard_normal(n), np.sinc(0.03 * np.arange(n))


@pytest.mark.parametrize("n", [2048, 2049, 2176, 2177, 32768, 32769])
def test_sizes_beside_the_switches(n):
    v, lags = _inputs(n)
    ref = qform_fft(v, lags)
    got = P.qform_toeplitz(torch.from_numpy(v).cuda(), torch.from_numpy(lags).cuda())
    # sums of n^2 terms whose roundings are random: far below 1e-12 of the sum of a positive form
    assert abs(got - ref) <= 1e-11 * abs(ref), (got, ref)


def test_overlapping_calls():
    sizes = [100, 400, 2176, 2300, 5000, 33000]
    data = []
    for n in sizes:
        v, lags = (torch.from_numpy(t).cuda() for t in _inputs(n))
        data.append((v, lags, P.qform_toeplitz(v, lags)))
    torch.cuda.synchronize()
    wrong = []

    def work(k):
        s = torch.cuda.Stream()
        for i in range(12):
            v, lags, ref = data[(k + i) % len(data)]
            got = P.qform_toeplitz(v, lags, stream=s)
            if got != ref:
                wrong.append((k, i, got, ref))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(14)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong[:3]
