"""The factorisation's block inverses by Newton steps, a batch at a time, against numpy's inverse (LAPACK)
in complex128: FP32 blocks by halves and FP64 ones on an FP32 inverse, with blocks in the batch for which
the iteration cannot start or does not contract (singular leading half, entries outside the FP32 range,
a condition beyond FP32), which go to the Gauss-Jordan kernel and leave their neighbours as they were."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2207_10701_gb300 as P  # noqa: E402


def _blocks(n, batch, seed):
    rng = np.random.default_rng(seed)
    a = rng.standard_normal((batch, n, n)) + 1j * rng.standard_normal((batch, n, n))
    return a + 2.0 * np.sqrt(n) * np.exp(1j * rng.uniform(0, 2 * np.pi, (batch, 1, 1))) * np.eye(n)


def _err(x, ref):
    return np.linalg.norm(x - ref, axis=(1, 2)) / np.linalg.norm(ref, axis=(1, 2))


def _inverse(a):
    return P.block_inverse(torch.from_numpy(a).cuda(), kernel=3).cpu().numpy()


@pytest.mark.parametrize("n", [162, 190, 224, 248])
def test_fp32_blocks_with_a_singular_leading_half(n):
    plain = _blocks(n, 5, n).astype(np.complex64)
    mixed = plain.copy()
    h = n // 2
    for z in (1, 4):                 # [[0, B], [C, 0]]
        mixed[z] = 0
        mixed[z, :h, h:] = plain[z, :h, :h]
        mixed[z, h:, :h] = plain[z, h:, h:]
    ref = np.linalg.inv(mixed.astype(np.complex128))
    got = _inverse(mixed)
    # (the bound of the Gauss-Jordan kernels on blocks of this condition)
    assert _err(got, ref).max() < 2e-5
    keep = [0, 2, 3]
    assert np.array_equal(got[keep], _inverse(plain)[keep])
    # inverted by halves and one step: closer than FP32 elimination by far
    assert _err(got, ref)[keep].max() < 2e-6


@pytest.mark.parametrize("n", [16, 33, 128, 131, 161, 248])
def test_fp64_blocks_beyond_fp32(n):
    plain = _blocks(n, 5, n)
    mixed = plain.copy()
    mixed[1] *= 1e45                 # outside the FP32 range
    u, _, v = np.linalg.svd(plain[3])
    mixed[3] = (u * np.logspace(0, -10, n)) @ v
    ref = np.linalg.inv(mixed)
    got = _inverse(mixed)
    e = _err(got, ref)
    # FP64 elimination: some n roundings of 1.1e-16 times the condition (below 10; 1e10 for block 3)
    assert e[[0, 1, 2, 4]].max() < 1e-13 and e[3] < 1e-3, e
    assert np.array_equal(got[[0, 2, 4]], _inverse(plain)[[0, 2, 4]])


@pytest.mark.parametrize("dtype,n", [(np.complex64, 176), (np.complex128, 40)])
def test_singular_block_is_reported(dtype, n):
    a = _blocks(n, 3, 5).astype(dtype)
    a[1] = 0
    with pytest.raises(P.RciError) as ei:
        _inverse(a)
    assert ei.value.status == 5      # RCI_ESINGULAR


@pytest.mark.parametrize("dtype,n", [(np.complex64, 160), (np.complex64, 163), (np.complex64, 250), (np.complex128, 249)])
def test_sizes_it_does_not_take(dtype, n):
    with pytest.raises(P.RciError) as ei:
        _inverse(_blocks(n, 1, 1).astype(dtype))
    assert ei.value.status == 1      # RCI_EINVAL
