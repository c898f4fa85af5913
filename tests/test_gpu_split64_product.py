"""The digit-split FP64 product by itself, against exact integer sums: terms in one pass of the
accumulators and in several, tiles and their edges, digits of mixed sign, digits that all agree (the
accumulators would pass what FP32 holds exactly) and rows of wide range."""
import pytest

np = pytest.importorskip("numpy")
torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2207_10701_gb300 as P  # noqa: E402

# An FP64 result that is rounded a handful of times
# (once a pass, and where passes are added) stays within 4 x 2^-53 of the sum of the terms' magnitudes;
# entries are cut 2^-55 of the row's largest below it, each side, over the 2 K real terms.
def _product_error(A, B, C0=None, alpha=1.0):
    """Largest |error| / bound of alpha A B + C0 for matrices of complex integers (as float64 pairs)."""
    a, b = A[0] + 1j * A[1], B[0] + 1j * B[1]
    dev = lambda t: torch.from_numpy(np.ascontiguousarray(t)).cuda()[None]  # noqa: E731
    c0 = None if C0 is None else dev(C0[0] + 1j * C0[1])
    got = P.cgemm_batched(dev(a), dev(b), c0, alpha=alpha, beta=1.0, kernel=4)[0].cpu().numpy()
    to = lambda t: np.array([[int(x) for x in r] for r in t], dtype=object)  # noqa: E731
    ar, ai, br, bi = to(A[0]), to(A[1]), to(B[0]), to(B[1])
    s = int(alpha)
    re, im = s * (ar.dot(br) - ai.dot(bi)), s * (ar.dot(bi) + ai.dot(br))
    mag = (abs(ar) + abs(ai)).dot(abs(br) + abs(bi)).astype(float)
    if C0 is not None:
        re, im = re + to(C0[0]), im + to(C0[1])
        mag = mag + abs(C0[0]) + abs(C0[1])
    K = A[0].shape[1]
    top = np.maximum(abs(A[0]), abs(A[1])).max(1)[:, None] * np.maximum(abs(B[0]), abs(B[1])).max(0)[None, :]
    bound = 4 * 2.0 ** -53 * mag + 2 * K * 2.0 ** -54 * top
    err = [[max(abs(int(g.real) - x), abs(int(g.imag) - y)) for g, x, y in zip(r, p, q)]
           for r, p, q in zip(got, re, im)]
    return float((np.array(err, dtype=float) / bound).max())


def _coherent(rng, rows, cols, digit):
    """Integers below 2^53 whose base-256 digits are all about `digit`."""
    v = np.zeros((rows, cols))
    for s in range(6):
        v = v * 256 + (digit + rng.integers(-2, 3, (rows, cols)))
    return v


@pytest.mark.parametrize("M,N,K", [(64, 64, 16), (70, 33, 96), (64, 65, 97), (64, 64, 129), (128, 40, 160),
                                   (65, 64, 171), (72, 17, 248)])
@pytest.mark.parametrize("kind", ["mixed", "coherent", "wide", "one coherent side"])
def test_product_against_exact_sums(M, N, K, kind):
    rng = np.random.default_rng(K)
    rand = lambda r, c: rng.integers(-2 ** 52, 2 ** 52, (r, c)).astype(float)  # noqa: E731
    C0 = None
    if kind == "mixed":
        A, B = [rand(M, K), rand(M, K)], [rand(K, N), rand(K, N)]
    elif kind == "coherent":   # the imaginary part sums 2 K terms of one sign, exactly (no cut entries)
        A, B = [_coherent(rng, M, K, 117)] * 2, [_coherent(rng, K, N, 115)] * 2
    elif kind == "wide":       # each term 2^-4 of the one before, thirteen times over
        w = np.exp2(-(4.0 * np.arange(K) % 52))
        A = [np.rint(rand(M, K) * w), np.rint(rand(M, K) * w)]
        B = [np.rint(rand(K, N) * w[::-1, None]), np.rint(rand(K, N) * w[:, None])]
        C0 = [rand(M, N), rand(M, N)]
    else:
        A, B = [_coherent(rng, M, K, 117)] * 2, [rand(K, N), rand(K, N)]
        C0 = [rand(M, N) * 2.0 ** 40, rand(M, N)]
    assert _product_error(A, B, C0, alpha=1.0 if kind == "coherent" else -1.0) <= 1.0


def test_split_product_refuses_what_it_cannot_take():
    A = torch.zeros((1, 8, 249), dtype=torch.complex128, device="cuda")
    B = torch.zeros((1, 249, 8), dtype=torch.complex128, device="cuda")
    with pytest.raises(P.RciError):
        P.cgemm_batched(A, B, kernel=4)
    with pytest.raises(P.RciError):
        P.cgemm_batched(A[:, :, :8], B[:, :8], alpha=0.5, kernel=4)
    with pytest.raises(P.RciError):
        P.cgemm_batched(A[:, :, :8].to(torch.complex64), B[:, :8].to(torch.complex64), kernel=4)
