"""FP64 sketches by digit slicing: entrywise error against exact integer products, on inputs
that reach the digits' limits."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gn():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2009_11392_gb300 as g
    return g


@pytest.fixture(scope="module")
def H(gn):
    return gn.Handle()


def sketch(gn, H, A, X, Y):
    m, n = A.shape
    r, rl = X.shape[1], Y.shape[1]
    AX = torch.empty(m, r, dtype=torch.float64, device="cuda")
    YtA = torch.empty(rl, n, dtype=torch.float64, device="cuda")
    H.sketch(A, X, Y, AX, YtA, H.workspace(m, n, r, rl - r, gn.F64))
    assert H.sync_status() == 0
    return AX, YtA


def same_sign(rows, cols, rng):
    """53-bit integers whose base-128 digits below 2^62 are all 60 .. 63, as Python integers and
    as FP64 (times 2^-62); the signs alternate between rows."""
    v = np.zeros((rows, cols), dtype=object)
    for _ in range(9):
        v = v * 128 + rng.integers(60, 64, (rows, cols)).astype(object)
    v = np.vectorize(lambda x: (x >> 10) << 10, otypes=[object])(v)
    v[1::2] *= -1
    return v, v.astype(np.float64) * 2.0 ** -62


@pytest.mark.parametrize("K", [1024, 1500, 3072])
def test_large_digits_of_one_sign(gn, H, K):
    """Every slice product adds up: the sums of the orders 4 and 5 pass 2^24 units unless they
    are cut.  A pass of 1024 then rounds its whole sum twice (as an integer, with the last
    orders), the sum of the passes once more each."""
    rng = np.random.default_rng(K)
    (a, af), (x, xf) = same_sign(4, K, rng), same_sign(3, K, rng)
    put = lambda t: torch.tensor(t, device="cuda")
    A = put(np.tile(af, (100, 1)))
    X = put(np.tile(xf, (14, 1)).T.copy())
    AX, _ = sketch(gn, H, A, X, torch.ones(400, 43, dtype=torch.float64, device="cuda"))
    exact, got = a.dot(x.T), AX[:4, :3].cpu().numpy()
    for i in range(4):
        for j in range(3):
            num, den = float(got[i, j]).as_integer_ratio()
            err = abs(num * 2 ** 124 // den - exact[i, j])
            assert err * 2 ** 53 <= 3 * ((K + 1023) // 1024) * abs(exact[i, j])
