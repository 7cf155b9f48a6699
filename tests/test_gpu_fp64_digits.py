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


def entrywise(got, left, right, rows, cols):
    """max |got - left right| / (|left| |right|) over sampled entries, in units of K 2^-53: at
    most 1 for an FP64 sum in any order."""
    a, b = (t.cpu().numpy().astype(np.longdouble) for t in (left[rows], right[:, cols]))
    size = np.abs(a) @ np.abs(b)
    err = np.abs(got[rows][:, cols].cpu().numpy() - a @ b)
    assert np.all(err[size == 0] == 0)
    return float((err[size > 0] / size[size > 0]).max()) / (left.shape[1] * 2.0 ** -53)


def scales(kind, m, n, r, l, rn):
    A, X, Y = rn(m, n), rn(n, r), rn(m, r + l)
    if kind == "hidden column":    # the largest entries meet zeros
        A[:, 3] = 1e20
        A[7] *= 1e18
        X[3] = 0.0
        Y[7] = 0.0
    elif kind == "selection":      # X and Y pick columns and rows
        X.zero_()
        Y.zero_()
        X[torch.randperm(n, device="cuda")[:r], torch.arange(r, device="cuda")] = 1.0
        Y[torch.randperm(m, device="cuda")[:r + l], torch.arange(r + l, device="cuda")] = -1.0
        A *= torch.exp2(torch.randint(-80, 80, (m, n), device="cuda").double())
    elif kind == "graded":         # 1e-30 .. 1 along the contractions, in opposite directions
        d = torch.logspace(0, -30, n, dtype=torch.float64, device="cuda")
        A *= d
        X *= d.flip(0)[:, None]
        Y *= torch.logspace(-30, 0, m, dtype=torch.float64, device="cuda")[:, None]
    elif kind == "sparse":         # 2 % of both operands
        A *= torch.rand_like(A) < 0.02
        X *= torch.rand_like(X) < 0.02
        Y *= torch.rand_like(Y) < 0.02
    return A, X, Y


# one pass and several, a last pass of one, fewer columns than a warp and one more than two
@pytest.mark.parametrize("kind", ["gaussian", "hidden column", "selection", "graded", "sparse"])
@pytest.mark.parametrize("m,n,r,l", [(700, 900, 40, 8), (2500, 1025, 17, 9), (1300, 5000, 65, 3)])
def test_entries_keep_the_bound_of_an_fp64_sum(gn, H, kind, m, n, r, l):
    g = torch.Generator(device="cuda").manual_seed(m)
    rn = lambda a, b: torch.randn(a, b, generator=g, device="cuda", dtype=torch.float64)
    A, X, Y = scales(kind, m, n, r, l, rn)
    AX, YtA = sketch(gn, H, A, X, Y)
    assert m * n * r > 1 << 24
    at = lambda k: torch.arange(0, k, max(1, k // 40), device="cuda")
    assert entrywise(AX, A, X, at(m), at(r)) <= 1.0
    assert entrywise(YtA, Y.T, A, at(r + l), at(n)) <= 1.0


# few rows and columns over a long contraction, for AX and for Y^T A
@pytest.mark.parametrize("m,n,r,l", [(40, 100000, 10, 5), (100, 30000, 10, 5), (60, 16000, 33, 1), (50000, 40, 12, 6)])
def test_skinny_products_stay_on_the_fp64_units(gn, H, m, n, r, l):
    """A tile of 128 rows would be mostly padding and its slices as long as the operands."""
    g = torch.Generator(device="cuda").manual_seed(m)
    rn = lambda a, b: torch.randn(a, b, generator=g, device="cuda", dtype=torch.float64)
    A, X, Y = rn(m, n), rn(n, r), rn(m, r + l)
    before = gn.kernel_launches()
    AX, YtA = sketch(gn, H, A, X, Y)
    # one launch for the skinny product, three per block of 8192 rows or 16384 columns for the other
    assert gn.kernel_launches() - before <= 1 + 3 * (max(m, n) // 8192 + 1)
    at = lambda k: torch.arange(0, k, max(1, k // 12), device="cuda")
    assert entrywise(AX, A, X, at(m), at(r)) <= 1.0
    assert entrywise(YtA, Y.T, A, at(r + l), at(n)) <= 1.0
