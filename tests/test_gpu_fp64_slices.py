"""The FP64 path's products (gn_sketch on GN_F64 operands), with nine digits per
operand above 2^24 multiply-adds and on the FP64 units below, at the sizes where
the blocking can go wrong, against exact integer products and against the FP64
units."""
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


def run(gn, H, A, X, Y, ws=None, units=False):
    m, n = A.shape
    r, rl = X.shape[1], Y.shape[1]
    AX = torch.empty(m, r, dtype=torch.float64, device="cuda")
    YtA = torch.empty(rl, n, dtype=torch.float64, device="cuda")
    ws = H.workspace(m, n, r, rl - r, gn.F64) if ws is None else ws
    H.set_fp64_tc(not units)
    try:
        H.sketch(A, X, Y, AX, YtA, ws)
        assert H.sync_status() == 0
    finally:
        H.set_fp64_tc(True)
    return AX, YtA


# the first four on the FP64 units (K of one element, one row or column more than a
# tile, K split eight ways); then one pass and several, ragged tiles, blocks of C past
# 8192 rows and 16384 columns, a leading dimension longer than a row (padded operands)
@pytest.mark.parametrize("m,n,r,l,pad", [(4, 1, 1, 1, 0), (300, 257, 31, 3, 0), (33, 65, 17, 1, 2),
                                         (97, 4099, 5, 4, 1), (1025, 1024, 17, 8, 3), (2049, 513, 40, 1, 5),
                                         (8193, 260, 9, 4, 0), (66, 16385, 33, 1, 0), (5000, 4099, 16, 8, 1)])
def test_fp64_sketch_exact_on_scaled_integers(gn, H, m, n, r, l, pad):
    """30-bit integers times per-row or per-column powers of two: every product is
    exact in the digits, so a pass of 1024 rounds once and the sum of p passes at
    most p - 1 times more, each relative to a partial sum of absolute values.  The
    FP64 units round once per term."""
    g = torch.Generator().manual_seed(m + n)
    ints = lambda a, b, bits: torch.randint(-(1 << bits), 1 << bits, (a, b), generator=g)
    Ai, Xi, Yi = ints(m, n, 30), ints(n, r, 20), ints(m, r + l, 20)
    put = lambda t: torch.nn.functional.pad(t, (0, pad)).cuda()[:, :t.shape[1]]
    rows = torch.exp2(torch.randint(-40, 40, (m, 1), generator=g).double())
    cols = torch.exp2(torch.randint(-40, 40, (1, n), generator=g).double())
    AX = run(gn, H, put(Ai.double() * rows), put(Xi.double()), put(Yi.double()))[0].cpu() / rows
    YtA = run(gn, H, put(Ai.double() * cols), put(Xi.double()), put(Yi.double()))[1].cpu() / cols
    for got, left, right in ((AX, Ai, Xi), (YtA, Yi.T, Ai)):
        at = torch.arange(0, got.shape[0], max(1, got.shape[0] // 64))
        # the left operand in two halves of 16 bits: each exact in FP64
        hi, lo, B = (left[at] >> 16).double().numpy(), (left[at] & 0xFFFF).double().numpy(), right.double().numpy()
        exact = (hi @ B).astype(np.longdouble) * 65536 + (lo @ B).astype(np.longdouble)
        size = left[at].abs().double().numpy() @ right.abs().double().numpy()
        err = np.abs(got[at].numpy().astype(np.longdouble) - exact).astype(np.float64)
        K = left.shape[1]
        passes = (K + 1023) // 1024 if K * got.shape[0] * got.shape[1] > 1 << 24 else K + 8
        # (np.longdouble carries 64 bits or more: the reference itself rounds below 2^-64)
        assert np.all(err <= 2.0 ** -53 * (2 * passes) * size)


def test_fp64_sketch_propagates_nonfinite_like_the_units(gn, H):
    m, n, r, l = 1100, 700, 24, 12
    torch.manual_seed(3)
    A = torch.randn(m, n, dtype=torch.float64, device="cuda")
    X = torch.randn(n, r, dtype=torch.float64, device="cuda")
    Y = torch.randn(m, r + l, dtype=torch.float64, device="cuda")
    A[5, 7] = float("nan")
    A[6, 8] = float("inf")
    A[7, 9], A[7, 11] = float("inf"), float("-inf")
    X[30, 4] = float("-inf")
    Y[1090, 2] = float("inf")
    A[1090, 3] = 0.0
    for fast, slow in zip(run(gn, H, A, X, Y), run(gn, H, A, X, Y, units=True)):
        assert torch.equal(fast.isnan(), slow.isnan())
        assert torch.equal(fast.isinf(), slow.isinf())
        inf = slow.isinf()
        assert torch.equal(fast[inf], slow[inf])
        fin = slow.isfinite()
        # n u |A||X|-size error: Gaussian entries, at most 1100 terms
        assert float((fast[fin] - slow[fin]).abs().max()) <= 1e-11


def test_fp64_sketch_runs_in_the_smallest_workspace(gn, H):
    """Without room for the slices the product runs on the FP64 units, and with
    an unaligned workspace the slices start at the next 256-byte boundary."""
    m, n, r, l = 1500, 1100, 20, 10
    torch.manual_seed(4)
    A = torch.randn(m, n, dtype=torch.float64, device="cuda")
    X = torch.randn(n, r, dtype=torch.float64, device="cuda")
    Y = torch.randn(m, r + l, dtype=torch.float64, device="cuda")
    small = torch.empty(8, dtype=torch.uint8, device="cuda")
    units = run(gn, H, A, X, Y, units=True, ws=small)
    for a, b in zip(run(gn, H, A, X, Y, ws=small), units):
        assert torch.equal(a, b)
    whole = H.workspace(m, n, r, l, gn.F64)
    odd = torch.empty(whole.numel() + 8, dtype=torch.uint8, device="cuda")[8:]
    for a, b in zip(run(gn, H, A, X, Y, ws=odd), run(gn, H, A, X, Y, ws=whole)):
        assert torch.equal(a, b)
