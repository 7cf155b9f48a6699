"""Infinities and NaN in the right-hand side of the triangular solves of gn_factors and
gn_apply: the same entries as on the FP64 units, and none before their column."""
import pytest
import torch

pytestmark = pytest.mark.gpu
INF, NAN = float("inf"), float("nan")


@pytest.fixture(scope="module")
def gn():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2009_11392_gb300 as g
    return g


@pytest.fixture(scope="module")
def H(gn):
    return gn.Handle()


def same(fast, slow):
    assert torch.equal(fast.isnan(), slow.isnan())
    assert torch.equal(fast.isinf(), slow.isinf())
    inf, fin = slow.isinf(), slow.isfinite()
    assert torch.equal(fast[inf], slow[inf])
    assert float((fast[fin] - slow[fin]).norm()) <= 1e-12 * float(slow[fin].norm())


def state(gn, r, l, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    rn = lambda a, b: torch.randn(a, b, generator=g, device="cuda", dtype=torch.float64)
    core = gn.Core.empty(r, l, "cuda")
    core.R.copy_(torch.triu(rn(r, r), 1) / r ** 0.5 + torch.eye(r, dtype=torch.float64, device="cuda"))
    core.Q.copy_(rn(r + l, r) / r ** 0.5)
    core.Q2.copy_(torch.eye(r, dtype=torch.float64, device="cuda"))
    core.R2.copy_(core.R)
    core.k = r
    return core, rn


def both(H, f):
    fast = f()
    H.set_fp64_tc(False)
    try:
        slow = f()
    finally:
        H.set_fp64_tc(True)
    assert H.sync_status() == 0
    return fast, slow


# few rows, digit-sliced products under base blocks of 128 and of 32 columns
@pytest.mark.parametrize("m,r", [(300, 300), (3000, 256), (9000, 300)])
@pytest.mark.parametrize("trunc", [0, 1])
def test_factors(gn, H, m, r, trunc):
    n, l = 50, 3
    core, rn = state(gn, r, l, m)
    if trunc:
        core.k, core.sgn = r - 3, 1
    AX = rn(m, r)
    AX[5, 140], AX[6, 200], AX[7, 20], AX[8, 130], AX[8, 250] = INF, NAN, -INF, INF, -INF
    YtA = rn(r + l, n)

    def run():
        F = torch.zeros(m, r, dtype=torch.float64, device="cuda")
        G = torch.zeros(r, n, dtype=torch.float64, device="cuda")
        H.factors(AX, YtA, core, F, G, H.workspace(max(m, 2 * r), max(n, 2 * r), r, l, gn.F64))
        return F
    fast, slow = both(H, run)
    same(fast, slow)
    if not trunc:   # F R = AX: the columns before a non-finite one stay finite, the others do not
        for row, col in ((5, 140), (6, 200), (7, 20), (8, 130)):
            assert bool(fast[row, :col].isfinite().all()) and not bool(fast[row, col:].isfinite().any())
    assert bool(fast[9:].isfinite().all())


@pytest.mark.parametrize("kw", [6, 1500])
@pytest.mark.parametrize("side", [0, 1])
def test_apply(gn, H, kw, side):
    m, n, r, l = 400, 420, 256, 4
    core, rn = state(gn, r, l, kw)
    AX, YtA = rn(m, r), rn(r + l, n)
    W = rn(n, kw) if side == 0 else rn(kw, m)
    AX[30, 140] = INF
    W[(2, 3) if side == 0 else (3, 2)] = NAN
    fast, slow = both(H, lambda: H.apply(AX, YtA, core, W, side=side))
    same(fast, slow)
