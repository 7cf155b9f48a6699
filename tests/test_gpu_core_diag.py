"""The detector's norms and truncation rank (gn_core) at the edges of their
128-column blocks and of the CTAs' shares, against a plain FP64 power iteration."""
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


def core_of(gn, H, C, eps, mode):
    rl, r = C.shape
    core = gn.Core.empty(r, rl - r, "cuda")
    core.C.copy_(C)
    n = max(rl, r)
    YtA = torch.zeros(rl, n, dtype=torch.float64, device="cuda")
    X = torch.zeros(n, r, dtype=torch.float64, device="cuda")
    ws = H.workspace(n + rl, n, r, rl - r, gn.F64)
    H.core(YtA, X, eps, mode | gn.CORE_C_GIVEN, core, ws)
    return core


def power(f, r, iters=6):
    z = torch.full((r,), r ** -0.5, dtype=torch.float64, device="cuda")
    for _ in range(iters):
        w = f(z)
        nw = w.norm()
        z = w / nw
    return float(nw.sqrt())


# one entry; fewer columns than CTAs; off the 8-column shares; 127 / 128 / 129: the
# block edge; several blocks with a ragged last one
@pytest.mark.parametrize("r", [1, 2, 15, 20, 33, 64, 100, 127, 128, 129, 257, 520, 1000])
def test_norm_estimates(gn, H, r):
    torch.manual_seed(r)
    C = torch.randn(r + r // 2 + 1, r, dtype=torch.float64, device="cuda")
    C *= torch.logspace(0, -3, r, dtype=torch.float64, device="cuda")
    core = core_of(gn, H, C, 1e-12, gn.AUTO | gn.EPS_RELATIVE)
    assert H.sync_status() == 0
    R = core.R
    solve = lambda z: torch.linalg.solve_triangular(
        R, torch.linalg.solve_triangular(R.T, z[:, None], upper=False), upper=True)[:, 0]
    # the products and solves round at r u kappa(R), kappa(R) below 1e5: 1e-8 at r = 1000
    assert abs(core.rinv_est / power(solve, r) - 1) <= 1e-8
    assert abs(core.c_norm_est / power(lambda z: R.T @ (R @ z), r) - 1) <= 1e-12
    assert core.k == r and core.sgn == 0
    assert abs(core.eps_abs / (1e-12 * core.c_norm_est) - 1) <= 1e-14


@pytest.mark.parametrize("r,p", [(20, 7), (100, 1), (130, 128), (300, 129)])
def test_truncation_rank_and_zero_pivots(gn, H, r, p):
    """Columns p.. of C are zero or tiny: an exactly zero pivot makes the estimate
    infinite, and either way the rank is p."""
    torch.manual_seed(r + p)
    C = torch.randn(r + 9, r, dtype=torch.float64, device="cuda")
    C[:, p:] = 0.0
    core = core_of(gn, H, C, 1e-10, gn.AUTO | gn.EPS_RELATIVE)
    assert core.sgn == 1 and core.k == p and core.rinv_est == float("inf")
    C[:, p:] = 1e-14 * torch.randn(r + 9, r - p, dtype=torch.float64, device="cuda")
    core = core_of(gn, H, C, 1e-10, gn.AUTO | gn.EPS_RELATIVE)
    assert core.sgn == 1 and core.k == p and 1e12 < core.rinv_est < 1e18
    core = core_of(gn, H, C, 1e-10, gn.SGN)   # an absolute threshold: no norm of C
    assert core.sgn == 1 and core.k == p and core.c_norm_est == 0.0
    assert H.sync_status() == 0


def test_nan_core_is_an_error(gn, H):
    C = torch.randn(60, 40, dtype=torch.float64, device="cuda")
    C[3, 5] = float("nan")
    with pytest.raises(gn.GNError) as e:
        core_of(gn, H, C, 1e-10, gn.AUTO | gn.EPS_RELATIVE)
    assert e.value.status == 6
    assert H.sync_status() == 6
