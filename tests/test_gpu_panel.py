"""The Householder panels of the core's QR (gn_core) at the edges of their row
split, with dropped columns and with entries near the ends of the FP64 range."""
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


def qr(gn, H, C):
    rl, r = C.shape
    core = gn.Core.empty(r, rl - r, "cuda")
    core.C.copy_(C)
    YtA = torch.zeros(rl, rl, dtype=torch.float64, device="cuda")
    X = torch.zeros(rl, r, dtype=torch.float64, device="cuda")
    H.core(YtA, X, 0.0, gn.PLAIN | gn.CORE_C_GIVEN, core, H.workspace(2 * rl, rl, r, rl - r, gn.F64))
    return core.Q, core.R


def check(C, Q, R):
    rl, r = C.shape
    scale = float(C.abs().max())
    C, R = C / scale, R / scale
    # Householder QR: backward error and loss of orthogonality of order r u per column
    assert float((Q @ R - C).norm() / C.norm()) <= 2e-15 * (r + 10)
    assert float((Q.T @ Q - torch.eye(r, dtype=torch.float64, device="cuda")).norm()) <= 2e-15 * r ** 0.5 * (r + 10)
    assert bool((torch.diagonal(R) >= 0).all()) and torch.equal(R, torch.triu(R))


# fewer rows than CTAs; one row per CTA or warp; partial panels; a last panel of one
# column; the register kernel's last size (3072 rows) and the first past it
@pytest.mark.parametrize("rl,r", [(2, 1), (3, 2), (16, 15), (17, 16), (33, 32), (34, 33), (64, 31), (65, 64), (97, 63),
                                  (130, 128), (700, 97), (1537, 40), (3008, 64), (3072, 33), (3073, 33)])
def test_qr_shapes(gn, H, rl, r):
    torch.manual_seed(rl)
    C = torch.randn(rl, r, dtype=torch.float64, device="cuda")
    check(C, *qr(gn, H, C))
    assert H.sync_status() == 0


@pytest.mark.parametrize("scale", [1e-300, 1e-200, 1e-140, 1e140, 1e150])
def test_qr_scales(gn, H, scale):
    """1e140: the sums of squares pass 1e280, where the scalars leave the fast
    form; 1e-200 and 1e-300: they underflow, as for any unscaled Householder QR,
    so only R's size is asked for above 1e-150."""
    torch.manual_seed(5)
    C = torch.randn(150, 60, dtype=torch.float64, device="cuda") * scale
    Q, R = qr(gn, H, C)
    if scale > 1e-150:
        check(C, Q, R)
    assert bool(Q.isfinite().all()) and bool(R.isfinite().all())
    assert H.sync_status() == 0


def test_qr_dropped_columns(gn, H):
    """Zero columns and a column whose tail is zero: H = I, R's entry is that of C."""
    torch.manual_seed(6)
    C = torch.randn(200, 70, dtype=torch.float64, device="cuda")
    C[:, 0] = 0.0
    C[:, 31:34] = 0.0
    C[:, 50] = C[:, 49]
    Q, R = qr(gn, H, C)
    check(C, Q, R)
    D = torch.diag(torch.arange(1.0, 41.0, dtype=torch.float64, device="cuda"))
    D = torch.cat([D, torch.zeros(9, 40, dtype=torch.float64, device="cuda")])
    Q, R = qr(gn, H, D)
    assert torch.equal(R, D[:40]) and torch.equal(Q, (D != 0).double())
    assert H.sync_status() == 0
