"""The triangular solves of gn_factors and gn_apply are backward stable: the residual
F R - AX stays at the rounding of a substitution whatever the condition of R's diagonal
blocks."""
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


def upper(kind, k, rn):
    """Upper triangular matrices whose diagonal blocks have ill-conditioned inverses."""
    eye = torch.eye(k, dtype=torch.float64, device="cuda")
    if kind == "graded":   # the R of a core whose spectrum decays over 1e16
        s = torch.logspace(0, -16, k, dtype=torch.float64, device="cuda")
        R = torch.linalg.qr((rn(k + k // 2, k) * s) @ rn(k, k))[1]
        return R * torch.sign(torch.diagonal(R))[:, None]
    if kind == "kahan":    # diag(s^i) (I - c N), condition 1e14 or more
        c = 0.285 * 256 / max(k, 256)
        s = (1 - c * c) ** 0.5
        return torch.pow(s, torch.arange(k, device="cuda").double())[:, None] * (eye - c * torch.triu(torch.ones_like(eye), 1))
    return eye + 0.3 * torch.triu(rn(k, k), 1)   # unit triangular


def backward(F, R, B, rows):
    """max over sampled rows of |F R - B| / (|F| |R|), the componentwise backward error."""
    f, r, b = (t.cpu().numpy().astype(np.longdouble) for t in (F[rows], R, B[rows].double()))
    return float((np.abs(f @ r - b) / np.maximum(np.abs(f) @ np.abs(r), np.longdouble(1e-300))).max())


# one and two blocks of 128 columns, ragged ones; rows on the FP64 units, on either side of
# the line between base blocks of 128 and of 32 columns, and with digit-sliced products
SIZES = [(64, 256), (3000, 200), (2000, 257), (8192, 300), (8193, 300), (8300, 129)]


@pytest.mark.parametrize("kind,m,k,trans", [(kind, m, k, 0) for kind in ("graded", "kahan", "unit") for m, k in SIZES] +
                         [(kind, m, k, 1) for kind in ("graded", "kahan", "unit") for m, k in SIZES])
def test_solve_is_backward_stable(gn, H, kind, m, k, trans):
    g = torch.Generator(device="cuda").manual_seed(k + m)
    rn = lambda a, b: torch.randn(a, b, generator=g, device="cuda", dtype=torch.float64)
    n, l, r = 40, 3, k + trans
    core = gn.Core.empty(r, l, "cuda")
    core.Q.copy_(rn(r + l, r))
    core.k = k
    R = upper(kind, k, rn)
    if trans:   # F = (AX Q_2) R_2^-T over the first k columns, Q_2 the identity
        core.Q2.zero_()
        core.Q2[:k, :k] = torch.eye(k, dtype=torch.float64, device="cuda")
        core.R2.zero_()
        core.R2[:k, :k] = R
        core.sgn = 1
    else:
        core.R.copy_(R)
    T = R.T if trans else R
    AX = torch.zeros(m, r, dtype=torch.float64, device="cuda")
    AX[:, :k] = rn(m, k) @ T
    F = torch.empty(m, r, dtype=torch.float64, device="cuda")
    G = torch.empty(r, n, dtype=torch.float64, device="cuda")
    big = max(m, n, k) + r + l
    H.factors(AX, rn(r + l, n), core, F, G, H.workspace(big, big, r, l, gn.F64))
    assert H.sync_status() == 0
    rows = torch.linspace(0, m - 1, 24, device="cuda").long()
    # substitution: (k + 4) u |F||R| (reciprocal pivots cost 4 u); the products' own error is below it
    assert backward(F[:, :k], T, AX[:, :k], rows) <= (k + 4) * 2.0 ** -53


@pytest.mark.parametrize("kind", ["graded", "kahan", "unit"])
@pytest.mark.parametrize("side", [0, 1])
def test_apply_solves_by_substitution(gn, H, kind, side):
    """A_hat W through the core against the same solve in plain FP64: R X = Q^T B with
    every other factor the identity, so that the output is the solution itself."""
    k, l, kw = 256, 4, 24
    g = torch.Generator(device="cuda").manual_seed(11)
    rn = lambda a, b: torch.randn(a, b, generator=g, device="cuda", dtype=torch.float64)
    core = gn.Core.empty(k, l, "cuda")
    eye = torch.eye(k + l, dtype=torch.float64, device="cuda")
    core.R.copy_(upper(kind, k, rn))
    core.Q.copy_(eye[:, :k])
    core.k = k
    AX, YtA = eye[:k, :k].contiguous(), eye
    if side == 0:      # out = R^-1 W[:k]
        W = torch.zeros(k + l, kw, dtype=torch.float64, device="cuda")
        W[:k] = core.R @ rn(k, kw)
        out = H.apply(AX, YtA, core, W, side=0)
        F, T, B = out.T, core.R.T, W[:k].T
    else:              # out[:, :k] = W R^-1
        W = rn(kw, k) @ core.R
        F, T, B = H.apply(AX, YtA, core, W, side=1)[:, :k], core.R, W
    assert H.sync_status() == 0
    assert backward(F, T, B, torch.arange(kw, device="cuda")) <= (k + 4) * 2.0 ** -53


@pytest.mark.parametrize("m", [1, 700, 1023])
def test_short_fp32_sketches_stay_on_the_fp64_units(gn, H, m):
    """F = (AX Q_2) R_2^-T with R_2 the identity: AX Q_2 entry by entry, with a column of AX
    1e10 times the others that Q_2 leaves out."""
    n, l, r, k = 40, 3, 300, 200
    g = torch.Generator(device="cuda").manual_seed(m)
    rn = lambda a, b: torch.randn(a, b, generator=g, device="cuda", dtype=torch.float64)
    core = gn.Core.empty(r, l, "cuda")
    core.Q.copy_(rn(r + l, r))
    core.Q2.copy_(rn(r, r))
    core.Q2[0] = 0.0
    core.R2.copy_(torch.eye(r, dtype=torch.float64, device="cuda"))
    core.k, core.sgn = k, 1
    AX = rn(m, r).float()
    AX[:, 0] = 1e10
    F = torch.empty(m, r, dtype=torch.float64, device="cuda")
    G = torch.empty(r, n, dtype=torch.float64, device="cuda")
    H.factors(AX, rn(r + l, n).float(), core, F, G, H.workspace(max(m, 2 * r), 2 * r, r, l, gn.BF16))
    assert H.sync_status() == 0
    a, q = AX.cpu().numpy().astype(np.longdouble), core.Q2[:, :k].cpu().numpy().astype(np.longdouble)
    err = np.abs(F[:, :k].cpu().numpy() - a[:, 1:] @ q[1:])
    assert np.all(err <= (r + 4) * 2.0 ** -53 * (np.abs(a[:, 1:]) @ np.abs(q[1:])))   # r u |AX||Q_2|


# base blocks of 128 and of 32 columns; FP32 sketches (eight digits) and FP64 ones (nine)
@pytest.mark.parametrize("m,r", [(3000, 256), (9000, 700), (40000, 300)])
@pytest.mark.parametrize("f64", [False, True])
def test_every_accepted_workspace_gives_the_same_factors(gn, H, m, r, f64):
    """From the smallest workspace that gn_factors takes up to gn_workspace_size: fewer rows at
    a time, or the FP64 units, with the residual of a substitution each time."""
    n, l = 60, 8
    g = torch.Generator(device="cuda").manual_seed(r)
    rn = lambda a, b: torch.randn(a, b, generator=g, device="cuda", dtype=torch.float64)
    core = gn.Core.empty(r, l, "cuda")
    core.R.copy_(torch.triu(rn(r, r), 1) / r ** 0.5 + torch.eye(r, dtype=torch.float64, device="cuda"))
    core.Q.copy_(rn(r + l, r))
    core.k = r
    dt = torch.float64 if f64 else torch.float32
    AX, YtA = rn(m, r).to(dt), rn(r + l, n).to(dt)
    full = H.workspace_bytes(m, 2 * r, r, l, gn.F64 if f64 else gn.BF16)
    buf = torch.empty(full, dtype=torch.uint8, device="cuda")
    rows = torch.linspace(0, m - 1, 16, device="cuda").long()

    def run(nbytes):
        F = torch.empty(m, r, dtype=torch.float64, device="cuda")
        G = torch.empty(r, n, dtype=torch.float64, device="cuda")
        H.factors(AX, YtA, core, F, G, buf[:nbytes])
        assert H.sync_status() == 0
        return F
    lo, need = 0, full   # run(lo) is refused, run(need) is not
    while need - lo > 256:
        mid = (lo + need) // 2
        try:
            run(mid)
            need = mid
        except gn.GNError as e:
            assert e.status == 4
            lo = mid
    assert need < full
    # eight digits: a window of 2^-56 below the largest entries of a row and a column, K <= 512
    tol = (r + 4) * 2.0 ** -53 + (0 if f64 else 512 ** 0.5 * 2.0 ** -52)
    for nbytes in (need, need + (full - need) // 5, (need + full) // 2, full):
        assert backward(run(nbytes), core.R, AX, rows) <= tol


def test_workspace_size_asks_for_what_the_factors_take(gn, H):
    """At a shape whose largest call is the factors', the smallest size that solves all rows
    together is the one asked for: it was 0.7 GB more at 32768 x 16384, r = 1000."""
    m, n, r, l = 32768, 16384, 1000, 500
    assert H.workspace_bytes(m, n, r, l, gn.BF16) <= 1.3e9
