"""The factors' and apply's triangular solves at the edges of their 128-column
blocks, against a plain FP64 solve."""
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


def state(gn, m, n, r, l, dtype, seed=0):
    """Sketches and a core with a well-conditioned R (unit diagonal up to a
    factor 2, off-diagonal N(0, 1 / r))."""
    g = torch.Generator(device="cuda").manual_seed(seed + r)
    rn = lambda a, b: torch.randn(a, b, generator=g, device="cuda", dtype=torch.float64)
    core = gn.Core.empty(r, l, "cuda")
    core.R.copy_(torch.triu(rn(r, r), 1) / r ** 0.5 + torch.diag(1 + torch.rand(r, generator=g, device="cuda", dtype=torch.float64)))
    core.Q.copy_(rn(r + l, r) / (r + l) ** 0.5)
    core.k = r
    return rn(m, r).to(dtype), rn(r + l, n).to(dtype), core, rn


def close(a, b, tol):
    return float((a - b).norm() / b.norm()) <= tol


# 33: the first size off one 32-column substitution; 128 / 129 / 256: block edges;
# 4200: more columns than one product slices (K > 4096)
@pytest.mark.parametrize("m,r", [(700, 33), (1, 64), (700, 128), (129, 129), (33000, 40), (300, 256), (2100, 383),
                                 (260, 4200)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_factors_solve(gn, H, m, r, dtype):
    n, l = 50, 3
    AX, YtA, core, _ = state(gn, m, n, r, l, dtype)
    F = torch.empty(m, r, dtype=torch.float64, device="cuda")
    G = torch.empty(r, n, dtype=torch.float64, device="cuda")
    big = max(m, n, r) + r + l
    ws = H.workspace(big, big, r, l, gn.BF16 if dtype == torch.float32 else gn.F64)
    H.factors(AX, YtA, core, F, G, ws)
    assert H.sync_status() == 0
    ref = torch.linalg.solve_triangular(core.R, AX.double(), upper=True, left=False)
    # R's condition number is below 10 r^1/2: r u 10 r^1/2 stays under 1e-10 at r = 4200
    assert close(F, ref, 1e-12 if r < 1000 else 1e-10)


@pytest.mark.parametrize("r", [20, 33, 129, 300, 4200])
@pytest.mark.parametrize("kw", [1, 64])
@pytest.mark.parametrize("side", [0, 1])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_apply_solve(gn, H, r, kw, side, dtype):
    m, n, l = 90, 70, 5
    AX, YtA, core, rn = state(gn, m, n, r, l, dtype)
    W = rn(n, kw) if side == 0 else rn(kw, m)
    out = H.apply(AX, YtA, core, W, side=side)
    assert H.sync_status() == 0
    AX, YtA = AX.double(), YtA.double()
    if side == 0:
        ref = AX @ torch.linalg.solve_triangular(core.R, core.Q.T @ (YtA @ W), upper=True)
    else:
        ref = torch.linalg.solve_triangular(core.R, W @ AX, upper=True, left=False) @ core.Q.T @ YtA
    assert close(out, ref, 1e-12 if r < 1000 else 1e-10)


@pytest.mark.parametrize("side", [0, 1])
def test_truncated_core_uses_the_second_factor(gn, H, side):
    """k < r: F = AX Q_2 R_2^{-T}, the solve from the last block back."""
    m, n, r, l, k, kw = 500, 60, 300, 7, 200, 5
    AX, YtA, core, rn = state(gn, m, n, r, l, torch.float64, seed=1)
    core.Q2.copy_(rn(r, r) / r ** 0.5)
    core.R2.copy_(core.R)
    core.k, core.sgn = k, 1
    W = rn(n, kw) if side == 0 else rn(kw, m)
    out = H.apply(AX, YtA, core, W, side=side)
    F = torch.empty(m, r, dtype=torch.float64, device="cuda")
    G = torch.empty(r, n, dtype=torch.float64, device="cuda")
    H.factors(AX, YtA, core, F, G, H.workspace(m, max(n, r + 1), r, l, gn.F64))
    assert H.sync_status() == 0
    Fr = torch.linalg.solve_triangular(core.R2[:k, :k].T, AX @ core.Q2[:, :k], upper=False, left=False)
    Gr = core.Q[:, :k].T @ YtA
    assert close(F[:, :k], Fr, 1e-12) and close(G[:k], Gr, 1e-12)
    assert close(out, Fr @ (Gr @ W) if side == 0 else (W @ Fr) @ Gr, 1e-12)


def test_small_workspaces_solve_in_row_groups(gn, H):
    """A workspace that holds fewer rows' slices gives the same F, bit for bit
    (every row is solved by itself)."""
    m, n, r, l = 3000, 900, 256, 8
    AX, YtA, core, _ = state(gn, m, n, r, l, torch.float32)
    out = []
    for ws_bytes in (H.workspace_bytes(m, n, r, l, gn.BF16), H.workspace_bytes(m, n, r, l, gn.BF16) * 55 // 100):
        F = torch.empty(m, r, dtype=torch.float64, device="cuda")
        G = torch.empty(r, n, dtype=torch.float64, device="cuda")
        try:
            H.factors(AX, YtA, core, F, G, torch.empty(ws_bytes, dtype=torch.uint8, device="cuda"))
        except gn.GNError as e:
            assert e.status == 4   # below what the call asks for
            continue
        out.append(F)
    assert H.sync_status() == 0
    assert all(torch.equal(out[0], f) for f in out[1:])


def test_zero_pivot_leaves_the_columns_before_it(gn, H):
    m, n, r, l = 300, 40, 200, 4
    AX, YtA, core, _ = state(gn, m, n, r, l, torch.float64)
    core.R[150, 150] = 0.0
    F = torch.empty(m, r, dtype=torch.float64, device="cuda")
    G = torch.empty(r, n, dtype=torch.float64, device="cuda")
    H.factors(AX, YtA, core, F, G, H.workspace(m, r + 1, r, l, gn.F64))
    assert H.sync_status() == 0
    ref = torch.linalg.solve_triangular(core.R[:150, :150], AX[:, :150], upper=True, left=False)
    assert close(F[:, :150], ref, 1e-12)
    assert not bool(F[:, 150].isfinite().any())


# 256-column blocks: on both sides of the line where they begin (m >= 8192, m r^2 >= 4e9);
# a last block of one column, of one half, of one half and a column, of both; more rows
# than one pass takes (32768)
@pytest.mark.parametrize("m,r", [(8191, 700), (8192, 698), (8192, 700), (8193, 768), (8200, 769), (8192, 770),
                                 (8192, 896), (8195, 897), (8192, 898), (9000, 1000), (33000, 350)])
@pytest.mark.parametrize("trans", [0, 1])
def test_wide_blocks(gn, H, m, r, trans):
    n, l = 40, 3
    AX, YtA, core, rn = state(gn, m, n, r, l, torch.float32 if m % 2 else torch.float64)
    ws = H.workspace(m, max(n, r + l + 1), r, l, gn.F64)
    k = r
    ref = AX.double()
    if trans:   # F = AX Q_2 R_2^-T over the first k columns
        k = r - 1
        core.Q2.copy_(rn(r, r) / r ** 0.5)
        core.R2.copy_(core.R)
        core.k, core.sgn = k, 1
        ref = torch.linalg.solve_triangular(core.R2[:k, :k].T, ref @ core.Q2[:, :k], upper=False, left=False)
    else:
        ref = torch.linalg.solve_triangular(core.R, ref, upper=True, left=False)
    F = torch.empty(m, r, dtype=torch.float64, device="cuda")
    G = torch.empty(r, n, dtype=torch.float64, device="cuda")
    H.factors(AX, YtA, core, F, G, ws)
    assert H.sync_status() == 0
    # R's condition number is below 10 r^1/2: r u 10 r^1/2 stays under 1e-10 at r = 1000
    assert close(F[:, :k], ref, 1e-12 if r < 1000 else 1e-10)
