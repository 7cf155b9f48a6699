"""That the K parts of the tensor-core sketches and the clusters of the batched cores run where
they are meant to, and are exact where their inputs are integers."""
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


@pytest.mark.parametrize("m,n,r,l", [(9001, 300, 33, 8), (300, 9001, 17, 4), (1500, 7000, 1, 1), (20000, 1200, 300, 150)])
@pytest.mark.parametrize("dtype", ["bf16", "e4m3"])
def test_sketch_parts_need_their_room(gn, H, m, n, r, l, dtype):
    """With the workspace asked for, K parts and the launch that sums them; with the operands'
    own scratch only (the scale images of e4m3), one launch for both products."""
    g = torch.Generator(device="cuda").manual_seed(m + r)
    ints = lambda a, b: torch.randint(-2, 3, (a, b), generator=g, device="cuda").float()
    A, X, Y = ints(m, n), ints(n, r), ints(m, r + l)
    t = lambda k: (k + 127) // 128
    if dtype == "e4m3":
        a, x, y, code = H.quantize_e4m3(A), H.quantize_e4m3(X, data=False), H.quantize_e4m3(Y, data=False), gn.E4M3
        least = 512 * (t(m) * t(n) + t(n) * t(r) + t(m) * t(r + l)) + 1024
        images = 3
    else:
        a, x, y, code = H.quantize(A), H.quantize(X), H.quantize(Y), gn.BF16
        least, images = 256, 0
    ws = H.workspace(m, n, r, l, code)
    assert ws.numel() > least
    for room, launches in ((ws, images + 2), (ws[:least], images + 1)):
        AX = torch.empty(m, r, device="cuda")
        YtA = torch.empty(r + l, n, device="cuda")
        before = gn.kernel_launches()
        H.sketch(a, x, y, AX, YtA, room)
        assert gn.kernel_launches() - before == launches
        assert H.sync_status() == 0
        assert torch.equal(AX.double(), A.double() @ X.double())   # sums below 2^24: exact in any order
        assert torch.equal(YtA.double(), Y.double().T @ A.double())


def problem(gn, m, n, r, l, g):
    d = {}
    for name, a, b in (("A", m, n), ("X", n, r), ("Y", m, r + l)):
        d[name] = gn.padded(a, b, torch.bfloat16, "cuda")
        d[name].copy_(torch.randint(-2, 3, (a, b), generator=g, device="cuda"))
    e = lambda a, b, t: torch.full((a, b), float("nan"), dtype=t, device="cuda")
    d.update(AX=e(m, r, torch.float32), YtA=e(r + l, n, torch.float32), Q=e(r + l, r, torch.float64),
             R=e(r, r, torch.float64), Q2=e(r, r, torch.float64), R2=e(r, r, torch.float64),
             k=torch.full((1,), -1, dtype=torch.int32, device="cuda"))
    return d


SHAPES = [(1, 1), (2, 1), (5, 30), (31, 1), (32, 1), (33, 16), (64, 32), (65, 1), (96, 96), (97, 48), (127, 1), (128, 64)]


@pytest.mark.parametrize("copies", [1, 40])   # 40 x 12 problems: one CTA per core
def test_batched_cores_are_backward_stable(gn, copies):
    """Integer sketches: the cores C = Y^T A X are exact, so Q R = C and Q_2 R_2 = R_1^T hold to
    the backward error of Householder QR.  A reflector's application to a column rounds a dot of
    M terms, its coefficient (from a norm of M squares, a sum and a reciprocal) and the update:
    2 M + 10 times 2^-53 of the column's norm; N of them factor it and N form Q."""
    bound = lambda M, N: 2 * N * (2 * M + 10) * 2.0 ** -53
    H = gn.Handle()
    g = torch.Generator(device="cuda").manual_seed(7)
    probs = [problem(gn, 256, 200, r, l, g) for r, l in SHAPES]
    rest = [problem(gn, 200, 160, 128, 64, g) for _ in range((copies - 1) * len(SHAPES))]
    ws = H.batched_prepare(probs + rest)
    truncated = 0
    for eps in (1e-10, 0.3):   # nothing below the first; a truncation and its second QR with the other
        H.batched_run(eps, gn.SGN | gn.EPS_RELATIVE, ws)
        assert H.sync_status() == 0
        for (r, l), p in zip(SHAPES, probs):
            A, X, Y = (p[k].double() for k in ("A", "X", "Y"))
            C = Y.T @ A @ X
            assert float((p["Q"] @ p["R"] - C).norm()) <= bound(r + l, r) * float(C.norm())
            k = int(p["k"])
            if 0 < k < r:
                truncated += 1
                R1, Q2, R2 = p["R"][:k], p["Q2"][:, :k], p["R2"][:k, :k]
                assert float((Q2 @ R2 - R1.T).norm()) <= bound(r, k) * float(R1.norm())
    assert truncated > 0
    H.close()
