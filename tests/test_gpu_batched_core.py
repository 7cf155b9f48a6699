"""The batched cores at the edges of their row split over four CTAs and of their
32-column lane groups, against the unbatched core."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gn():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2009_11392_gb300 as g
    return g


def problem(gn, m, n, r, l, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    d = {}
    for name, a, b in (("A", m, n), ("X", n, r), ("Y", m, r + l)):
        d[name] = gn.padded(a, b, torch.bfloat16, "cuda")
        d[name].copy_(torch.randn(a, b, generator=g, device="cuda"))
    e = lambda a, b, t: torch.full((a, b), float("nan"), dtype=t, device="cuda")
    d.update(AX=e(m, r, torch.float32), YtA=e(r + l, n, torch.float32), Q=e(r + l, r, torch.float64),
             R=e(r, r, torch.float64), Q2=e(r, r, torch.float64), R2=e(r, r, torch.float64),
             k=torch.full((1,), -1, dtype=torch.int32, device="cuda"))
    return d


# one column; fewer rows than CTAs x warps; around 32, 64, 96, 128 columns; 192 rows
SHAPES = [(1, 1), (1, 3), (2, 1), (3, 2), (5, 30), (31, 1), (32, 1), (33, 16), (63, 2), (64, 32), (65, 1), (96, 96),
          (97, 48), (127, 1), (128, 1), (128, 64)]


@pytest.mark.parametrize("copies", [1, 40])   # 40 x 16 problems: one CTA per core
def test_cores(gn, copies):
    H = gn.Handle()
    probs = [problem(gn, 256, 200, r, l, 10 + i) for i, (r, l) in enumerate(SHAPES)]
    rest = [problem(gn, 200, 160, 128, 64, 99) for _ in range((copies - 1) * len(SHAPES))]
    ws = H.batched_prepare(probs + rest)
    H.batched_run(1e-10, gn.AUTO | gn.EPS_RELATIVE, ws)
    assert H.sync_status() == 0
    for (r, l), p in zip(SHAPES, probs):
        core = gn.Core.empty(r, l, "cuda")
        cws = H.workspace(256, 200, r, l, gn.BF16)
        H.core(p["YtA"], p["X"], 1e-10, gn.AUTO | gn.EPS_RELATIVE, core, cws)
        assert int(p["k"]) == core.k == r
        # Gaussian cores: condition numbers below 1e4 (square ones the largest), C equal
        # to FP32-accumulated slices on both sides
        eye = torch.eye(r, dtype=torch.float64, device="cuda")
        assert float((p["Q"].T @ p["Q"] - eye).norm()) <= 2e-13
        C = core.Q @ core.R
        assert float((p["Q"] @ p["R"] - C).norm() / C.norm()) <= 1e-5
        assert torch.equal(p["R"], torch.triu(p["R"])) and bool((torch.diagonal(p["R"]) >= 0).all())
    H.close()
