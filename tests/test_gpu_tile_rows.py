"""Sketches around the line between 128- and 256-row tiles, where the launch has fewer
than four tall tiles per SM, on integers that are exact in FP32."""
import pytest
import torch

pytestmark = pytest.mark.gpu


# outputs that end one row into a tall tile or one row short of it, ragged last column
# tiles, a remainder of the K blocks; the last two below the line
@pytest.mark.parametrize("m,n,r,l", [(16384, 8192, 500, 250), (16385, 8191, 500, 250), (8193, 8447, 511, 129),
                                     (8192, 4100, 300, 150), (4097, 2049, 64, 32)])
@pytest.mark.parametrize("dtype", ["bf16", "e4m3"])
def test_sketch_tile_rows_exact(m, n, r, l, dtype):
    """Entries in {-2 .. 2}: sums of at most 16385 products stay below 2^24, so every
    order of additions gives the integer itself."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2009_11392_gb300 as gn
    H = gn.Handle()
    g = torch.Generator(device="cuda").manual_seed(m + r)
    ints = lambda a, b: torch.randint(-2, 3, (a, b), generator=g, device="cuda").float()
    A, X, Y = ints(m, n), ints(n, r), ints(m, r + l)
    if dtype == "e4m3":
        a, x, y, code = H.quantize_e4m3(A), H.quantize_e4m3(X, data=False), H.quantize_e4m3(Y, data=False), gn.E4M3
    else:
        a, x, y, code = H.quantize(A), H.quantize(X), H.quantize(Y), gn.BF16
    AX = torch.full((m, r), float("nan"), device="cuda")
    YtA = torch.full((r + l, n), float("nan"), device="cuda")
    H.sketch(a, x, y, AX, YtA, H.workspace(m, n, r, l, code))
    assert H.sync_status() == 0
    assert torch.equal(AX.double(), A.double() @ X.double())
    assert torch.equal(YtA.double(), Y.double().T @ A.double())
