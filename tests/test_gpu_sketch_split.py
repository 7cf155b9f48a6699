"""The tensor-core sketches where their K ranges run in parts (few long chains), on
integers that are exact in FP32, with and without room for the parts; and the bf16
quantization's aligned and unaligned rows."""
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


# long K of Y^T A, of AX, of both; one row or column past a tile; outputs of 1, 15,
# 17 and 33 columns; odd leading dimensions
@pytest.mark.parametrize("m,n,r,l", [(9001, 300, 33, 8), (300, 9001, 17, 4), (2049, 1025, 15, 2), (1500, 7000, 1, 1),
                                     (20000, 1200, 300, 150), (640, 5000, 128, 64)])
@pytest.mark.parametrize("dtype", ["bf16", "split", "e4m3"])
@pytest.mark.parametrize("room", [True, False])
def test_sketch_parts_exact(gn, H, m, n, r, l, dtype, room):
    """Entries in {-2 .. 2}: sums of at most 20000 products stay below 2^24, so every
    order of additions gives the integer itself."""
    g = torch.Generator(device="cuda").manual_seed(m + r)
    ints = lambda a, b: torch.randint(-2, 3, (a, b), generator=g, device="cuda").float()
    A, X, Y = ints(m, n), ints(n, r), ints(m, r + l)
    lo = None
    if dtype == "e4m3":
        a, x, y, code = H.quantize_e4m3(A), H.quantize_e4m3(X, data=False), H.quantize_e4m3(Y, data=False), gn.E4M3
    else:
        a, x, y, code = H.quantize(A), H.quantize(X), H.quantize(Y), gn.BF16
        if dtype == "split":
            lo = torch.zeros_like(a.new_empty(m, a.stride(0)))[:, :n]
            lo.copy_((A / 256).bfloat16())   # A + A / 256: still exact, the second source is read
            A = A + A / 256
            code = gn.BF16X2
    AX = torch.empty(m, r, device="cuda")
    YtA = torch.empty(r + l, n, device="cuda")
    ws = H.workspace(m, n, r, l, code)
    if not room and dtype != "e4m3":
        ws = ws[:256]
    H.sketch(a, x, y, AX, YtA, ws, A_lo=lo)
    assert H.sync_status() == 0
    assert torch.equal(AX.double(), A.double() @ X.double())
    assert torch.equal(YtA.double(), Y.double().T @ A.double())


@pytest.mark.parametrize("rows,cols", [(1, 1), (3, 7), (5, 255), (4, 257), (2, 1000), (300, 33)])
@pytest.mark.parametrize("src", [torch.float32, torch.float64])
@pytest.mark.parametrize("pad", [0, 1, 4])
def test_quantize_rows(gn, H, rows, cols, src, pad):
    """Rows that start on and off 16-byte boundaries."""
    torch.manual_seed(rows * cols)
    wide = torch.randn(rows, cols + pad, dtype=src, device="cuda") * 10
    A = wide[:, pad:] if pad == 1 else wide[:, :cols]
    x32 = A.float()
    hi, lo = H.quantize(A, split=True)
    assert torch.equal(hi, x32.bfloat16())
    assert torch.equal(lo, (x32 - hi.float()).bfloat16())
    assert torch.equal(H.quantize(A), hi)
    assert H.sync_status() == 0
