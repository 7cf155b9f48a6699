"""bf16 quantization of more rows or columns than 32 bits count."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols", [(1, 2 ** 31 + 9), (2 ** 31 + 3, 1)])
def test_more_than_2_31(rows, cols):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2009_11392_gb300 as gn
    need = 4 * rows * cols + 2 * rows * (cols + 8)
    if torch.cuda.mem_get_info()[0] < need + (8 << 30):
        pytest.skip("not enough device memory")
    H = gn.Handle()
    A = torch.zeros(rows, cols, device="cuda")
    at = torch.tensor([0, 1, 2 ** 30 - 1, 2 ** 30, 2 ** 30 + 7, 2 ** 31 - 1, 2 ** 31, rows * cols - 1], device="cuda")
    flat = A.view(-1)
    flat[at] = torch.arange(1.0, 9.0, device="cuda") / 3
    hi = H.quantize(A)
    assert H.sync_status() == 0
    got = hi[0, at] if rows == 1 else hi[at, 0]
    assert torch.equal(got, flat[at].bfloat16())
    # all eight in the one column; of the last 64 columns 2^31 - 1, 2^31 and the last
    assert int(torch.count_nonzero(hi[:, :1] if cols == 1 else hi[:, -64:])) == (8 if cols == 1 else 3)
    H.close()
    del A, flat, hi
    torch.cuda.empty_cache()
