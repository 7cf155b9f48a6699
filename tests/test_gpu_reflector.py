"""The reflector's two scalars (a square root and a reciprocal from single-precision estimates)
through cores of one column, where R is the norm and Q the normalised column, over the exponents
on either side of the range in which they are taken that way."""
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


def column(gn, C):
    H = gn.Handle()
    M = C.shape[0]
    core = gn.Core.empty(1, M - 1, "cuda")
    core.C.copy_(torch.tensor(C, device="cuda"))
    n = 4
    YtA = torch.zeros(M, n, dtype=torch.float64, device="cuda")
    X = torch.zeros(n, 1, dtype=torch.float64, device="cuda")
    ws = H.workspace(M + 1, M + 1, 1, M - 1, gn.F64)
    H.core(YtA, X, 0.0, gn.PLAIN | gn.CORE_C_GIVEN, core, ws)
    assert H.sync_status() == 0
    out = float(core.R), core.Q.cpu().numpy()
    H.close()
    return out


# ||C||^2 has exponent about 2 e: -900 and 900 are where sqrt and division take over
@pytest.mark.parametrize("e", [-460, -452, -451, -450, -449, -448, -300, -1, 0, 1, 300, 447, 448, 449, 450, 451, 460])
@pytest.mark.parametrize("M", [2, 3, 50])
def test_norm_and_normalised_column(gn, e, M):
    rng = np.random.default_rng(e + 1000 * M)
    for sign in (1.0, -1.0):
        c = rng.standard_normal(M)
        c[0] = sign * abs(c[0])
        C = (c * 2.0 ** e)[:, None]
        R, Q = column(gn, C)
        norm = np.sqrt((c.astype(np.longdouble) ** 2).sum())
        # M roundings of the sum of squares, halved by the root, and the root's own two
        assert abs(R * 2.0 ** -e - norm) <= (M / 2 + 3) * 2.0 ** -53 * norm
        assert np.abs(Q[:, 0] - (c / norm).astype(np.float64)).max() <= (M + 12) * 2.0 ** -53


@pytest.mark.parametrize("e", [-440, -100, 0, 77, 440])
def test_pythagorean_norms_are_exact_to_two_ulp(gn, e):
    """3^2 + 4^2, 5^2 + 12^2, 20^2 + 21^2, ... squares and their sums exact in FP64."""
    for a, b, h in ((3, 4, 5), (12, 5, 13), (-20, 21, 29), (-8, -15, 17), (696, -697, 985)):
        R, _ = column(gn, np.array([[a * 2.0 ** e], [b * 2.0 ** e]]))
        assert abs(R - h * 2.0 ** e) <= 2 * np.spacing(h * 2.0 ** e)
