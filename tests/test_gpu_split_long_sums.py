"""Split products over more than 1024 terms that all have one sign and lie near the power-of-two bounds: their sum does
not fit 64 bits in units of 2^-53 of the scale."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def plan(lib):
    p = lib.rpcholqr_plan_create(0, 4096, 2048, 2048, mode=lib.SPLIT64)
    yield p
    p.close()


@pytest.mark.parametrize("K", [1024, 1025, 1500, 2048])
@pytest.mark.parametrize("v", [0.99, 1.0 - 2.0 ** -53, -(1.0 - 2.0 ** -53)])
def test_sums_near_the_bounds(lib, plan, K, v):
    m, N = 300, 70
    X = torch.full((m, K), v, dtype=torch.float64, device="cuda")
    Y = torch.full((K, N), abs(v), dtype=torch.float64, device="cuda")
    X[5, :] = 0.25 * X[6, :]
    Y[:, 3] = -0.5 * Y[:, 4]
    want = X[:, :1] * Y[:1, :] * K
    # scale 1 (less in row 5 and column 3): per term the dropped digit pairs 6 2^-56 and each operand's rounding 2^-56, per
    # window of 128 half a unit of 2^-53, the result and `want` an ulp each
    tol = K * 9 * 2.0 ** -56 + 16 * 2.0 ** -54 + K * 2.0 ** -51
    C, info = lib.rpcholqr_ozaki_gemm(plan, X, Y)
    assert info.cpu().tolist() == [0, -1]
    assert float((C - want).abs().max()) <= tol
    B = torch.full((m, N), 3.0, dtype=torch.float64, device="cuda")
    C, info = lib.rpcholqr_ozaki_update(plan, X, Y, B)
    assert info.cpu().tolist() == [0, -1]
    assert float((C - (B - want)).abs().max()) <= tol
