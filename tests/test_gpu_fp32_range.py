"""FP32 mode on rows far heavier than the sampled ones: Gram sums beyond the largest FP32 number, each 256 rows' within it."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("power", [-60, -67, -68])
def test_heavy_rows_outside_the_sample(lib, power):
    m, n, s, seed = 1 << 19, 16, 48, 5
    g = torch.Generator(device="cuda").manual_seed(1)
    A = torch.randn(m, n, generator=g, device="cuda", dtype=torch.float32)
    A[lib.rpcholqr_sample_indices(seed, m, s).long()] *= 2.0 ** power
    plan = lib.rpcholqr_plan_create(0, m, n, s, mode=lib.FP32)
    try:
        Q, R, info = lib.rpcholqr_factor_f32(plan, A, s, seed)
        assert info.cpu().tolist() == [0, -1]
        Qd = Q.double()
        # Q is A_1 R_1^{-1} with both rounded to FP32 and kappa(A_1) < 10: n u kappa for each
        tol = 2 * 16 * 2.0 ** -24 * 10
        assert float(torch.linalg.matrix_norm(Qd.T @ Qd - torch.eye(n, dtype=torch.float64, device="cuda"), 2)) <= tol
        assert float((Qd @ R.double() - A.double()).norm() / A.double().norm()) <= tol
    finally:
        plan.close()
