"""GPU test of the FP32 mode's one-row-per-thread solve (up to 16 columns): widths around its edges and around whole 16-byte
groups, row counts around a CTA, rows that are not 16-byte aligned, at the FP32 target of the mode (1e-5)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 7, 8, 9, 12, 15, 16, 17])
@pytest.mark.parametrize("m,pad,shift", [(255, 0, 0), (256, 3, 1), (257, 4, 0), (4097, 4, 2), (100003, 0, 0)])
def test_factor_f32_narrow(lib, n, m, pad, shift):
    g = torch.Generator(device="cuda").manual_seed(100 * n + m)
    ld = n + pad
    flat = torch.randn(m * ld + shift, generator=g, device="cuda")     # shift: rows off every 16-byte boundary
    A = flat[shift:].view(m, ld)[:, :n]
    out = torch.full((m * ld + shift,), 7.0, device="cuda")
    Qv = out[shift:].view(m, ld)
    plan = lib.rpcholqr_plan_create(0, m, n, 3 * n, mode=lib.FP32)
    try:
        Q, R, info = lib.rpcholqr_factor_f32(plan, A, 3 * n, 3, Q=Qv[:, :n])
        assert info.cpu().tolist() == [0, -1]
        Qd, Rd, Ad = Q.double(), R.double(), A.double()
        assert float((Qd.T @ Qd - torch.eye(n, dtype=torch.float64, device="cuda")).abs().max()) <= 1e-5
        assert float(torch.linalg.norm(Ad - Qd @ Rd) / torch.linalg.norm(Ad)) <= 1e-5
        assert bool((Qv[:, n:] == 7.0).all()) and bool((out[:shift] == 7.0).all())     # nothing beside the matrix
        flat[shift:].view(m, ld)[m - 1, n - 1] = float("inf")
        assert lib.rpcholqr_factor_f32(plan, A, 3 * n, 3)[2].cpu().tolist()[0] == lib.ERR_NONFINITE
    finally:
        plan.close()
