"""GPU test of the FP32 mode over the row solve's panel heights (32, 64 and 128 rows, chosen by the row count and the
width), ragged widths, and rows that are not 16-byte aligned, at the FP32 target of the mode (1e-5)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows_per_sm", [20, 100, 300])
@pytest.mark.parametrize("n,pad", [(1, 0), (31, 0), (32, 1), (33, 3), (64, 0), (129, 2), (192, 0), (193, 0), (257, 1)])
def test_factor_f32_shapes(lib, rows_per_sm, n, pad):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    m = rows_per_sm * sms + 37
    g = torch.Generator(device="cuda").manual_seed(n + rows_per_sm)
    wide = torch.randn((m, n + pad), generator=g, device="cuda") * torch.linspace(1.0, 4.0, n + pad, device="cuda")
    A = wide[:, :n]
    plan = lib.rpcholqr_plan_create(0, m, n, 3 * n, mode=lib.FP32)
    Q0 = torch.full((m, n + pad), 7.0, device="cuda")
    Q, R, info = lib.rpcholqr_factor_f32(plan, A, 3 * n, 3, Q=Q0[:, :n])
    assert info.cpu().tolist() == [0, -1]
    Qd, Rd, Ad = Q.double(), R.double(), A.double()
    assert float((Qd.T @ Qd - torch.eye(n, dtype=torch.float64, device="cuda")).abs().max()) <= 1e-5
    assert float(torch.linalg.norm(Ad - Qd @ Rd) / torch.linalg.norm(Ad)) <= 1e-5
    assert bool((Q0[:, n:] == 7.0).all())        # nothing written beside the matrix
    A2 = A.clone()
    A2[m - 1, n - 1] = float("inf")
    assert lib.rpcholqr_factor_f32(plan, A2, 3 * n, 3)[2].cpu().tolist()[0] == 2
    plan.close()
