"""GPU test of the row passes' panel shapes: a solved row does not depend on the panel it was solved in, so a call
short enough for the small panels (4 to 8 warps of 16 rows) gives the bits of a call that takes the big ones, at
widths around every shape (32 rows per warp up to 64 columns, 16 above) and row counts around a panel."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 8, 16, 17, 32, 48, 49, 64, 65, 100, 128])
def test_short_calls_give_the_bits_of_long_ones(lib, n):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    m = 2 * 64 * sms + 300                       # beyond the line of either width
    g = torch.Generator(device="cuda").manual_seed(n)
    X = torch.randn((m, n), generator=g, dtype=torch.float64, device="cuda")
    T = torch.triu(torch.randn((n, n), generator=g, dtype=torch.float64, device="cuda")) / n
    T.diagonal().copy_(1.0 + torch.rand(n, generator=g, dtype=torch.float64, device="cuda"))
    plan = lib.rpcholqr_plan_create(0, m, n, n)
    Y, info = lib.rpcholqr_solve_rows(plan, X, T)
    assert info.cpu().tolist() == [0, -1]
    # backward stable row by row: |Y T - X| <= ~2 n u |Y| |T|
    bound = 2 * (n + 2) * 2.0 ** -53 * (Y.abs() @ T.abs()) + 1e-300
    assert bool(((Y @ T - X).abs() <= 2 * bound).all())
    for rows in (1, 15, 16, 17, 63, 64, 65, 129, 64 * sms, 64 * sms + 1, 100 * sms):
        Ys, info = lib.rpcholqr_solve_rows(plan, X[m - rows:], T)
        assert info.cpu().tolist() == [0, -1]
        assert torch.equal(Ys, Y[m - rows:]), rows
        A1, G, info = lib.rpcholqr_precondition_gram(plan, X[m - rows:], T)
        assert info.cpu().tolist() == [0, -1]
        assert torch.equal(A1, Ys), rows
        ref = Ys.T @ Ys
        assert bool(((G - ref).abs() <= 2 * (rows + 2) * 2.0 ** -53 * (Ys.abs().T @ Ys.abs()) + 1e-300).all())
    plan.close()
