"""Calls narrower than 129 columns on a plan made for more.  FP64: their fused row pass leaves one Gram partial per CTA in the
plan's buffer, more of them than the plan's own width takes; the workspace holds them, and every result has the bits of a
plan made for the width.  SPLIT64: the first pass is the narrow one (its rows' bits), the Gram and pass 2 stream images."""
import numpy as np
import pytest
import torch

import inputs

PLANS = [(3072, 384, 1152), (4096, 384, 1152), (10000, 192, 576), (10000, 300, 900)]


@pytest.mark.parametrize("m,n,s", PLANS)
def test_workspace_holds_the_narrow_partials(lib, m, n, s):
    np_ = -(-n // 64) * 64
    partials = min(152, -(-m // 64)) * 128 * 128          # panels have 64 rows or more, one CTA per SM at most
    sample = s * np_
    squares = 5 * np_ * np_                               # R_s, R1, G and two fragment tables
    tables = 2 * (np_ // 8) * 64
    sketch = 17 * 32 * np_ + 32 * 32 + 32 + np_
    assert lib.rpcholqr_workspace_size(m, n, s) >= 8 * (sample + squares + tables + sketch + partials)


@pytest.mark.gpu
@pytest.mark.parametrize("m,n,s", [PLANS[0], PLANS[2]])
def test_narrow_calls_on_a_wide_plan(lib, m, n, s):
    wide = lib.rpcholqr_plan_create(0, m, n, s)
    try:
        for k in (64, 100, 128):
            A = torch.from_numpy(np.ascontiguousarray(inputs.usv(m, k, 1e4, 60 + k))).cuda()
            own = lib.rpcholqr_plan_create(0, m, k, 3 * k)
            try:
                for call in (lambda p: lib.rpcholqr_factor(p, A, 3 * k, 7), lambda p: lib.rpcholqr_cholqr(p, A)):
                    a, b = call(wide), call(own)
                    assert a[2].cpu().tolist() == b[2].cpu().tolist() == [0, -1]
                    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
            finally:
                own.close()
    finally:
        wide.close()


@pytest.mark.gpu
@pytest.mark.parametrize("k", [17, 64, 65, 100, 128])
def test_narrow_calls_on_a_wide_split_plan(lib, k):
    m, n, s = 9001, 384, 1152
    A = torch.from_numpy(np.ascontiguousarray(inputs.usv(m, k, 1e4, 90 + k))).cuda()
    wide = lib.rpcholqr_plan_create(0, m, n, s, mode=lib.SPLIT64)
    own = lib.rpcholqr_plan_create(0, m, k, 3 * k, mode=lib.SPLIT64)
    try:
        (Q, R, info), (Q1, R1, info1) = (lib.rpcholqr_factor(p, A, 3 * k, 7) for p in (wide, own))
        assert info.cpu().tolist() == info1.cpu().tolist() == [0, -1]
        # A_1 is the same; the Gram's row ranges differ, so R_1 does by its rounding: k u kappa(A_1), kappa(A_1) < 10
        tol = 2 * k * 2.0 ** -53 * 10
        assert float((R - R1).norm() / R1.norm()) <= tol
        assert float((Q - Q1).norm() / Q1.norm()) <= tol
        eye = torch.eye(k, dtype=torch.float64, device="cuda")
        assert float(torch.linalg.matrix_norm(Q.T @ Q - eye, 2)) <= 1e-13
    finally:
        wide.close()
        own.close()
