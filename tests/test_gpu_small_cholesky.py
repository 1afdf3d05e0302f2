"""Cholesky at the edge of one 32-column block (one launch up to it): R_1 against numpy's factor, the pivot of a matrix that is
not positive definite, and the split mode's R_1^{-1} through the factorisation."""
import numpy as np
import pytest
import torch

import inputs

pytestmark = pytest.mark.gpu
WIDTHS = [1, 2, 7, 8, 9, 16, 17, 31, 32, 33]


@pytest.mark.parametrize("n", WIDTHS)
def test_factor_and_pivot(lib, n):
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n + 40, n))
    G = X.T @ X
    plan = lib.rpcholqr_plan_create(0, 200, n, max(n, 3))
    try:
        R, info = lib.rpcholqr_cholesky(plan, torch.from_numpy(G).cuda())
        assert info.cpu().tolist() == [0, -1]
        ref = np.linalg.cholesky(G).T
        # both are backward stable: n u kappa(G) of the norm, kappa below 100 here
        assert np.linalg.norm(R.cpu().numpy() - ref) <= 2 * (n + 1) * 2.0 ** -53 * 100 * np.linalg.norm(ref)
        assert np.array_equal(np.tril(R.cpu().numpy(), -1), np.zeros((n, n)))
        for p in {0, n // 2, n - 1}:
            bad = G.copy()
            bad[p, p] = -1.0
            _, info = lib.rpcholqr_cholesky(plan, torch.from_numpy(bad).cuda())
            assert info.cpu().tolist() == [lib.ERR_NOT_SPD, p]
    finally:
        plan.close()


@pytest.mark.parametrize("n", WIDTHS)
def test_split_inverse(lib, n):
    m, s = 5000, max(3 * n, 3)
    A = inputs.usv(m, n, 1e3 if n > 1 else 1.0, 80 + n)
    plan = lib.rpcholqr_plan_create(0, m, n, s, mode=lib.SPLIT64)
    try:
        Q, R, info = lib.rpcholqr_factor(plan, torch.from_numpy(np.ascontiguousarray(A)).cuda(), s, 2)
        assert info.cpu().tolist() == [0, -1] and not lib.rpcholqr_plan_split_pass2_fp64(plan)
        Q = Q.cpu().numpy()
        assert np.linalg.norm(Q.T @ Q - np.eye(n), 2) <= 1e-13
        assert np.linalg.norm(Q @ R.cpu().numpy() - A) <= 1e-14 * np.linalg.norm(A)
    finally:
        plan.close()
