"""Accuracy of the split first pass: its error reaches Q multiplied by kappa(A), so its products keep every digit pair down to
2^-62 of the scale.  Q of the whole factorisation against Q in extended precision: the split mode is to be as close as the
FP64 mode."""
import numpy as np
import pytest
import torch

import inputs

pytestmark = pytest.mark.gpu
LD = np.longdouble


def q_extended(A):
    """Q of A in extended precision: A R^{-1} with R of an FP64 QR, then Cholesky-QR of that."""
    def solve(X, R):
        X = X.astype(LD)
        for c in range(R.shape[0]):
            X[:, c] = (X[:, c] - X[:, :c] @ R[:c, c].astype(LD)) / LD(R[c, c])
        return X
    A1 = solve(A, np.linalg.qr(A)[1])
    G, n = A1.T @ A1, A1.shape[1]
    R = np.zeros((n, n), dtype=LD)
    for j in range(n):
        v = G[j, j:] - R[:j, j] @ R[:j, j:]
        R[j, j:] = v / np.sqrt(v[0])
    Q = solve(A1, R)
    return Q


@pytest.mark.parametrize("n", [33, 64, 100, 128])
def test_q_is_as_close_as_in_fp64(lib, n):
    m, s = 1200, 3 * n
    err = {"FP64": 0.0, "SPLIT64": 0.0}
    for seed in range(3):
        A = inputs.usv(m, n, 1e5, 300 + seed)
        Qx = q_extended(A)
        for mode in err:
            plan = lib.rpcholqr_plan_create(0, m, n, s, mode=getattr(lib, mode))
            Q, _, info = lib.rpcholqr_factor(plan, torch.from_numpy(np.ascontiguousarray(A)).cuda(), s, seed)
            assert info.cpu().tolist() == [0, -1]
            q = Q.cpu().numpy().astype(LD)
            q = q * np.sign((q * Qx).sum(axis=0))
            err[mode] += float(np.sqrt(((q - Qx) ** 2).sum()))
            plan.close()
    assert err["SPLIT64"] <= 1.25 * err["FP64"], err
