"""Accuracy of the split first pass: its error reaches Q multiplied by kappa(A), so its products keep every digit pair down to
2^-62 of the scale.  The subtracting product against exact integers, and Q of the whole factorisation against Q in extended
precision, where the split mode is to be as close as the FP64 mode."""
from fractions import Fraction

import numpy as np
import pytest
import torch

import inputs

pytestmark = pytest.mark.gpu
LD = np.longdouble


def integers(x):
    """Entries as integers in units of 2^-120 (exact for the entries used here)."""
    return np.array([[int(Fraction(float(v)) * 2 ** 120) for v in row] for row in x], dtype=object)


@pytest.mark.parametrize("K,N", [(34, 40), (64, 64), (128, 17)])
def test_subtracting_product(lib, K, N):
    # sums of full-size terms that nearly cancel, so that the result's own rounding is far below the product's
    rng = np.random.default_rng(K)
    X, Y = rng.uniform(-0.99, 0.99, (130, K // 2)), rng.uniform(-0.99, 0.99, (K // 2, N))
    X = np.hstack([X, X + rng.uniform(-0.001, 0.001, X.shape)])
    Y = np.vstack([Y, -Y + rng.uniform(-0.001, 0.001, Y.shape)])
    plan = lib.rpcholqr_plan_create(0, 1024, 128, 384, mode=lib.SPLIT64)
    try:
        C, info = lib.rpcholqr_ozaki_update(plan, torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda(),
                                            torch.zeros(130, N, dtype=torch.float64, device="cuda"))
        assert info.cpu().tolist() == [0, -1]
    finally:
        plan.close()
    exact = integers(X) @ integers(Y)                                   # units of 2^-240
    err = np.array([[float(Fraction(float(c)) + Fraction(int(e), 2 ** 240)) for c, e in zip(rc, re)]
                    for rc, re in zip(C.cpu().numpy(), exact)])
    bound = lambda a, axis: 2.0 ** (np.floor(np.log2(np.abs(a).max(axis=axis))) + 1)   # noqa: E731
    units = err / (np.outer(bound(X, 1), bound(Y, 0)) * 2.0 ** -53)
    # units of 2^-53 of the scale, mean square: one rounding, 1/12; K terms of two operands rounded to 2^-56 of their bounds
    # (1/192 each) times a factor of 1/3 in the mean square: K / 288; a fifth for the sample.  The pairs with a + b = 9, if
    # dropped, would add 6 K (128^2 / 3)^2 2^-34 = K / 96.
    assert float(np.mean(units ** 2)) <= 1.2 * (1 / 12 + K / 288)


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
