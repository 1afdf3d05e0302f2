"""GPU tests of the blocked sketch QR (panels of 32 columns, row groups of a 64th of the rows) where its tiles end:
widths around a panel, as many rows as columns, fewer rows than groups, a sample too long for the panel to stay in
shared memory, and the one-CTA form of the batched kernel with its panel in and out of shared memory."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def _sample(s, n, kappa, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    v = np.linalg.qr(rng.standard_normal((n, n)))[0]
    sig = kappa ** -(np.arange(n) / max(1, n - 1))
    return rng.standard_normal((s, n)) @ (sig[:, None] * v.T)


@pytest.mark.parametrize("s,n,kappa", [(1, 1, 1.0), (2, 1, 1.0), (31, 31, 1e4), (32, 32, 1e4), (33, 32, 1e8),
                                       (64, 33, 1e12), (65, 64, 1e3), (97, 65, 1e16), (513, 96, 1e16), (1025, 129, 1e6),
                                       (385, 160, 1e16), (13600, 33, 1e6)])
def test_sketch_r_is_the_triangular_factor(lib, s, n, kappa):
    A = _sample(s, n, kappa, 7 * s + n)
    plan = lib.rpcholqr_plan_create(0, s, n, s)
    Rs, info = lib.rpcholqr_sketch_r_from_sample(plan, torch.from_numpy(A).cuda())
    assert info.cpu().tolist() == [0, -1]
    R = Rs.cpu().numpy()
    plan.close()
    assert np.all(np.diag(R) > 0) and np.all(np.tril(R, -1) == 0)
    # A + E = Q R with columnwise small E: R^T R and A^T A agree relative to the column norms, to the rounding of
    # s-term sums and n reflections (and of the two products compared here)
    c = np.linalg.norm(A, axis=0)
    assert np.max(np.abs(R.T @ R - A.T @ A) / np.outer(c, c)) <= 2 * (s + n) * U


@pytest.mark.parametrize("shift", [1, 7, 35])   # coprime to the row count: distinct rows
def test_powers_of_two_are_exact(lib, shift):
    # columns +-2^e e_i, permuted: every norm, square root and reciprocal is a power of two (the ends of the fixed-point
    # ranges), so R is exactly the diagonal of the column scales, to the last bit
    s, n = 96, 40
    scale = 2.0 ** ((np.arange(n) * 7) % 23 - 11)
    A = np.zeros((s, n))
    A[(np.arange(n) * shift + 5) % s, np.arange(n)] = np.where(np.arange(n) % 3, scale, -scale)
    plan = lib.rpcholqr_plan_create(0, s, n, s)
    Rs, info = lib.rpcholqr_sketch_r_from_sample(plan, torch.from_numpy(A).cuda())
    assert info.cpu().tolist() == [0, -1]
    assert np.array_equal(Rs.cpu().numpy(), np.diag(scale))
    plan.close()


@pytest.mark.parametrize("m,n,s", [(2000, 40, 120), (2000, 40, 2000), (3000, 33, 33), (700, 128, 640)])
def test_one_cta_gives_the_cluster_bits(lib, m, n, s):
    A = torch.from_numpy(_sample(m, n, 1e6, m + n)).cuda()
    plan = lib.rpcholqr_plan_create(0, m, n, s)
    Q1, R1, i1 = lib.rpcholqr_factor(plan, A, s, 5)
    Qs, Rs, i2, _ = lib.rpcholqr_factor_batched(plan, [A], [s], [5])
    assert i1.cpu().tolist() == i2.cpu().tolist() == [0, -1]
    assert torch.equal(Q1, Qs[0]) and torch.equal(R1, Rs[0])
    plan.close()
