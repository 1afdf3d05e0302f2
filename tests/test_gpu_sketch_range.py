"""Range of the sketch QR: R_s, Q and R of A 2^k are those of A with R scaled by 2^k, bit for bit, also where the columns'
squares underflow, or come near the largest FP64 number, and where every column has a scale of its own.  (Scaling by powers of
two is exact in every step, so any other bit is a lost one.)  Sums of squares that overflow are refused."""
import pytest
import torch

pytestmark = pytest.mark.gpu
POWERS = [-530, -525, -520, -514, -512, -451, -449, 449, 451, 500, 505]


def times_pow2(a, k):
    """a 2^k in two exact steps."""
    return a * 2.0 ** (k // 2) * 2.0 ** (k - k // 2)


def matrix(m, n):
    g = torch.Generator(device="cuda").manual_seed(1000 + n)
    return torch.randn(m, n, generator=g, device="cuda", dtype=torch.float64)


@pytest.mark.parametrize("mode", ["FP64", "SPLIT64"])
@pytest.mark.parametrize("m,n,s", [(600, 1, 3), (900, 40, 120), (2000, 130, 390), (14000, 33, 13000)])   # the last: panel in place
def test_powers_of_two(lib, mode, m, n, s):
    A = matrix(m, n)
    plan = lib.rpcholqr_plan_create(0, m, n, s, mode=getattr(lib, mode))
    try:
        Rs0, _ = lib.rpcholqr_sketch_r(plan, A, s, 3)
        Q0, R0, info = lib.rpcholqr_factor(plan, A, s, 3)
        assert info.cpu().tolist() == [0, -1]
        for k in POWERS:
            Ak = times_pow2(A, k)
            Rs, info = lib.rpcholqr_sketch_r(plan, Ak, s, 3)
            assert info.cpu().tolist() == [0, -1], k
            assert torch.equal(Rs, times_pow2(Rs0, k)), k
            Q, R, info = lib.rpcholqr_factor(plan, Ak, s, 3)
            assert info.cpu().tolist() == [0, -1], k
            assert torch.equal(Q, Q0) and torch.equal(R, times_pow2(R0, k)), k
    finally:
        plan.close()


@pytest.mark.parametrize("m,n,s", [(900, 40, 120), (2000, 130, 390)])
def test_columns_of_different_scales(lib, m, n, s):
    A = matrix(m, n)
    d = torch.tensor([2.0 ** (0, -515, 300, -460, 400, -300, 460)[c % 7] for c in range(n)], dtype=torch.float64, device="cuda")
    plan = lib.rpcholqr_plan_create(0, m, n, s)
    try:
        Rs0, _ = lib.rpcholqr_sketch_r(plan, A, s, 3)
        Rs, info = lib.rpcholqr_sketch_r(plan, A * d, s, 3)
        assert info.cpu().tolist() == [0, -1]
        assert torch.equal(Rs, Rs0 * d)
    finally:
        plan.close()


def test_batched_and_zero_columns(lib):
    m, n, s = 900, 40, 120
    A = matrix(m, n)
    As = [A, times_pow2(A, -520), times_pow2(A, 505)]
    zero = A.clone()
    zero[:, 7] = 0.0
    plan = lib.rpcholqr_plan_create(0, m, n, s)
    try:
        Qs, Rs, info, _ = lib.rpcholqr_factor_batched(plan, As + [zero], [s] * 4, [3] * 4)
        torch.cuda.synchronize()
        assert info.cpu().tolist()[:6] == [0, -1] * 3
        assert int(info.cpu().view(-1)[6]) == lib.ERR_SINGULAR_SKETCH
        for i, a in enumerate(As):
            Q, R, _ = lib.rpcholqr_factor(plan, a, s, 3)
            assert torch.equal(Qs[i], Q) and torch.equal(Rs[i], R)
        for bad in (zero, times_pow2(A, 511), times_pow2(A, 560)):   # the last two: sums of squares that overflow
            _, _, info = lib.rpcholqr_factor(plan, bad, s, 3)
            assert int(info[0]) == lib.ERR_SINGULAR_SKETCH
    finally:
        plan.close()
