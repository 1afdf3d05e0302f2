"""GPU test of the split mode's diagonal-block solve at its edges: widths around the 16-column substitutions, the 32-column
halves and the 64-column blocks, row counts around the 128-row tiles and past one tile per SM, leading dimensions that
leave odd rows on 8 bytes only.  Bounds are those of the split mode: ||Q^T Q - I|| <= 1e-13 and the residual within 10x
of the FP64 oracle's."""
import numpy as np
import pytest
import torch

import inputs

pytestmark = pytest.mark.gpu
WIDTHS = [1, 15, 16, 17, 31, 32, 33, 47, 48, 49, 63, 64, 65, 80, 97, 127, 128, 129, 193]


@pytest.mark.parametrize("n", WIDTHS)
def test_split_block_edges(lib, oracle_mod, n):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    s = max(3 * n, 8)
    few = -(-s // 128) * 128
    rows = [(s + 1, 0), (few - 1, 1), (few, 3), (few + 1, 2)] + ([(128 * sms + 17, 1)] if n in (17, 65, 129) else [])
    plan = lib.rpcholqr_plan_create(0, max(m for m, _ in rows), n, s, mode=lib.SPLIT64)
    for m, pad in rows:
        if m < s:
            continue
        A = inputs.usv(m, n, 1e6 if n > 1 else 1.0, 40 + n)
        buf = torch.full((m, n + pad), float("nan"), dtype=torch.float64, device="cuda")   # the padding is not read
        X = buf[:, :n]
        X.copy_(torch.from_numpy(A))
        Q, R, info = lib.rpcholqr_factor(plan, X, s, 5)
        assert info.cpu().tolist() == [0, -1], (m, pad)
        Qh, Rh = Q.cpu().numpy(), R.cpu().numpy()
        o = oracle_mod.rpcholqr(A, s, 5)
        assert oracle_mod.orth_error(Qh) <= 1e-13, (m, pad)
        assert oracle_mod.residual(A, Qh, Rh) <= 10 * oracle_mod.residual(A, o["Q"], o["R"]) + 2.0 ** -52, (m, pad)
        free = [i for i in range(m) if i not in set(oracle_mod.sample_indices(5, m, s).tolist())]
        if free:                                     # the solve's own check: a row outside the sample, the last column
            X[free[-1], n - 1] = float("inf")
            _, _, info = lib.rpcholqr_factor(plan, X, s, 5)
            assert int(info[0]) == lib.ERR_NONFINITE, (m, pad)
    plan.close()
