"""Calls narrower than 129 columns on an FP64 plan made for more: their fused row pass leaves one Gram partial per CTA
in the plan's buffer, more of them than the plan's own width takes.  The workspace holds them, and every result has the
bits of a plan made for the width."""
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
