"""A wait of the split mode's block solve that gives up: the thread that issues the MMAs issues no more of them, so that one
commit at most is open when the kernel waits for its own MMAs and frees its tensor memory."""
import os
import re

import numpy as np
import pytest
import torch

import inputs

OZAKI = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2406_11751_gb300", "csrc", "ozaki.cu")


def test_no_issue_after_a_wait_gave_up():
    body = re.sub(r"//[^\n]*", "", open(OZAKI).read())
    body = body[body.index("k_split_solve(const double* X"):]
    body = body[:body.index("\n}")]
    issues = [m.start() for m in re.finditer(r"ss_issue<", body)]
    assert len(issues) == 2
    for at in issues:
        guard = body[body.rindex("if (", 0, at):at]
        assert "(tid & 255) == 0" in guard and "&& ok)" in guard, guard
    # an mbarrier's phase is named by its parity alone: the closing wait takes the number of the last commit made
    assert re.search(r"mbar_wait\(bar, \(commits - 1\) & 1u\)", body)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [32, 64, 128])
def test_short_limits_report_and_recover(lib, oracle_mod, n):
    m, s = 40000, 3 * n
    A = inputs.usv(m, n, 1e4, 70 + n)
    Ad = torch.from_numpy(np.ascontiguousarray(A)).cuda()
    plan = lib.rpcholqr_plan_create(0, m, n, s, mode=lib.SPLIT64)
    try:
        for limit in (1, 2, 8, 64):
            lib.rpcholqr_plan_set_option(plan, lib.OPT_SPIN_LIMIT, limit)
            for _ in range(3):
                _, _, info = lib.rpcholqr_factor(plan, Ad, s, 3)
                assert info.cpu().tolist()[0] in (0, lib.ERR_TIMEOUT)
        lib.rpcholqr_plan_set_option(plan, lib.OPT_SPIN_LIMIT, 1 << 24)
        Q, R, info = lib.rpcholqr_factor(plan, Ad, s, 3)
        assert info.cpu().tolist() == [0, -1]
        o = oracle_mod.rpcholqr(A, s, 3)
        assert np.linalg.norm(R.cpu().numpy() - o["R"], 2) <= 1e-12 * np.linalg.norm(o["R"], 2)
        assert oracle_mod.orth_error(Q.cpu().numpy()) <= 1e-13
    finally:
        plan.close()
