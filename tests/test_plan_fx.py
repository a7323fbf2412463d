"""Workspace of the FP64 form by shape alone (CPU): the fixed-point contractions hold at least one k
over all q, so a q list that would need more than 64 GiB for them keeps the CUDA cores' form."""
import pytest

import paper_1604_03525_gb300 as epw

GiB = 1 << 30


@pytest.mark.parametrize("nw,nat,nRe,nRp", [(18, 6, 43, 19), (8, 2, 249, 249), (1, 1, 27, 27)])
def test_long_q_lists_keep_the_small_plan(nw, nat, nRe, nRp):
    same = nRe == nRp
    per_q = 16 * ((nRe if same else nRe + nRp) + 3 * (3 * nat) ** 2) + 256 * nat  # phases, D, e and C in FP64
    for nq in (10 ** 5, 10 ** 6, 10 ** 7):
        ws, _ = epw.plan_linewidth(nw, nat, nRe, nRp, nRe, 3, nq, epw.FP64, same_ep=same, same_eph=True)
        assert ws < max(64 * GiB, nq * per_q + GiB)
