"""Phonons and bands of the FP32 form come out to the bit whatever the length of the list: the sums over R
and the rotations have forms for few and for many points (one chain over R, the same roundings in every
eigensolver), since what is cast to FP32 afterwards must not depend on them.  Bits: no tolerance.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def epw():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1604_03525_gb300 as epw
    return epw


@pytest.mark.parametrize("nw,nat", [(2, 1), (3, 2), (4, 2), (5, 3), (6, 3), (8, 1), (9, 4), (12, 5), (18, 6)])
@pytest.mark.parametrize("nR", [19, 57])
def test_points_do_not_depend_on_their_list(epw, nw, nat, nR):
    """More than 65,536 matrix elements at once, and the same points in pieces of one to hundreds."""
    rng = np.random.default_rng(300 + nw)
    wm = W.make_model("sc", nw, nat, [1.0 + 0.1 * i for i in range(nat)], nR, 7, rng)
    m = epw.Model(wm)
    one = rng.random((1, 3))
    get = lambda k, q: m.interp(k, q, precision=epw.FP32, want_g=False)  # noqa: E731
    for which, n in (("k", 66000 // nw ** 2 + 200), ("q", 66000 // (3 * nat) ** 2 + 200)):
        x = rng.random((n, 3))
        pick = (lambda y: get(y, one)[0]) if which == "k" else (lambda y: get(one, y)[2])
        whole = pick(x)
        for b in (1, 2, 40, 600):
            b = min(b, n // 2)
            for a in (0, n - b):
                assert np.array_equal(whole[a:a + b], pick(x[a:a + b])), (which, b)
