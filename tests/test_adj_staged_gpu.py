"""The per-pair adjoint of the staged FP32 forms (only the terms whose FP32 Gaussians do not
underflow) at the edges of its blocks and warps and of its band counts, against the FP64 form.

Tolerance 2e-4 of the largest entry of dL/dg and 2e-4 of dL/dT and dL/dE_F's term sums: the
TF32x3 tolerance of the other adjoint tests.
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


@pytest.mark.parametrize("nq", [1, 31, 129, 300])
@pytest.mark.parametrize("lat,nw,nat", [("sc", 1, 2), ("sc", 2, 3), ("fcc", 3, 1), ("sc", 4, 2), ("hex", 5, 3),
                                        ("sc", 7, 2), ("diamond", 8, 2)])
def test_against_fp64(epw, lat, nw, nat, nq):
    rng = np.random.default_rng(8000 + 10 * nw + nat)
    wm = W.make_model(lat, nw, nat, [1.0 + 0.1 * i for i in range(nat)], 19, 27, rng)
    k, q = rng.random((3, 3)), rng.random((nq, 3))
    cot = rng.random((3, nw))  # one sign: dL/dT does not cancel
    m = epw.Model(wm)
    par = dict(T=300.0, EF=0.1, sigma=0.06)
    ref = m.linewidth_backward(k, q, cot, precision=epw.FP64, **par)
    got = m.linewidth_backward(k, q, cot, precision=epw.TF32X3, **par)
    m.sync()
    assert np.abs(got[0] - ref[0]).max() < 2e-4 * np.abs(ref[0]).max()
    assert abs(got[1] - ref[1]) < 2e-4 * abs(ref[1]) + 1e-12
    assert abs(got[2] - ref[2]) < 2e-4 * max(abs(ref[2]), 10 * abs(ref[1]))
