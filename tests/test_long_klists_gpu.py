"""k lists of thousands of points in the FP64 adjoint, whose sum over k has terms that may all have one sign,
against sums over short pieces.

Tolerance 1e-9, that of every FP64 form in these tests (relative to the largest entry).
"""
import dataclasses

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


@pytest.fixture(scope="module")
def one_band(epw):
    rng = np.random.default_rng(9100)
    wm = W.make_model("sc", 1, 1, [1.0], 27, 27, rng)
    g = np.zeros_like(wm.g)
    g[0] = wm.g[0]  # (R = 0 comes first: g(k, q) does not depend on k)
    return dataclasses.replace(wm, g=g), rng


@pytest.mark.parametrize("nk", [2049, 6000, 40000])
def test_gradient_of_a_long_k_list(epw, one_band, nk):
    wm, rng = one_band
    assert not wm.Re[0].any()
    k, q = rng.random((nk, 3)), rng.random((31, 3))
    cot = np.ones((nk, 1))
    m = epw.Model(wm)
    par = dict(T=300.0, EF=0.1, sigma=3.0, precision=epw.FP64)
    got = m.linewidth_backward(k, q, cot, **par)
    ref = [sum(x) for x in zip(*(m.linewidth_backward(k[i:i + 1500], q, cot[i:i + 1500], **par)
                                 for i in range(0, nk, 1500)))]
    for a, b in zip(got, ref):
        assert np.abs(a - b).max() < 1e-9 * np.abs(b).max()
