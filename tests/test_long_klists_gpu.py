"""k lists of tens of thousands of points in FP64: the adjoint, whose sum over k has terms that may all have one
sign, and lists beyond the 65,535 blocks of a grid's second axis, against sums over short pieces.

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


def test_phonons_of_a_dense_k_grid(epw, one_band):
    """41^3 k x 8 q, more k than a grid has blocks along its second axis; weights given, so that the sums over
    pieces add up (lambda after its 1/N(E_F))."""
    wm, rng = one_band
    nk = 41 ** 3
    k, q, wk = rng.random((nk, 3)), rng.random((8, 3)), rng.random(nk) / nk
    m = epw.Model(wm)
    par = dict(T=300.0, EF=0.1, sigma=0.2, precision=epw.FP64)
    pi, lam, zeta, dos = (np.asarray(x) for x in m.phonon_selfenergy(k, q, wk, **par))
    parts = [[np.asarray(x) for x in m.phonon_selfenergy(k[i:i + 9000], q, wk[i:i + 9000], **par)]
             for i in range(0, nk, 9000)]
    for got, ref in ((pi, sum(p[0] for p in parts)), (lam * dos, sum(p[1] * p[3] for p in parts)),
                     (zeta, sum(p[2] for p in parts)), (dos, sum(p[3] for p in parts))):
        assert np.abs(got - ref).max() < 1e-9 * np.abs(ref).max()


def test_linewidths_of_a_dense_k_grid(epw, one_band):
    wm, rng = one_band
    k, q = rng.random((70000, 3)), rng.random((9, 3))
    m = epw.Model(wm)
    par = dict(T=300.0, EF=0.1, sigma=0.2, precision=epw.FP64)
    got = m.linewidth(k, q, **par)
    ref = np.concatenate([m.linewidth(k[i:i + 30000], q, **par) for i in range(0, 70000, 30000)])
    assert np.abs(got - ref).max() < 1e-9 * np.abs(ref).max()
