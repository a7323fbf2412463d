"""The sums over blocks of q are compensated term by term: weights 1, 2^-60, -1, 0 on the consecutive terms
of a thread leave the second's share, which a plain sum of any group of them loses.

All q are the same point and the weights powers of two, so every block's term is the same number times its
weight, exactly; what is left is exact up to the sum's own roundings, a few of 2^-53: 1e-12.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

PATTERN = np.array([1.0, 2.0 ** -60, -1.0, 0.0])


@pytest.fixture(scope="module")
def epw():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1604_03525_gb300 as epw
    return epw


def _model(nw):
    rng = np.random.default_rng(88 + nw)
    return W.make_model("fcc", nw, 1, [1.0], 19, 19, rng), rng


@pytest.mark.parametrize("prec", ["FP64", "FP32"])
@pytest.mark.parametrize("nw", [1, 2, 4])
def test_linewidth(epw, nw, prec):
    wm, rng = _model(nw)
    k, q = rng.random((2, 3)), rng.random((1, 3))
    m = epw.Model(wm)
    par = dict(T=300.0, EF=0.1, sigma=1.0, precision=getattr(epw, prec))
    # 12 terms for each of the 128 threads of a k: thread (warp, lane) has the bands and blocks lane, lane + 32, ...
    # of its quarter of [blocks][nw]
    nqb = 128 * 12 // nw
    w = PATTERN[(np.arange(nqb) // (32 // nw)) % 4]
    one = m.linewidth(k, np.repeat(q, 128, axis=0), np.full(128, 2.0 ** -7), **par)
    got = m.linewidth(k, np.repeat(q, 128 * nqb, axis=0), np.repeat(w, 128) * 2.0 ** -7, **par)
    assert np.abs(got - one * (nqb // 4) * PATTERN[1]).max() < 1e-12 * np.abs(got).max()


@pytest.mark.parametrize("prec", ["FP64", "FP32"])
def test_self_energy(epw, prec):
    wm, rng = _model(4)
    k, q, omega = rng.random((2, 3)), rng.random((1, 3)), np.array([-0.3, 0.2])
    m = epw.Model(wm)
    par = dict(T=300.0, EF=0.1, delta=0.5, precision=getattr(epw, prec))
    nqw = 4 * 48  # warps of 32 q, a quarter of them in turn to a thread
    one = m.selfenergy(k, np.repeat(q, 32, axis=0), omega, np.full(32, 2.0 ** -5), **par)[0]
    got = m.selfenergy(k, np.repeat(q, 32 * nqw, axis=0), omega, np.repeat(PATTERN[np.arange(nqw) % 4], 32) * 2.0 ** -5,
                       **par)[0]
    assert np.abs(got - one * (nqw // 4) * PATTERN[1]).max() < 1e-12 * np.abs(got).max()
