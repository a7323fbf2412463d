"""The fixed-point contractions by themselves: the bands of a one-band model are H(k+q), nothing else, so
they are compared with sums in extended precision; and sums whose digits all agree (one q many times over:
the same phases, the same Xbar), which is where an FP32 accumulator of a digit level could round.  And
zero temperature, where the step of the occupations meets narrow Gaussians.

Tolerances: 1. the one-axis phase factors and their two products are good to 4 x 2^-53 each, the digits to
2^-55 and the sum to 2^-52 of the row's largest element per term: with nR terms of size at most h,
|error| < nR h 2^-50.  2. a level of digit products that exceeds 2^24 rounds by one unit at most 32 times per
256 terms, 2^-41 of the row's scale beside a sum of at least 2^6 of it: 2^-47 relative, 1e-13 with the
other FP64 steps.  3. 1e-9, that of every FP64 form in these tests.
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


@pytest.mark.parametrize("nR,scale", [(27, 1.0), (81, 1.0), (251, 1.0), (81, 1e-6)])
def test_sums_in_extended_precision(epw, nR, scale):
    """scale: the hoppings beside the on-site energy, a row whose elements differ by as much."""
    rng = np.random.default_rng(40 + nR)
    wm = W.make_model("sc", 1, 1, [1.0], nR, 7, rng)
    H = wm.H.copy()
    H[1:] *= scale
    wm = dataclasses.replace(wm, H=H)
    k, q = rng.random((40, 3)), rng.random((3000, 3))
    ekq = epw.Model(wm).interp(k, q, want_g=False)[1][..., 0]
    i, j = rng.integers(0, 40, 300), rng.integers(0, 3000, 300)
    L = np.longdouble
    pi2 = 8 * np.arctan(L(1))
    kR, qR = (x.astype(L) @ wm.Re.astype(L).T for x in (k[i], q[j]))
    a = pi2 * ((kR - np.rint(kR)) + (qR - np.rint(qR)))
    ref = (np.cos(a) * wm.H[:, 0, 0].real.astype(L) - np.sin(a) * wm.H[:, 0, 0].imag.astype(L)).sum(axis=1)
    err = np.abs(ekq[i, j].astype(L) - ref).max()
    assert err < len(wm.Re) * np.abs(wm.H).max() * 2.0 ** -50


@pytest.mark.parametrize("seed", range(6))
@pytest.mark.parametrize("nq", [128, 2048, 4096])
def test_digits_that_agree(epw, nq, seed):
    rng = np.random.default_rng(60 + seed)
    wm = W.make_model("fcc", 2, 1, [1.0], 43, 43, rng)
    nk = 1 + 120000 // nq
    k, q, cot = rng.random((nk, 3)), rng.random((1, 3)), np.ones((nk, 2))
    m = epw.Model(wm)
    par = dict(T=300.0, EF=0.1, sigma=1.0, precision=epw.FP64)
    got = m.linewidth_backward(k, np.repeat(q, nq, axis=0), cot, np.full(nq, 1.0 / nq), **par)
    ref = m.linewidth_backward(k, q, cot, np.ones(1), **par)
    for a, b in zip(got, ref):
        assert np.abs(a - b).max() < 1e-13 * np.abs(b).max()


@pytest.mark.parametrize("sigma", [0.02, 0.004])
@pytest.mark.parametrize("lat,nw,nat,nRe,nRp,nk,nq", [("sc", 1, 1, 27, 81, 470, 470), ("fcc", 4, 1, 120, 79, 12, 300),
                                                      ("hex", 5, 3, 93, 93, 6, 129), ("diamond", 8, 2, 141, 141, 6, 255),
                                                      ("fcc", 18, 1, 43, 19, 2, 65)])
def test_zero_temperature(epw, oracle_lib, lat, nw, nat, nRe, nRp, nk, nq, sigma):
    rng = np.random.default_rng(70 + nw)
    wm = W.make_model(lat, nw, nat, [1.0 + 0.1 * i for i in range(nat)], nRe, nRp, rng)
    k, q = rng.random((nk, 3)), rng.random((nq, 3))
    ref = oracle_lib.linewidth(wm, k, q, None, 0.0, 0.1, sigma)
    m = epw.Model(wm)
    got = m.linewidth(k, q, T=0.0, EF=0.1, sigma=sigma, precision=epw.FP64)
    m.sync()
    assert np.isfinite(got).all()
    assert np.abs(got - ref).max() <= 1e-9 * np.abs(ref).max() + 1e-250
