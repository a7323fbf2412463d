"""A vertex, a weight or a cotangent that is not finite shows in the result even where no Gaussian reaches a
term, as it does when every term is formed: zero times it is not zero.
"""
import dataclasses

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

# Gaussians so narrow that no term of a few pairs is within them
PAR = dict(T=300.0, EF=0.1, sigma=1e-7)


@pytest.fixture(scope="module")
def epw():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1604_03525_gb300 as epw
    return epw


def _model(lat, nw, nat, nRe, nRp, bad=None):
    rng = np.random.default_rng(7300 + nw)
    wm = W.make_model(lat, nw, nat, [1.0 + 0.1 * i for i in range(nat)], nRe, nRp, rng)
    if bad is not None:
        g = wm.g.copy()
        g[3, 2, 1, nw - 1, 0] = bad
        wm = dataclasses.replace(wm, g=g)
    return wm, rng


# (sizes at which FP64 takes the fixed-point forms and TF32x3 the staged one)
SHAPES = [("sc", 2, 2, 81, 33, 60, 130), ("fcc", 3, 1, 79, 79, 60, 130), ("hex", 5, 3, 57, 57, 12, 130),
          ("diamond", 8, 2, 55, 55, 9, 130)]


@pytest.mark.parametrize("prec", ["FP64", "TF32X3", "FP32"])
@pytest.mark.parametrize("lat,nw,nat,nRe,nRp,nk,nq", SHAPES)
@pytest.mark.parametrize("what", ["vertex nan", "vertex inf", "cotangent", "weight"])
def test_gradient(epw, lat, nw, nat, nRe, nRp, nk, nq, prec, what):
    wm, rng = _model(lat, nw, nat, nRe, nRp, {"vertex nan": np.nan, "vertex inf": np.inf}.get(what))
    k, q, cot, wq = rng.random((nk, 3)), rng.random((nq, 3)), rng.random((nk, nw)), rng.random(nq)
    if what == "cotangent":
        cot[nk // 2, 0] = np.nan
    if what == "weight":
        wq[nq - 1] = np.inf
    m = epw.Model(wm)
    dg, dT, dE = m.linewidth_backward(k, q, cot, wq, precision=getattr(epw, prec), **PAR)
    m.sync()
    # (a column n of Xbar reaches every entry of dL/dg through the rotation by U_k)
    assert np.isnan(dg).all() and np.isnan(dT) and np.isnan(dE)


@pytest.mark.parametrize("lat,nw,nat,nRe,nRp,nk,nq", SHAPES)
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_weights_in_fp64(epw, lat, nw, nat, nRe, nRp, nk, nq, bad):
    wm, rng = _model(lat, nw, nat, nRe, nRp)
    k, q, wq, wk = rng.random((nk, 3)), rng.random((nq, 3)), rng.random(nq), rng.random(nk)
    m = epw.Model(wm)
    wq[5] = wk[7] = bad
    assert np.isnan(m.linewidth(k, q, wq, precision=epw.FP64, **PAR)).all()
    pi, lam, zeta, dos = m.phonon_selfenergy(k, q, wk, precision=epw.FP64, **PAR)
    assert np.isnan(pi).all() and np.isnan(zeta).all() and not np.isfinite(dos)
