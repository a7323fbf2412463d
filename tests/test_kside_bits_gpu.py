"""The k side of the FP32 and split forms is cast to FP32 and split: a value that moves by its last FP64
place can be cast the other way, and nothing averages it, since every q of that k reads it.  So its phases,
H(k) sums and rotations do not depend on how many k a call has.

Tolerance: the same pairs and the same FP32 terms on both sides, so only the FP64 sums of positive terms
can be grouped otherwise, 200 terms of 2^-53: 1e-13 (one band energy that is cast the other way moves a
linewidth by 1e-7).
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


def _between_floats(epw, lat, nw, nat, nRe, nRp, nk, tries):
    """Models whose lowest band at the first k lies half way between two FP32 numbers (as far as FP64 places
    it: the on-site energies are shifted by the distance), and the k list (more than 65,536 elements of H(k))."""
    rng = np.random.default_rng(6100 + nw)
    wm = W.make_model(lat, nw, nat, [1.0 + 0.1 * i for i in range(nat)], nRe, nRp, rng)
    assert not wm.Re[0].any() and wm.wRe[0] == 1.0
    q = rng.random((40, 3))
    for _ in range(tries):
        k = rng.random((nk, 3))
        e = epw.Model(wm).interp(k, q[:1], precision=epw.FP32, want_g=False)[0][0, 0]
        f = np.float32(e)
        half = (np.float64(f) + np.float64(np.nextafter(f, np.float32(9.0)))) / 2
        H = wm.H.copy()
        H[0] += (half - e) * np.eye(nw)
        yield dataclasses.replace(wm, H=H), k, q


@pytest.mark.parametrize("prec", ["FP32", "TF32X3", "BF16X3"])
@pytest.mark.parametrize("lat,nw,nat,nRe,nRp,nk", [("sc", 2, 2, 81, 33, 17000), ("fcc", 4, 1, 79, 79, 4200),
                                                   ("hex", 5, 3, 57, 57, 2700), ("diamond", 8, 2, 19, 19, 1100),
                                                   ("fcc", 18, 1, 43, 19, 220)])
def test_linewidth_of_a_k_does_not_depend_on_the_list(epw, lat, nw, nat, nRe, nRp, nk, prec):
    par = dict(T=300.0, EF=0.1, sigma=0.3, precision=getattr(epw, prec))
    for wm, k, q in _between_floats(epw, lat, nw, nat, nRe, nRp, nk, 12):
        m = epw.Model(wm)
        whole = m.linewidth(k, q, **par)
        for n in (1, 3, nk // 20, nk // 2):
            part = m.linewidth(k[:n], q, **par)
            assert np.abs(whole[:n] - part).max() < 1e-13 * np.abs(whole).max()
