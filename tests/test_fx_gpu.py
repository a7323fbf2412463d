"""FP64 contractions on the tensor cores (digit planes, fixed-point sums) and the FP64 per-pair
kernels that read them, against the FP64 oracle at the edges of their tiles and forms: q counts
around the 128-row tile, one to eighteen bands (one thread's registers and local memory, unrolled
and not), R counts whose K is and is not a multiple of 32, Re != Rp, T = 0, narrow and wide
Gaussians, scales far from one and vertices that are not finite.

Tolerance 1e-9, that of every FP64 form in these tests (floor 1e-6 of the largest value).
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


def _rel(got, ref):
    return float(np.max(np.abs(got - ref) / np.maximum(np.abs(ref), 1e-6 * np.abs(ref).max())))


def _model(lat, nw, nat, nRe, nRp, seed=0):
    rng = np.random.default_rng(4000 + 31 * nw + nat + seed)
    return W.make_model(lat, nw, nat, [1.0 + 0.1 * i for i in range(nat)], nRe, nRp, rng), rng


# (lattice, nw, nat, Re, Rp, nk, nq): sizes at which the library takes these forms
CASES = [
    ("sc", 1, 1, 27, 81, 470, 470), ("sc", 2, 1, 33, 7, 300, 257), ("sc", 3, 6, 33, 57, 5, 129),
    ("fcc", 4, 1, 120, 79, 3, 127), ("fcc", 4, 1, 120, 120, 130, 128), ("sc", 4, 4, 57, 57, 2, 1),
    ("hex", 5, 3, 93, 93, 2, 129), ("sc", 6, 2, 81, 33, 3, 300), ("diamond", 8, 2, 141, 141, 3, 255),
    ("hex", 9, 2, 33, 51, 2, 100), ("diamond", 12, 2, 55, 43, 2, 129), ("fcc", 18, 1, 43, 19, 2, 65),
    ("sc", 18, 6, 7, 27, 1, 33),
]


@pytest.mark.parametrize("T,sigma", [(300.0, 0.05), (0.0, 0.004), (50.0, 0.6)])
@pytest.mark.parametrize("lat,nw,nat,nRe,nRp,nk,nq", CASES)
def test_linewidth(epw, oracle_lib, lat, nw, nat, nRe, nRp, nk, nq, T, sigma):
    wm, rng = _model(lat, nw, nat, nRe, nRp)
    k, q = rng.random((nk, 3)), rng.random((nq, 3))
    q[0] = 0.0  # acoustic modes left out
    wq = None if nq % 2 else rng.random(nq) / nq
    ref = oracle_lib.linewidth(wm, k, q, wq, T, 0.1, sigma)
    m = epw.Model(wm)
    got = m.linewidth(k, q, wq, T=T, EF=0.1, sigma=sigma, precision=epw.FP64)
    m.sync()
    if ref.max() > 1e-250:
        assert _rel(got, ref) < 1e-9


def test_scale_invariance(epw):
    """The digits are relative to each row's exponent: a vertex scaled by 2^-200 gives the same
    linewidth scaled by 2^-400, bit for bit."""
    wm, rng = _model("fcc", 4, 1, 120, 79)
    k, q = rng.random((4, 3)), rng.random((200, 3))
    par = dict(T=300.0, EF=0.0, sigma=0.05, precision=epw.FP64)
    one = epw.Model(wm).linewidth(k, q, **par)
    two = epw.Model(dataclasses.replace(wm, g=wm.g * 2.0 ** -200)).linewidth(k, q, **par)
    assert np.array_equal(two, one * 2.0 ** -400)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_vertex_that_is_not_finite_shows(epw, bad):
    wm, rng = _model("fcc", 4, 1, 120, 79)
    g = wm.g.copy()
    g[3, 5, 1, 2, 0] = bad
    k, q = rng.random((4, 3)), rng.random((200, 3))
    got = epw.Model(dataclasses.replace(wm, g=g)).linewidth(k, q, T=300.0, EF=0.0, sigma=0.05, precision=epw.FP64)
    assert np.isnan(got).all()


@pytest.mark.parametrize("where", ["k", "q"])
def test_a_point_that_is_not_finite_is_reported(epw, where):
    wm, rng = _model("fcc", 4, 1, 120, 79)
    pts = {"k": rng.random((4, 3)), "q": rng.random((200, 3))}
    pts[where][2, 1] = np.nan
    with pytest.raises(epw.EPWError) as e:
        epw.Model(wm).linewidth(pts["k"], pts["q"], T=300.0, EF=0.0, sigma=0.05, precision=epw.FP64)
    assert e.value.status == 4  # EPW_ERR_NOT_CONVERGED


@pytest.mark.parametrize("nk", [1, 3, 5, 130])
@pytest.mark.parametrize("nw,nRe,nRp", [(1, 27, 27), (4, 135, 19), (4, 13, 249)])
def test_kside_vertex_forms_agree(epw, nw, nRe, nRp, nk):
    """Few k (CUDA cores) and many (digit planes): the linewidth of each k alone and in the list."""
    wm, rng = _model("fcc", nw, 1, nRe, nRp)
    k, q = rng.random((nk, 3)), rng.random((150, 3))
    m = epw.Model(wm)
    par = dict(T=300.0, EF=0.0, sigma=0.3, precision=epw.FP64)
    all_k = m.linewidth(k, q, **par)
    for i in {0, nk // 2, nk - 1}:
        one = m.linewidth(k[i:i + 1], q, **par)
        assert np.abs(all_k[i] - one[0]).max() < 1e-12 * np.abs(one).max()


@pytest.mark.parametrize("lat,nw,nat,nRe,nRp,nk,nq", [("sc", 1, 1, 27, 81, 9000, 33), ("fcc", 4, 1, 120, 79, 700, 7),
                                                      ("hex", 5, 3, 57, 93, 40, 33), ("diamond", 8, 2, 55, 87, 30, 9)])
def test_phonons(epw, oracle_lib, lat, nw, nat, nRe, nRp, nk, nq):
    """Warps of 32 q around a full and a nearly empty one, few and many k per warp.  Pi'' cancels between
    terms of both signs: relative to its largest entry."""
    wm, rng = _model(lat, nw, nat, nRe, nRp)
    k, q = rng.random((nk, 3)), rng.random((nq, 3))
    wk = rng.random(nk) / nk
    ref = oracle_lib.phonon_self(wm, k, q, wk, 300.0, 0.1, 0.1)
    m = epw.Model(wm)
    got = m.phonon_selfenergy(k, q, wk, T=300.0, EF=0.1, sigma=0.1, precision=epw.FP64)
    m.sync()
    assert np.abs(got[0] - ref[0]).max() < 1e-9 * np.abs(ref[0]).max()
    assert _rel(got[1], ref[1]) < 1e-9 and _rel(got[2], ref[2]) < 1e-9


@pytest.mark.parametrize("nq", [2047, 2049, 4099])
def test_gradient_of_a_long_q_list(epw, nq):
    """The adjoint's sum over q in one part and in several (each part has its own fixed point): the
    gradient over the list against the sum over pieces of at most 700 q."""
    wm, rng = _model("fcc", 4, 1, 43, 19)
    k, q = rng.random((3, 3)), rng.random((nq, 3))
    wq, cot = rng.random(nq) / nq, rng.random((3, 4))
    m = epw.Model(wm)
    par = dict(T=300.0, EF=0.1, sigma=0.1, precision=epw.FP64)
    got = m.linewidth_backward(k, q, cot, wq, **par)
    ref = [sum(x) for x in zip(*(m.linewidth_backward(k, q[i:i + 700], cot, wq[i:i + 700], **par)
                                 for i in range(0, nq, 700)))]
    m.sync()
    for a, b in zip(got, ref):
        assert np.abs(a - b).max() < 1e-9 * np.abs(b).max()


@pytest.mark.parametrize("nk,nq", [(1, 2000), (3, 257), (20, 129)])
def test_interpolation_of_a_list(epw, oracle_lib, nk, nq):
    wm, rng = _model("fcc", 4, 1, 120, 79)
    k, q = rng.random((nk, 3)), rng.random((nq, 3))
    ek, ekq, om, g = epw.Model(wm).interp(k, q)
    rk, rkq, rom, rg = oracle_lib.interp(wm, k, q)
    assert _rel(ek, rk) < 1e-9 and _rel(ekq, rkq) < 1e-9 and _rel(om, rom) < 1e-9
    # |g|^2 summed over the bands at k + q and the modes does not depend on the eigenvectors' phases
    a, b = ((np.abs(x) ** 2).sum(axis=(2, 3)) for x in (g, rg))
    assert _rel(a, b) < 1e-9


@pytest.mark.parametrize("nw,nat,nRe,nRp", [(1, 1, 27, 19), (4, 1, 79, 43), (5, 3, 33, 57)])
@pytest.mark.parametrize("nk", [32, 33, 64, 65, 130])
def test_kside_vertex_fp32(epw, nw, nat, nRe, nRp, nk):
    """The FP32 k-side vertex over its tiles (32 and 64 k, g in FP64 and as an FP32 copy): each k alone
    and in the list, within the FP32 form's tolerance."""
    wm, rng = _model("hex", nw, nat, nRe, nRp)
    k, q = rng.random((nk, 3)), rng.random((150, 3))
    m = epw.Model(wm)
    par = dict(T=300.0, EF=0.0, sigma=0.3, precision=epw.FP32)
    all_k = m.linewidth(k, q, **par)
    for i in {0, 31, nk - 1}:
        one = m.linewidth(k[i:i + 1], q, **par)
        assert np.abs(all_k[i] - one[0]).max() < 2e-3 * np.abs(one).max()
