"""The batched FP64 eigensolves of the preparation: every matrix order and both ends of the
counts that choose between lanes per matrix (few matrices) and one thread per matrix (many).

Tolerance: Jacobi to an off-diagonal weight of 1e-30 of the matrix's leaves eigenvalues within a
few n ulp of the norm (here below 8 eV, n <= 18): 1e-12 eV against numpy's FP64 eigvalsh.
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


def _phase(x, R):
    return np.exp(2j * np.pi * (x @ R.T))


@pytest.mark.parametrize("nw", range(1, 19))
@pytest.mark.parametrize("nk", [1, 33, 700, 20011])
def test_bands_match_numpy(epw, nw, nk):
    rng = np.random.default_rng(nw)
    wm = W.make_model("sc", nw, 1, [1.0], 7, 1, rng)
    k = rng.random((nk, 3))
    k[0] = 0.0
    ref = np.linalg.eigvalsh(np.tensordot(_phase(k, wm.Re), wm.H, axes=(1, 0)))
    m = epw.Model(wm)
    # one atom's acoustic modes at a generic q; the k side is what varies
    eps = m.interp(k, rng.random((1, 3)), want_g=False)[0]
    m.sync()
    assert np.abs(eps - ref).max() < 1e-12


@pytest.mark.parametrize("nat", range(1, 7))
@pytest.mark.parametrize("nq", [1, 65, 3000, 25000])
def test_linewidth_does_not_depend_on_the_count(epw, nat, nq):
    """Eigenvectors: the linewidth of q = the first of a long list, alone and as the only one with
    weight, agrees (the long list's D(q) take another form)."""
    rng = np.random.default_rng(70 + nat)
    wm = W.make_model("fcc", 2, nat, [1.0 + 0.1 * i for i in range(nat)], 13, 13, rng)
    k, q = rng.random((2, 3)), rng.random((nq, 3))
    m = epw.Model(wm)
    par = dict(T=300.0, EF=0.0, sigma=0.4, precision=epw.FP64)
    w = np.zeros(nq)
    w[nq - 1] = 1.0
    one = m.linewidth(k, q[nq - 1:], **par)
    assert np.abs(m.linewidth(k, q, w, **par) - one).max() < 1e-11 * np.abs(one).max()


@pytest.mark.parametrize("nat", range(1, 7))
@pytest.mark.parametrize("n", [1, 700, 25000])
def test_both_kinds_of_rotations(epw, nat, n):
    """The FP32 form takes its FP64 phonons and bands from jacobi_herm's rotations, the FP64 form from
    the cheaper ones: omega^2 and e_k agree to 1e-12 of the largest (a few n ulp each)."""
    rng = np.random.default_rng(170 + nat)
    wm = W.make_model("fcc", 3 * nat, nat, [1.0 + 0.1 * i for i in range(nat)], 13, 13, rng)
    m = epw.Model(wm)
    x, one = rng.random((n, 3)), rng.random((1, 3))
    for k, q in ((one, x), (x, one)):
        a, b = (m.interp(k, q, precision=p, want_g=False) for p in (epw.FP32, epw.FP64))
        assert np.abs(a[0] - b[0]).max() < 1e-12 * np.abs(b[0]).max()
        wa, wb = (np.sign(w[2]) * w[2] ** 2 for w in (a, b))
        assert np.abs(wa - wb).max() < 1e-12 * np.abs(wb).max()
