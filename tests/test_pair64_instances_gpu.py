"""The FP64 per-pair kernels over every band count and one to four atoms (their instances go by bounds on
both): a list long enough for them against pieces short enough for the CUDA cores' kernels.

Tolerance 1e-9, that of every FP64 form in these tests (relative to the largest entry).
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


@pytest.mark.parametrize("nat", [1, 2, 3, 4])
@pytest.mark.parametrize("nw", range(1, 11))
def test_instances(epw, nw, nat):
    rng = np.random.default_rng(900 + 10 * nw + nat)
    nR = 27 if nw == 1 else 7  # 4 nw^2 nR (1 + 3nat) instructions a pair on the CUDA cores
    wm = W.make_model("sc", nw, nat, [1.0 + 0.1 * i for i in range(nat)], nR, nR, rng)
    per = 0.032 * 4 * nw * nw * nR * (1 + 3 * nat)  # us of 19,456 pairs at once
    nq = 200
    nk = max(9, int(200.0 / per * 19456 / nq) + 1)
    step = 2 if per < 140.0 else 0
    k, q, cot = rng.random((nk, 3)), rng.random((nq, 3)), rng.random((nk, nw))
    wk, wq = rng.random(nk) / nk, rng.random(nq) / nq
    m = epw.Model(wm)
    par = dict(T=300.0, EF=0.1, sigma=0.1, precision=epw.FP64)
    if step == 0:  # wide models: every piece takes these kernels; against the FP32 form
        got = m.linewidth(k, q, wq, **par)
        ref = m.linewidth(k, q, wq, **dict(par, precision=epw.FP32))
        assert np.abs(got - ref).max() < 2e-3 * np.abs(ref).max()
        return
    pieces = [slice(i, i + max(1, nk // 8)) for i in range(0, nk, max(1, nk // 8))]
    got = m.linewidth(k, q, wq, **par)
    ref = np.concatenate([m.linewidth(k[p], q, wq, **par) for p in pieces])
    assert np.abs(got - ref).max() < 1e-9 * np.abs(ref).max()
    if nw > 8 or nat > 3:
        return
    got = m.linewidth_backward(k, q, cot, wq, **par)
    ref = [sum(x) for x in zip(*(m.linewidth_backward(k[p], q, cot[p], wq, **par) for p in pieces))]
    for a, b in zip(got, ref):
        assert np.abs(a - b).max() < 1e-9 * np.abs(b).max()
    pi, lam, zeta, dos = m.phonon_selfenergy(k, q, wk, **par)
    parts = [m.phonon_selfenergy(k[p], q, wk[p], **par) for p in pieces]
    for a, b in ((pi, sum(x[0] for x in parts)), (np.asarray(lam) * dos, sum(np.asarray(x[1]) * x[3] for x in parts)),
                 (zeta, sum(x[2] for x in parts))):
        assert np.abs(a - b).max() < 1e-9 * np.abs(b).max()
