"""FP64 calls on a device whose memory is nearly all taken (by a tensor of the caller's): the fixed-point
contractions' workspace does not fit, the CUDA cores' does, and the call runs as it did without them.

Tolerance 1e-9, that of every FP64 form in these tests (relative to the largest entry).
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

LEFT = 7 << 28  # 1.75 GiB: the contraction chunk of the fixed-point forms alone is 2 GiB


def test_fp64_calls_with_little_memory_left():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1604_03525_gb300 as epw
    rng = np.random.default_rng(51)
    wm = W.make_model("fcc", 4, 1, [1.0], 43, 43, rng)
    k, q, cot = rng.random((700, 3)), rng.random((4000, 3)), rng.random((700, 4))
    par = dict(T=300.0, EF=0.1, sigma=0.1, precision=epw.FP64)
    kd, qd = (torch.tensor(x, device="cuda") for x in (k, q))
    job = lambda m: dict(model=m, k=kd, q=qd, **par)  # noqa: E731

    def calls():
        out = []
        for f in (lambda m: [m.linewidth(k, q, **par)], lambda m: m.linewidth_backward(k, q, cot, **par),
                  lambda m: m.phonon_selfenergy(k, q, **par), lambda m: [x.cpu() for x in epw.Batch([job(m)]).run()]):
            m = epw.Model(wm)
            out += [np.asarray(x) for x in f(m)]
            m.sync()
            m.close()
        return out

    ref = calls()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - LEFT, dtype=torch.uint8, device="cuda")
    try:
        got = calls()
    finally:
        del hold
        torch.cuda.empty_cache()
    for a, b in zip(got, ref):
        assert np.abs(a - b).max() < 1e-9 * np.abs(b).max()
