"""The work that users of this framework have it do, as cases that can be timed.

A case is a dict: the operation (``op``), the material (lattice, nw Wannier functions, nat
atoms, shell targets of the Re and Rp sets), the precision, the sizes of the k and q lists and
the parameters.  The four named materials are the repository's own configurations (``sc`` nw = 1,
``fcc`` nw = 4, ``diamond`` nw = 8, ``hex`` nw = 5); the uneven batch draws others.  Models and
lists are made here from the seed: Hermitian hoppings and random complex vertices that decay with
|R|, force constants of a random spring network (omega^2 >= 0, acoustic sum rule), the Fermi level
at the median band energy, k lists in an energy window around it where a user would sample one.
"""
from __future__ import annotations

import functools
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_1604_03525_gb300 as epw

KB = 8.617333262e-5  # eV / K
OMEGA_MIN = 1e-5     # eV, the entry points' default
DEV = "cuda"

LATTICES = {
    "sc": (np.eye(3), np.zeros((1, 3))),
    "fcc": (np.array([[0.0, 0.5, 0.5], [0.5, 0.0, 0.5], [0.5, 0.5, 0.0]]), np.zeros((1, 3))),
    "diamond": (np.array([[0.0, 0.5, 0.5], [0.5, 0.0, 0.5], [0.5, 0.5, 0.0]]),
                np.array([[0.0, 0.0, 0.0], [0.25, 0.25, 0.25]])),
    "hex": (np.array([[1.0, 0.0, 0.0], [-0.5, math.sqrt(3.0) / 2.0, 0.0], [0.0, 0.0, 1.6]]),
            np.array([[0.0, 0.0, 0.0], [0.5, math.sqrt(3.0) / 6.0, 0.8], [0.0, math.sqrt(3.0) / 3.0, 0.8]])),
}

#: The repository's configurations: lattice, nw, nat, Re and Rp shell targets, sigma (eV), T (K).
MATERIALS = {
    "sc": dict(lattice="sc", nw=1, nat=1, nre=27, nrp=27, sigma=0.050, T=300.0),
    "fcc": dict(lattice="fcc", nw=4, nat=1, nre=120, nrp=120, sigma=0.020, T=300.0),
    "diamond": dict(lattice="diamond", nw=8, nat=2, nre=249, nrp=249, sigma=0.010, T=300.0),
    "hex": dict(lattice="hex", nw=5, nat=3, nre=300, nrp=300, sigma=0.015, T=50.0),
}


def listed():
    m = MATERIALS
    return [
        # The first call of every user: the plain FP64 method (the default precision) on a toy
        # model, 8^3 k x 8^3 q.  Latency and launches.
        dict(name="linewidth_sc_fp64", op="linewidth", prec="fp64", nk=512, nq=512, q="grid", **m["sc"]),
        # A metal's linewidths in a 0.2 eV window of E_F on a 40^3 grid, production precision.
        dict(name="linewidth_fcc_bf16x3", op="linewidth", prec="bf16x3", nk=1000, nq=64000, q="grid", **m["fcc"]),
        # The same metal in the default precision, on the coarser grid that a check or a
        # convergence study uses.
        dict(name="linewidth_fcc_fp64", op="linewidth", prec="fp64", nk=125, nq=13824, q="grid", **m["fcc"]),
        # The largest: a semiconductor's band edges on 60^3 grid points plus 10^5 random ones.
        dict(name="linewidth_diamond_bf16x3", op="linewidth", prec="bf16x3", nk=256, nq=316000, q="mixed",
             **m["diamond"]),
        # The same material on a few k and an odd number of random q, as in a convergence series.
        dict(name="linewidth_diamond_tf32x3", op="linewidth", prec="tf32x3", nk=37, nq=9001, q="random",
             **m["diamond"]),
        # A reference run for a precision sweep: the default precision, a handful of k.
        dict(name="linewidth_diamond_fp64", op="linewidth", prec="fp64", nk=24, nq=8000, q="grid", **m["diamond"]),
        # One step of fitting the vertex through the autograd interface: Im Sigma, then the gradients
        # with respect to g(Re,Rp), T and E_F.
        dict(name="grad_hex_tf32x3", op="grad", prec="tf32x3", nk=216, nq=13824, q="grid", **m["hex"]),
        # The adjoint in the default precision, as a gradient check takes it.
        dict(name="grad_hex_fp64", op="grad", prec="fp64", nk=27, nq=1728, q="grid", **m["hex"]),
        # A screening run: seven uneven systems replayed as one batch (CUDA graph).
        dict(name="batch_uneven_bf16x3", op="batch", prec="bf16x3", nk=150, nq=4096, q="grid", nsys=7, lattice="fcc",
             nw=0, nat=0, nre=0, nrp=0, sigma=0.050, T=300.0),
        # Phonon linewidths, coupling strengths and alpha^2 F of a metal: a dense k grid, few q.
        dict(name="phonon_fcc_fp64", op="phonon", prec="fp64", nk=8000, nq=216, q="grid", **m["fcc"]),
        # Spectral function along a short k path on 201 frequencies, in single precision.
        dict(name="spectral_fcc_fp32", op="spectral", prec="fp32", nk=21, nq=8000, q="grid", nomega=201, **m["fcc"]),
        # Interpolated bands, frequencies and g along a q path from a few k, on the host.
        dict(name="interp_diamond_fp64", op="interp", prec="fp64", nk=3, nq=1001, q="random", **m["diamond"]),
    ]


#: Uneven systems of the batch: nw, nat, Re target, Rp target (sizes of the repository's draw).
UNEVEN = [("sc", 1, 1, 27, 57), ("fcc", 4, 1, 120, 79), ("diamond", 8, 2, 141, 141), ("hex", 5, 3, 93, 151),
          ("sc", 2, 2, 81, 33), ("diamond", 12, 2, 55, 87), ("fcc", 18, 1, 43, 79)]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["linewidth"] * 5 + ["grad"] * 2 + ["phonon", "spectral", "interp", "batch"])
    prec = rng.choice(["fp64", "fp64", "bf16x3", "tf32x3", "fp32"])
    mat = dict(MATERIALS[rng.choice(["sc", "fcc", "diamond", "hex"])])
    if op == "linewidth" and rng.random() < 0.3:  # an uneven system: Re and Rp sets differ
        lattice, nw, nat, nre, nrp = rng.choice(UNEVEN)
        mat = dict(lattice=lattice, nw=nw, nat=nat, nre=nre, nrp=nrp, sigma=0.050, T=300.0)
    q = rng.choice(["grid", "random"])
    case = dict(op=op, prec=prec, nk=0, nq=0, q=q, **mat)
    if op == "batch":
        case = dict(op=op, prec=rng.choice(["bf16x3", "tf32x3"]), nk=_log(rng, 50, 150), nq=rng.randint(9, 16) ** 3,
                    q="grid", nsys=rng.randint(2, 7), lattice="fcc", nw=0, nat=0, nre=0, nrp=0, sigma=0.050, T=300.0)
        return case
    # pairs that cost at most about what the largest listed case of the kind does
    nm = 3 * case["nat"]
    per = 8.0 * case["nw"] ** 2 * (case["nre"] + nm * case["nrp"])  # contraction flops of a pair
    rate = {"fp64": 0.6e12, "fp32": 1.5e12, "tf32x3": 8e12, "bf16x3": 8e12}[prec]
    if case["nw"] > 8 or nm > 9:
        rate /= 4
    if op == "grad":
        rate /= 4
    if op == "spectral":
        case["nomega"] = rng.choice([64, 101, 200])
        rate /= 8
    most = 0.1 * rate / per
    if op == "interp":
        case["q"] = "random"  # points of a path: away from Gamma's zero modes
        most = min(most, 2e8 / (16.0 * nm * case["nw"] ** 2))
    most = max(2000, min(most, 4e7))
    if op == "phonon":
        case["nq"] = _log(rng, 8, 512)
        case["nk"] = max(1, min(_log(rng, 64, 20000), int(most / case["nq"])))
    else:
        case["nk"] = max(1, min(_log(rng, 1, 500 if op != "interp" else 8), int(most / 128)))
        case["nq"] = max(64, min(_log(rng, 100, 100000), int(most / case["nk"])))
    if case["q"] == "grid":
        case["nq"] = max(4, int(case["nq"] ** (1 / 3))) ** 3
    return case


# ------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=None)
def _shells(lattice, target, box):
    """Whole shells of lattice vectors by length until `target` (the 3^3 box for the toy model)."""
    A = LATTICES[lattice][0]
    r = np.arange(-box, box + 1)
    R = np.stack(np.meshgrid(r, r, r, indexing="ij"), axis=-1).reshape(-1, 3)
    length = np.round(np.linalg.norm(R @ A, axis=1), 9)
    R, length = (x[np.lexsort((R[:, 2], R[:, 1], R[:, 0], length))] for x in (R, length))
    n = target
    while n < len(R) and length[n] == length[n - 1]:
        n += 1
    return R[:n].astype(np.int32)


def _cnormal(rng, shape):
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)) / math.sqrt(2.0)


def _model(lattice, nw, nat, nre, nrp, seed):
    """H(Re), Phi(R), g(Re,Rp) as a user reads them from files (host), g also on the GPU."""
    rng = np.random.default_rng(seed)
    A, tau = LATTICES[lattice]
    tau = tau[:nat] if len(tau) >= nat else np.concatenate([tau, rng.random((nat - len(tau), 3)) @ A])
    mass = 1.0 + 0.1 * np.arange(nat)
    Re, Rp = (_shells(lattice, n, 1 if n == 27 and lattice == "sc" else 7) for n in (nre, nrp))
    nR, mid = len(Re), 0  # the shells are closed under R -> -R; R = 0 comes first
    minus = {tuple(r): i for i, r in enumerate(Re.tolist())}
    opp = np.array([minus[tuple(-r)] for r in Re])
    le, lp = np.linalg.norm(Re @ A, axis=1), np.linalg.norm(Rp @ A, axis=1)
    # hoppings of about 1 eV, on-site energies in [-1, 1] eV, H(-R) = H(R)^dagger
    X = _cnormal(rng, (nR, nw, nw)) * np.exp(-le / 0.7)[:, None, None]
    H = (X + X[opp].conj().transpose(0, 2, 1)) / math.sqrt(2.0)
    H[mid][np.diag_indices(nw)] = rng.uniform(-1, 1, nw)
    # springs: each bond a random positive stiffness; Phi(-R) = Phi(R)^T, sum_R Phi = 0 per row
    Phi = np.zeros((nR, 3 * nat, 3 * nat))
    for a in range(nat):
        for b in range(nat):
            d = np.linalg.norm(Re @ A + tau[b] - tau[a], axis=1)
            L = rng.standard_normal((nR, 3, 3))
            K = L @ L.transpose(0, 2, 1) / 3.0 * np.exp(-d / 0.7)[:, None, None]
            if a == b:
                K[mid] = 0.0
            sa, sb = slice(3 * a, 3 * a + 3), slice(3 * b, 3 * b + 3)
            Phi[:, sa, sb] -= K
            Phi[opp, sb, sa] -= K.transpose(0, 2, 1)
            Phi[mid, sa, sa] += K.sum(axis=0)
            Phi[mid, sb, sb] += K.sum(axis=0)
    Phi *= 0.1 ** 2 * mass.min() / sum(np.linalg.norm(P) for P in Phi)  # omega <= 0.1 eV
    gen = torch.Generator(device=DEV).manual_seed(seed)
    env = torch.from_numpy(0.1 * np.exp(-le[:, None] / 1.0 - lp[None, :] / 1.5)).to(DEV)
    g = torch.randn((nR, len(Rp), 3 * nat, nw, nw), dtype=torch.complex128, device=DEV, generator=gen)
    g *= env[:, :, None, None, None]
    return SimpleNamespace(lattice=lattice, nw=nw, nat=nat, mass=mass, Re=Re, wRe=np.ones(nR), H=H, Rph=Re,
                           wRph=np.ones(nR), Phi=Phi.astype(np.complex128), Rp=Rp, wRp=np.ones(len(Rp)),
                           g=g.cpu().numpy(), g_gpu=g)


def _grid(n):
    i = np.arange(n) / n
    return np.stack(np.meshgrid(i, i, i, indexing="ij"), axis=-1).reshape(-1, 3)


def _qlist(kind, nq, rng):
    if kind == "grid":
        return _grid(round(nq ** (1 / 3)))
    if kind == "mixed":  # a uniform grid plus random points, all with the same weight
        n = int((nq * 0.7) ** (1 / 3) + 1e-9)
        return np.concatenate([_grid(n), rng.random((nq - n ** 3, 3))])
    return rng.random((nq, 3))


def _bands(wm, k):
    ph = np.exp(2j * np.pi * (k @ wm.Re.T))
    return np.linalg.eigvalsh(np.tensordot(ph, wm.H, axes=(1, 0)))


def _lists(case, wm, seed):
    """E_F at the median band energy; k in a window of E_F (the whole zone for the phonon side)."""
    rng = np.random.default_rng(seed + 1)
    EF = float(np.median(_bands(wm, _grid(6))))
    q = _qlist(case["q"], case["nq"], rng)
    nk = case["nk"]
    if case["op"] == "phonon" or case["nw"] == 1:
        n = round(nk ** (1 / 3))
        k = _grid(n) + rng.random(3) / n if n ** 3 == nk else rng.random((nk, 3))
    elif case["op"] in ("spectral", "interp"):  # a path through the zone
        a, b = rng.random((2, 3))
        k = a + (b - a) * np.linspace(0.0, 1.0, nk)[:, None]
    else:
        k = rng.random((4 * nk + 64, 3))
        near = np.abs(_bands(wm, k) - EF).min(axis=1)
        k = k[np.sort(np.argsort(near, kind="stable")[:nk])]
    return k, q, EF


def _systems(case, seed):
    """The batch's systems: sizes fixed by the case, k counts uneven."""
    out = []
    for i, (lattice, nw, nat, nre, nrp) in enumerate(UNEVEN[:case["nsys"]]):
        c = dict(case, op="linewidth", lattice=lattice, nw=nw, nat=nat, nre=nre, nrp=nrp)
        c["nk"] = max(1, case["nk"] * (1, 4, 2, 3, 4, 1, 1)[i] // (1 if nw < 12 else 4))
        out.append((c, seed * 16 + i))
    return out


def _inputs(case, seed):
    seed = 2 * seed + 160403525
    wm = _model(case["lattice"], case["nw"], case["nat"], case["nre"], case["nrp"], seed)
    k, q, EF = _lists(case, wm, seed)
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(DEV)  # noqa: E731
    nk = len(k)
    s = SimpleNamespace(case=case, wm=wm, k=dev(k), q=dev(q), EF=EF, T=case["T"], sigma=case["sigma"],
                        prec=epw.PRECISIONS[case["prec"]])
    if case["op"] == "grad":
        s.cot = dev(np.random.default_rng(seed + 2).standard_normal((nk, case["nw"])))
    if case["op"] == "spectral":
        s.omega, s.delta = dev(np.linspace(-0.5, 0.5, case["nomega"])), 0.02
    if case["op"] == "phonon":
        s.grid, s.sigma_ph = dev(np.linspace(0.0, 0.12, 241)), 0.002
    return s


def prepare(case, seed):
    if case["op"] == "batch":
        states = [prepare(c, sd) for c, sd in _systems(case, seed)]
        batch = epw.Batch([dict(model=s.model, k=s.k, q=s.q, T=s.T, EF=s.EF, sigma=s.sigma, precision=s.prec)
                           for s in states])
        return SimpleNamespace(case=case, states=states, batch=batch)
    s = _inputs(case, seed)
    s.model = epw.Model(s.wm)
    if case["op"] == "grad":
        s.g = s.wm.g_gpu.requires_grad_(True)
        # T and E_F as host scalars that are fitted too
        s.Tt = torch.tensor(s.T, dtype=torch.float64, requires_grad=True)
        s.Et = torch.tensor(s.EF, dtype=torch.float64, requires_grad=True)
    s.wm.g = s.wm.g_gpu = None  # a user's program lets the host copy go
    return s


def run(s):
    op = s.case["op"]
    if op == "batch":
        return list(s.batch.run())
    par = dict(T=s.T, EF=s.EF, precision=s.prec)
    if op == "linewidth":
        return s.model.linewidth(s.k, s.q, sigma=s.sigma, **par)
    if op == "grad":
        out = _autograd().linewidth(s.model, s.g, s.Tt, s.Et, s.k, s.q, sigma=s.sigma, precision=s.prec)
        return [out.detach(), *torch.autograd.grad(out, (s.g, s.Tt, s.Et), grad_outputs=s.cot)]
    if op == "phonon":
        pi, lam, nesting, dos = s.model.phonon_selfenergy(s.k, s.q, sigma=s.sigma, **par)
        omega = torch.from_numpy(s.model.interp(s.k[:1], s.q, precision=s.prec, want_g=False)[2]).to(DEV)
        return [pi, lam, nesting, dos, epw.eliashberg(omega, lam, s.grid, s.sigma_ph)]
    if op == "spectral":
        return list(s.model.selfenergy(s.k, s.q, s.omega, delta=s.delta, **par))
    return list(s.model.interp(s.k, s.q, precision=s.prec))


def _autograd():
    from paper_1604_03525_gb300 import autograd
    return autograd


# -------------------------------------------------------------------- work
def _count(c):
    nre, nrp = (len(_shells(c["lattice"], n, 1 if n == 27 and c["lattice"] == "sc" else 7))
                for n in (c["nre"], c["nrp"]))
    nw, nm, nk, nq = c["nw"], 3 * c["nat"], c["nk"], c["nq"]
    ng = nre * nrp * nm * nw * nw
    # per pair: H(k+q) and g(k,q) U_k; per k: g(Re,Rp) -> g(k,Rp), and its rotation by U_k
    pair = 8.0 * nw * nw * (nre + nm * nrp)
    flops = nk * nq * pair + 8.0 * nk * (ng + nrp * nm * nw ** 3) + 8.0 * nq * nre * nm * nm
    read = 16 * (nre * (nw * nw + nm * nm) + ng) + 24 * (nk + nq)
    write = 8 * nk * nw
    if c["op"] == "grad":  # the forward, its recomputation, the adjoint of the vertex contraction
        flops += nk * nq * (pair + 8.0 * nw * nw * nm * nrp) + 16.0 * nk * ng
        write += 16 * ng
    elif c["op"] == "phonon":
        write = 8 * nq * (2 * nm + 1) + 8
    elif c["op"] == "spectral":
        flops += 4.0 * nk * nq * nm * nw * nw * c["nomega"]
        write = 24 * nk * nw * c["nomega"]
    elif c["op"] == "interp":
        flops += 8.0 * nk * nq * nm * (nw ** 3 + nm * nw * nw)
        write = 8 * (nk * nw + nk * nq * nw + nq * nm) + 16 * nk * nq * nm * nw * nw
    return {"bytes": float(read + write), "flops": flops}


def work(case):
    if case["op"] == "batch":
        parts = [_count(c) for c, _ in _systems(case, 0)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    return _count(case)


# ------------------------------------------------------------------- exact
def _phase(x, R):
    a = x @ torch.from_numpy(R.astype(np.float64)).to(DEV).T
    return torch.polar(torch.ones_like(a), 2 * math.pi * (a - torch.round(a)))


def _phonons(s):
    wm = s.wm
    P = _phase(s.q, wm.Re)
    msq = np.repeat(np.sqrt(wm.mass), 3)
    Phi = torch.from_numpy(wm.Phi / np.outer(msq, msq)).to(DEV)
    w2, e = torch.linalg.eigh((P @ Phi.reshape(len(wm.Re), -1)).reshape(len(s.q), 3 * wm.nat, -1))
    om = torch.sign(w2) * torch.sqrt(torch.abs(w2))
    keep = om >= OMEGA_MIN
    m = torch.from_numpy(np.repeat(wm.mass, 3)).to(DEV)
    E = e / torch.sqrt(2.0 * m[None, :, None] * torch.where(keep, om, torch.ones_like(om))[:, None, :])
    return om, keep, E * keep[:, None, :]


def _pairs(s, g):
    """For each k and each block of q: slices, e_k, e_k+q, |g|^2 [q, nu, m, n] (differentiable in g)."""
    wm = s.wm
    nw, nm = wm.nw, 3 * wm.nat
    H = torch.from_numpy(wm.H).to(DEV).reshape(len(wm.Re), -1)
    om, keep, E = _phonons(s)
    Pk = _phase(s.k, wm.Re)
    ek, Uk = torch.linalg.eigh((Pk @ H).reshape(-1, nw, nw))
    step = max(1, int(2.5e8 / (16 * nm * nw * nw)))
    for i in range(len(s.k)):
        G = torch.tensordot(Pk[i], g, dims=1) @ Uk[i]  # [Rp, alpha, j, n]
        Hk = Pk[i][:, None] * H
        for a in range(0, len(s.q), step):
            b = slice(a, min(a + step, len(s.q)))
            ekq, U = torch.linalg.eigh((_phase(s.q[b], wm.Re) @ Hk).reshape(-1, nw, nw))
            X = (_phase(s.q[b], wm.Rp) @ G.reshape(len(wm.Rp), -1)).reshape(-1, nm, nw, nw)
            Y = U.conj().transpose(1, 2)[:, None] @ X
            gm = torch.einsum("qav,qamn->qvmn", E[b], Y)
            yield i, b, ek[i], ekq, gm.real ** 2 + gm.imag ** 2, om[b], keep[b]


def _occ(e, EF, T):
    return torch.sigmoid(-(e - EF) / (KB * T))


def _bose(om, keep, T):
    return torch.where(keep, 1.0 / torch.expm1(torch.where(keep, om, torch.ones_like(om)) / (KB * T)), 0.0)


def _delta(x, sigma):
    return torch.exp(-(x / sigma) ** 2) / (sigma * math.sqrt(math.pi))


def _linewidth(s, g, T, EF, each=None):
    out = torch.zeros((len(s.k), s.wm.nw), dtype=torch.float64, device=DEV)
    for i, b, ek, ekq, g2, om, keep in _pairs(s, g):
        n, f = _bose(om, keep, T)[:, :, None, None], _occ(ekq, EF, T)[:, None, :, None]
        x, w = (ek[None, None, None, :] - ekq[:, None, :, None]), om[:, :, None, None]
        t = g2 * ((n + f) * _delta(x + w, s.sigma) + (n + 1 - f) * _delta(x - w, s.sigma))
        row = math.pi / len(s.q) * (t * keep[:, :, None, None]).sum(dim=(0, 1, 2))
        if each is not None:
            each(i, row)
        out[i] += row.detach()
    return out


def _spectral(s):
    nk, nw, nom = len(s.k), s.wm.nw, len(s.omega)
    om0 = torch.cat([s.omega, torch.zeros(1, dtype=torch.float64, device=DEV)])
    sig = torch.zeros((nk, nw, nom + 1), dtype=torch.complex128, device=DEV)
    eks = torch.zeros((nk, nw), dtype=torch.float64, device=DEV)
    for i, b, ek, ekq, g2, om, keep in _pairs(s, s.wm.g_gpu):
        eks[i] = ek
        n, f = _bose(om, keep, s.T)[:, :, None], _occ(ekq, s.EF, s.T)[:, None, :]
        for j in range(nom + 1):
            x = om0[j] - (ekq[:, None, :] - s.EF) + 1j * s.delta
            L = (n + f) / (x + om[:, :, None]) + (n + 1 - f) / (x - om[:, :, None])
            L = L * keep[:, :, None] / len(s.q)
            sig[i, :, j] += torch.einsum("qvm,qvmn->n", L, g2.to(torch.complex128))
    s2, re = -sig.imag[..., :nom], sig.real[..., :nom] - sig.real[..., nom:]
    den = s.omega - (eks - s.EF)[..., None] - re
    return [sig[..., :nom].contiguous(), s2.abs() / (math.pi * (den ** 2 + s2 ** 2))]


def _phonon_side(s):
    nq, nm = len(s.q), 3 * s.wm.nat
    pi, lam = (torch.zeros((nq, nm), dtype=torch.float64, device=DEV) for _ in range(2))
    nest, dos = torch.zeros(nq, dtype=torch.float64, device=DEV), torch.zeros(1, dtype=torch.float64, device=DEV)
    omega = _phonons(s)[0]
    for i, b, ek, ekq, g2, om, keep in _pairs(s, s.wm.g_gpu):
        dn, dm = _delta(ek - s.EF, s.sigma), _delta(ekq - s.EF, s.sigma)
        df = (_occ(ek, s.EF, s.T)[None, None, :] - _occ(ekq, s.EF, s.T)[:, :, None])[:, None]
        x = ek[None, None, None, :] - ekq[:, None, :, None] - om[:, :, None, None]
        k4 = keep.to(torch.float64)
        pi[b] += (g2 * df * _delta(x, s.sigma)).sum(dim=(2, 3)) * k4
        z = dm[:, :, None] * dn[None, None, :]
        lam[b] += (g2 * z[:, None]).sum(dim=(2, 3)) * k4
        nest[b] += z.sum(dim=(1, 2))
        if b.start == 0:
            dos += dn.sum()
    nk = len(s.k)
    pi, lam, nest, dos = 2 * math.pi * pi / nk, lam / nk, nest / nk, dos / nk
    lam = torch.where(lam > 0, lam / (dos * torch.where(lam > 0, omega, torch.ones_like(omega))), 0.0)
    a2f = torch.stack([(0.5 / nq * omega * lam * _delta(x - omega, s.sigma_ph)).sum() for x in s.grid])
    return [pi, lam, nest, dos, a2f]


def exact(case, seed):
    if case["op"] == "batch":
        return [exact(c, sd) for c, sd in _systems(case, seed)]
    pairs = case["nk"] * case["nq"]
    if pairs > 2.5e6 or pairs * case["nw"] ** 2 > 4e7 or pairs * case["nw"] ** 2 * case["nat"] > 8e7 or (
            case["op"] == "spectral" and pairs * case["nomega"] > 4e7):
        return None  # too long in 64 bits
    s = _inputs(case, seed)
    if case["op"] == "linewidth":
        return _linewidth(s, s.wm.g_gpu, s.T, s.EF)
    if case["op"] == "grad":
        g = s.wm.g_gpu.requires_grad_(True)
        T = torch.tensor(s.T, dtype=torch.float64, device=DEV, requires_grad=True)
        EF = torch.tensor(s.EF, dtype=torch.float64, device=DEV, requires_grad=True)
        out = _linewidth(s, g, T, EF, each=lambda i, row: (row * s.cot[i]).sum().backward())
        return [out, g.grad, T.grad, EF.grad]
    if case["op"] == "phonon":
        return _phonon_side(s)
    if case["op"] == "spectral":
        return _spectral(s)
    eps = torch.stack([torch.linalg.eigvalsh((_phase(k + s.q, s.wm.Re) @ torch.from_numpy(s.wm.H).to(DEV).reshape(
        len(s.wm.Re), -1)).reshape(-1, s.wm.nw, s.wm.nw)) for k in s.k])
    ek = torch.from_numpy(_bands(s.wm, s.k.cpu().numpy()))
    return [ek, eps, _phonons(s)[0], None]  # g depends on the eigenvectors' phases
