"""The work this library is measured on: its public calls over the sizes, forms
and options its users run, with seeded inputs made on the GPU and the same
results in plain 64-bit torch.

A case is a dict of plain values; ``kind`` names the call:

* ``apply``        ``FockPlan.apply``: V_x psi, E_x (and dE_x/domega) of a Gamma-point set
* ``fixed``        ``FockPlan.apply_fixed``: V_x fixed by an occupied set, on trial orbitals
* ``kpoints``      ``FockKPlan.apply``: Bloch orbitals on a k mesh
* ``batch``        ``FockBatch.run``: uneven systems as one graph
* ``grad``         ``autograd.exchange_energy``, forward and backward
* ``sternheimer``  ``FockPlan.sternheimer``: linear-response CG

``prec`` is the form (0 FP64, 1 mixed, 2 double-float).  The mixed form works in
complex64, so its results are handed on at that width (complex64 and float32),
as a program that chose the form keeps them.  ``batch`` / ``block`` /
``streams`` are the plan's pair-loop settings, 0 for its defaults; the large
Gamma-point cases use the ones the autotuner settles on.
"""

import itertools
import math

import numpy as np
import torch

from paper_1305_7313_gb300 import ERFC, SPENCER_ALAVI, FockBatch, FockKPlan, FockPlan
from paper_1305_7313_gb300.autograd import exchange_energy

FP64, MIXED, DF64 = 0, 1, 2
# grid sizes a drawn case takes, and the cell the workloads give a grid: L = 27 N / 96 at 12 Ha
GRIDS = (24, 32, 36, 48, 64, 72, 96)


def _case(kind, name=None, **kw):
    c = dict(kind=kind, N=48, L=13.5, ecut=12.0, nb=16, prec=FP64, omega=0.0, dex=False, uneven=False,
             skew=False, batch=0, block=0, streams=0)
    c.update(kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest system of the workloads (a few water-like orbitals): latency and launches count
        _case("apply", "apply_fp64_n24_b8", N=24, L=10.0, ecut=10.0, nb=8),
        # a medium cell inside a hybrid-functional SCF step, mixed form, fractional
        # occupations, an odd number of bands, and the screening derivative asked for
        _case("apply", "apply_mixed_n48_b37", nb=37, prec=MIXED, omega=0.106, dex=True, uneven=True),
        # a general (triclinic) cell in FP64 with fractional occupations and an odd number of bands
        _case("apply", "apply_fp64_n64_b31", N=64, L=18.0, nb=31, omega=0.3, dex=True, uneven=True, skew=True),
        # the reference-accuracy ground state: large cell, FP64, closed shell, tuned settings
        _case("apply", "apply_fp64_n96_b48", N=96, L=27.0, nb=48, batch=76, block=8, streams=2),
        # the same cell in double-float arithmetic
        _case("apply", "apply_df64_n96_b64", N=96, L=27.0, nb=64, prec=DF64, batch=76, block=32, streams=4),
        # the production hybrid step: large cell, hundreds of bands, mixed form, tuned settings (the largest case)
        _case("apply", "apply_mixed_n96_b256", N=96, L=27.0, nb=256, prec=MIXED, omega=0.106, batch=76, block=8,
              streams=4),
        # the inner SCF loop: V_x fixed by the occupied set, applied to a block of trial orbitals
        _case("fixed", "fixed_mixed_n96_b96_t41", N=96, L=27.0, nb=96, nt=41, prec=MIXED, omega=0.106),
        # a small cell sampled at two k points in FP64
        _case("kpoints", "kpoints_fp64_n24_k2_b6", N=24, L=9.0, ecut=8.0, nb=6, mesh="1,1,2", uneven=True),
        # a small cell on a 2 x 2 x 2 mesh, mixed form
        _case("kpoints", "kpoints_mixed_n48_k8_b32", nb=32, prec=MIXED, omega=0.106, mesh="2,2,2"),
        # many independent snapshots or images of different sizes in one graph
        _case("batch", "batch_mixed_6_systems", prec=MIXED, grids="48,48,64,64,72,96", bands="33,96,17,80,57,24"),
        # orbital optimisation: the energy and its gradient with respect to the orbitals and omega
        _case("grad", "grad_mixed_n72_b128", N=72, L=20.0, nb=128, prec=MIXED, omega=0.106),
        # linear response on top of the ground state
        _case("sternheimer", "sternheimer_fp64_n48_32", nb=32, nrhs=32),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# the most bands a drawn apply takes on a grid, so that it costs no more than the largest listed case
_MOST = {MIXED: {24: 512, 32: 512, 36: 512, 48: 384, 64: 320, 72: 256, 96: 192},
         FP64: {24: 256, 32: 192, 36: 160, 48: 128, 64: 80, 72: 64, 96: 40},
         DF64: {24: 256, 32: 256, 36: 224, 48: 192, 64: 128, 72: 96, 96: 64}}


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "fixed", "kpoints", "batch", "grad", "sternheimer"])
    N = rng.choice(GRIDS)
    prec = rng.choice([FP64, MIXED, MIXED, DF64] if kind in ("apply", "fixed") else [FP64, MIXED])
    L = round(27.0 * N / 96.0 * rng.uniform(0.9, 1.0), 3)
    omega = rng.choice([0.0, 0.106, 0.3])
    if kind == "apply":
        tuned = rng.random() < 0.5
        return _case("apply", N=N, L=L, nb=_logint(rng, 3, _MOST[prec][N]), prec=prec, omega=omega,
                     dex=omega > 0 and rng.random() < 0.5, uneven=rng.random() < 0.4, skew=rng.random() < 0.25,
                     batch=76 if tuned else 0, block=8 if tuned else 0, streams=rng.choice([2, 3, 4]) if tuned else 0)
    if kind == "fixed":
        most = _MOST[prec][N] // 2
        return _case("fixed", N=N, L=L, nb=_logint(rng, 3, most), nt=_logint(rng, 1, most), prec=prec, omega=omega,
                     uneven=rng.random() < 0.4)
    if kind == "kpoints":
        N = rng.choice([24, 32, 36, 48])
        mesh = rng.choice(["1,1,1", "1,1,2", "1,2,2", "2,2,2"])
        nk = math.prod(int(m) for m in mesh.split(","))
        most = max(2, (_MOST[prec][N] if prec == FP64 else 256) // (2 * nk))
        return _case("kpoints", N=N, L=round(27.0 * N / 96.0 * rng.uniform(0.8, 0.9), 3), nb=_logint(rng, 1, most),
                     prec=prec, omega=omega, mesh=mesh, uneven=rng.random() < 0.4)
    if kind == "batch":
        n = rng.randint(2, 8)
        grids = [rng.choice([24, 32, 48, 64, 72, 96]) for _ in range(n)]
        bands = [_logint(rng, 5, _MOST[MIXED][g] // 3) for g in grids]
        return _case("batch", prec=MIXED, grids=",".join(map(str, grids)), bands=",".join(map(str, bands)))
    if kind == "grad":
        return _case("grad", N=N, L=L, nb=_logint(rng, 4, _MOST[MIXED][N] * 3 // 4), prec=MIXED, omega=omega or 0.2)
    N = rng.choice([24, 32, 36, 48, 64])
    return _case("sternheimer", N=N, L=round(27.0 * N / 96.0 * rng.uniform(0.9, 1.0), 3), nb=rng.randint(4, 48),
                 nrhs=rng.randint(4, 48))


# ------------------------------------------------------------------- inputs


def _cell(case, L=None):
    L = case["L"] if L is None else L
    a = L * np.eye(3)
    if case["skew"]:
        a = a + L * np.array([[0.0, 0.04, 0.0], [0.03, 0.0, 0.02], [0.0, -0.03, 0.0]])
    return a


def _recip(cell):
    c23, c31, c12 = np.cross(cell[1], cell[2]), np.cross(cell[2], cell[0]), np.cross(cell[0], cell[1])
    vol = (cell[0, 0] * c23[0] + cell[0, 1] * c23[1]) + cell[0, 2] * c23[2]
    return np.stack([c23, c31, c12]) * (2.0 * 3.14159265358979323846 / vol), abs(vol)


def _g2(b, m, k=(0.0, 0.0, 0.0)):
    u = [m[..., a] + k[a] for a in range(3)]
    c = [(u[0] * b[0, x] + u[1] * b[1, x]) + u[2] * b[2, x] for x in range(3)]
    return (c[0] * c[0] + c[1] * c[1]) + c[2] * c[2]


def _sphere(cell, ecut, k=(0.0, 0.0, 0.0)):
    """Miller indices and |k + G|^2 in the library's documented order: by |k + G|^2, then m1, m2, m3."""
    b, _ = _recip(cell)
    mx = [int(math.sqrt(2 * ecut) * np.linalg.norm(cell[a]) / (2 * math.pi) + abs(k[a])) + 1 for a in range(3)]
    m = np.stack(np.meshgrid(*[np.arange(-x, x + 1) for x in mx], indexing="ij"), -1).reshape(-1, 3)
    g2 = _g2(b, m.astype(np.float64), k)
    m, g2 = m[g2 <= 2 * ecut], g2[g2 <= 2 * ecut]
    o = np.lexsort((m[:, 2], m[:, 1], m[:, 0], g2))
    return m[o], g2[o]


def _orthonormal(c, real):
    s = c.conj() @ c.T
    w, u = np.linalg.eigh((s.real if real else s).cpu().numpy())
    x = torch.from_numpy((u / np.sqrt(w)) @ u.conj().T).to(c.device)
    return x.T.to(c.dtype) @ c


def _orbitals(m, g2, nb, seed, real=True):
    """Orthonormal orbitals c(G) ~ N(0, 1) exp(-|k + G|^2 / 4); real: c(-G) = c(G)*."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    c = torch.view_as_complex(torch.randn(nb, len(m), 2, generator=gen, device="cuda", dtype=torch.float64))
    c = c * torch.exp(-0.25 * torch.from_numpy(g2).cuda())
    if not real:
        return _orthonormal(c, False).contiguous()
    key = ((m[:, 0] + 512) * 1024 + m[:, 1] + 512) * 1024 + m[:, 2] + 512
    neg = ((512 - m[:, 0]) * 1024 + 512 - m[:, 1]) * 1024 + 512 - m[:, 2]
    o = np.argsort(key)
    mir = torch.from_numpy(o[np.searchsorted(key, neg, sorter=o)]).cuda()
    c = 0.5 * (c + c[:, mir].conj())
    c = _orthonormal(c, True)
    return (0.5 * (c + c[:, mir].conj())).contiguous()


def _occ(case, n, seed):
    if not case["uneven"]:
        return np.full(n, 2.0)
    return np.sort(np.random.default_rng(seed + 5).uniform(0.05, 2.0, n))[::-1].copy()


def _mesh(case):
    n = [int(x) for x in case["mesh"].split(",")]
    k = np.array(list(itertools.product(*[[i / m for i in range(m)] for m in n])))
    w = np.full(len(k), 1.0 / len(k))
    return k, w


def _systems(case):
    g, b = [[int(x) for x in case[key].split(",")] for key in ("grids", "bands")]
    return [(n, 27.0 * n / 96.0, nb) for n, nb in zip(g, b)]


def _potential(case, cell, seed):
    """Three Gaussian wells on the grid, float64 [N, N, N] on the device."""
    n = case["N"]
    r = np.random.default_rng(seed + 7)
    f = torch.stack(torch.meshgrid(*[torch.arange(n, device="cuda", dtype=torch.float64) / n] * 3, indexing="ij"), -1)
    a = torch.from_numpy(cell).cuda()
    v = torch.zeros(n, n, n, device="cuda", dtype=torch.float64)
    for _ in range(3):
        d = f - torch.from_numpy(r.random(3)).cuda()
        d = (d - torch.round(d)) @ a
        v = v - 1.5 * torch.exp(-(d * d).sum(-1) / (2 * 0.9 ** 2))
    return v.contiguous()


def _response(case, seed):
    cell = _cell(case)
    m, g2 = _sphere(cell, case["ecut"])
    v = _potential(case, cell, seed)
    u = _orbitals(m, g2, case["nb"], seed)
    scale = 10.0 ** (-2.0 * (np.arange(case["nrhs"]) % 4))
    w = (_orbitals(m, g2, case["nrhs"], seed + 1) * torch.from_numpy(scale).cuda()[:, None]).contiguous()
    eps = float(v.min()) - 1.0 - 0.01 * np.arange(case["nrhs"])
    return dict(cell=cell, m=m, g2=g2, v=v, u=u, w=w, eps=eps, alpha=1.0, tol=1e-8)


def _kind(case):
    return (SPENCER_ALAVI, None) if case["omega"] == 0 else (ERFC, case["omega"])


def prepare(case, seed):
    kernel, omega = _kind(case)
    cell, kind = _cell(case), case["kind"]
    if kind == "batch":
        plans, psi, occ = [], [], []
        for s, (n, L, nb) in enumerate(_systems(case)):
            c = _cell(case, L)
            plans.append(FockPlan(n, c.ravel(), case["ecut"], kernel, omega, case["prec"]))
            psi.append(_orbitals(*_sphere(c, case["ecut"]), nb, seed + 100 * s))
            occ.append(np.full(nb, 2.0))
        torch.cuda.synchronize()
        return dict(case=case, batch=FockBatch(plans, psi, occ, persistent=0))
    if kind == "kpoints":
        k, w = _mesh(case)
        plan = FockKPlan(case["N"], cell.ravel(), case["ecut"], k, w, kernel, omega, case["prec"])
        psi = [_orbitals(*_sphere(cell, case["ecut"], kk), case["nb"], seed + 100 * i, real=False)
               for i, kk in enumerate(k)]
        occ = np.stack([_occ(case, case["nb"], seed + i) for i in range(len(k))])
        return dict(case=case, plan=plan, psi=psi, occ=occ)
    if kind == "grad":
        psi = _orbitals(*_sphere(cell, case["ecut"]), case["nb"], seed).to(torch.complex64)
        return dict(case=case, cell=cell.ravel(), kernel=kernel, psi=psi, occ=_occ(case, case["nb"], seed))
    plan = FockPlan(case["N"], cell.ravel(), case["ecut"], kernel, omega, case["prec"])
    if kind == "sternheimer":
        return dict(case=case, plan=plan, **_response(case, seed))
    if case["batch"]:
        plan.set_batch(case["batch"])
    if case["block"]:
        plan.set_band_block(case["block"])
    if case["streams"]:
        plan.set_streams(case["streams"])
    m, g2 = _sphere(cell, case["ecut"])
    st = dict(case=case, plan=plan, psi=_orbitals(m, g2, case["nb"], seed), occ=_occ(case, case["nb"], seed))
    if kind == "fixed":
        st["phi"] = _orbitals(m, g2, case["nt"], seed + 1)
        plan.set_occupied(st["psi"], st["occ"])
    return st


def run(state):
    case = state["case"]
    kind, mixed = case["kind"], case["prec"] == MIXED
    array = (lambda t: t.to(torch.complex64)) if mixed else (lambda t: t)
    number = np.float32 if mixed else np.float64
    if kind == "apply":
        v, e, d = state["plan"].apply(state["psi"], state["occ"], want_dex=case["dex"])
        out = {"vpsi": array(v), "ex": number(e)}
        if case["dex"]:
            out["dex"] = number(d)
        return out
    if kind == "fixed":
        return {"vphi": array(state["plan"].apply_fixed(state["phi"]))}
    if kind == "kpoints":
        v, e = state["plan"].apply(state["psi"], state["occ"])
        return {"vpsi": [array(x) for x in v], "ex": number(e)}
    if kind == "batch":
        e, _ = state["batch"].run()
        return {"vpsi": [array(x) for x in state["batch"].vpsi], "ex": np.asarray(e, dtype=number)}
    if kind == "grad":
        psi = state["psi"].detach().requires_grad_(True)
        omega = torch.tensor(case["omega"], dtype=torch.float64, requires_grad=True)
        e = exchange_energy(psi, state["occ"], case["N"], state["cell"], case["ecut"], state["kernel"], omega,
                            case["prec"])
        e.backward()
        return {"ex": e.detach().to(torch.float32), "psi_grad": psi.grad, "omega_grad": omega.grad.to(torch.float32)}
    g, iters, resid = state["plan"].sternheimer(state["v"], state["u"], state["eps"], state["w"], state["alpha"],
                                                state["tol"])
    return {"g": g, "iters": iters, "resid": resid}


# ------------------------------------------------ what a pass cannot do without


def _npw(case, L=None):
    _, vol = _recip(_cell(case, L))
    return vol * (2 * case["ecut"]) ** 1.5 / (6 * math.pi ** 2)


def work(case):
    """Bytes: the coefficients (and potential) read once and the results written
    once; flops: the transforms, 5 n log2 n per complex transform, two pair
    densities per complex transform at the Gamma point, forward and back."""
    fft = lambda n: 5.0 * n ** 3 * 3 * math.log2(n)  # noqa: E731
    kind, nb = case["kind"], case["nb"]
    if kind == "batch":
        w = {"bytes": 0.0, "flops": 0.0}
        for n, L, b in _systems(case):
            w["bytes"] += 2 * 16.0 * b * _npw(case, L)
            w["flops"] += (b * (b + 1) / 2 + b) * fft(n)
        return w
    npw, f = _npw(case), fft(case["N"])
    if kind == "kpoints":
        ns = nb * math.prod(int(x) for x in case["mesh"].split(","))
        return {"bytes": 2 * 16.0 * ns * npw, "flops": (ns * (ns + 1) + 2 * ns) * f}
    if kind == "fixed":
        return {"bytes": 16.0 * (2 * case["nt"] + nb) * npw, "flops": (nb * case["nt"] + case["nt"]) * f}
    if kind == "sternheimer":  # about ten applications of H a ket, two real kets per complex transform
        return {"bytes": 16.0 * (nb + 2 * case["nrhs"]) * npw + 8.0 * case["N"] ** 3, "flops": 10.0 * case["nrhs"] * f}
    width = 8.0 if kind == "grad" else 16.0
    return {"bytes": 2 * width * nb * npw, "flops": (nb * (nb + 1) / 2 + nb) * f}


# --------------------------------------------------------- the same in 64 bits


def _kernel(g2, vol, omega):
    """v(G) and dv/domega: truncated Coulomb (omega = 0) or erfc-screened."""
    zero = g2 == 0
    s = torch.where(zero, torch.ones_like(g2), g2)
    if omega == 0:
        rc = (3 * vol / (4 * math.pi)) ** (1.0 / 3.0)
        v = 8 * math.pi * torch.sin(0.5 * torch.sqrt(s) * rc) ** 2 / s
        return torch.where(zero, torch.full_like(v, 2 * math.pi * rc * rc), v), torch.zeros_like(v)
    v = -4 * math.pi * torch.expm1(-s / (4 * omega * omega)) / s
    v = torch.where(zero, torch.full_like(v, math.pi / omega ** 2), v)
    return v, -(2 * math.pi / omega ** 3) * torch.exp(-g2 / (4 * omega * omega))


def _table(cell, n, omega, q=(0.0, 0.0, 0.0), half=False):
    b, vol = _recip(cell)
    f = np.fft.fftfreq(n, 1.0 / n)
    last = np.abs(np.fft.rfftfreq(n, 1.0 / n)) if half else f
    m = np.stack(np.meshgrid(f, f, last, indexing="ij"), -1)
    return _kernel(torch.from_numpy(_g2(b, m, q)).cuda(), vol, omega)


def _real_space(c, m, n, vol):
    i = torch.from_numpy(((m[:, 0] % n) * n + m[:, 1] % n) * n + m[:, 2] % n).cuda()
    x = torch.zeros(len(c), n ** 3, dtype=torch.complex128, device="cuda")
    x[:, i] = c
    return torch.fft.ifftn(x.view(-1, n, n, n), dim=(1, 2, 3)) * (n ** 3 / math.sqrt(vol)), i


def _sphere_of(w, i, n, vol):
    out = []
    for k in range(0, len(w), 16):
        out.append(torch.fft.fftn(w[k:k + 16].to(torch.complex128), dim=(1, 2, 3)).view(-1, n ** 3)[:, i])
    return torch.cat(out) * (math.sqrt(vol) / n ** 3)


def _exact_gamma(c, occ, cell, ecut, n, omega, trial=None):
    m, _ = _sphere(cell, ecut)
    _, vol = _recip(cell)
    v, dv = _table(cell, n, omega, half=True)
    wgt = torch.full((n // 2 + 1,), 2.0, dtype=torch.float64, device="cuda")
    wgt[0] = wgt[-1] = 1.0
    psi, i = _real_space(c, m, n, vol)
    psi = psi.real.contiguous()
    f = torch.from_numpy(np.ascontiguousarray(occ)).cuda()
    other = psi if trial is None else _real_space(trial, m, n, vol)[0].real.contiguous()
    w = torch.zeros_like(other)
    e = torch.zeros(2, dtype=torch.float64, device="cuda")
    step = max(1, min(64, (1 << 25) // n ** 3))
    for a in range(len(psi)):
        j0 = a if trial is None else 0
        for j in range(j0, len(other), step):
            k = slice(j, min(j + step, len(other)))
            rho = torch.fft.rfftn(psi[a] * other[k], dim=(1, 2, 3))
            if trial is None:
                p = (rho.real ** 2 + rho.imag ** 2) * wgt
                both = f[a] * f[k] * torch.where(torch.arange(k.start, k.stop, device="cuda") == a, 1.0, 2.0)
                e[0] += (both * (p * v).sum((1, 2, 3))).sum()
                e[1] += (both * (p * dv).sum((1, 2, 3))).sum()
            phi = torch.fft.irfftn(rho * v, s=(n, n, n), dim=(1, 2, 3))
            w[k] -= f[a] * psi[a] * phi
            if trial is None:
                g = f[k].clone()
                g[torch.arange(k.start, k.stop, device="cuda") == a] = 0.0
                w[a] -= torch.einsum("j,jxyz,jxyz->xyz", g, other[k], phi)
    e = e * (-0.5 * vol / float(n) ** 6)
    return _sphere_of(w, i, n, vol), float(e[0]), float(e[1])


def _exact_k(case, seed):
    cell, n = _cell(case), case["N"]
    _, vol = _recip(cell)
    kpt, wk = _mesh(case)
    u, idx, f = [], [], []
    for a, kk in enumerate(kpt):
        m, g2 = _sphere(cell, case["ecut"], kk)
        x, i = _real_space(_orbitals(m, g2, case["nb"], seed + 100 * a, real=False), m, n, vol)
        u.append(x)
        idx.append(i)
        f.append(torch.from_numpy(wk[a] * _occ(case, case["nb"], seed + a)).cuda())
    w = [torch.zeros_like(x) for x in u]
    e = torch.zeros((), dtype=torch.float64, device="cuda")
    for a in range(len(u)):
        for b in range(a, len(u)):
            v, _ = _table(cell, n, case["omega"], kpt[b] - kpt[a])
            for s in range(case["nb"]):
                t = slice(s if a == b else 0, case["nb"])
                rho = torch.fft.fftn(u[a][s].conj() * u[b][t], dim=(1, 2, 3))
                self_ = torch.arange(t.start, t.stop, device="cuda") == (s if a == b else -1)
                p = ((rho.real ** 2 + rho.imag ** 2) * v).sum((1, 2, 3))
                e += f[a][s] * (f[b][t] * torch.where(self_, 1.0, 2.0) * p).sum()
                phi = torch.fft.ifftn(rho * v, dim=(1, 2, 3))
                w[b][t] -= f[a][s] * u[a][s] * phi
                g = torch.where(self_, torch.zeros_like(f[b][t]), f[b][t])
                w[a][s] -= (g[:, None, None, None] * u[b][t] * phi.conj()).sum(0)
    return {"vpsi": [_sphere_of(x, i, n, vol) for x, i in zip(w, idx)], "ex": float(e) * (-0.5 * vol / float(n) ** 6)}


def _exact_response(case, seed):
    s, n = _response(case, seed), case["N"]
    _, vol = _recip(s["cell"])
    kin = 0.5 * torch.from_numpy(s["g2"]).cuda()
    eps = torch.from_numpy(s["eps"]).cuda()[:, None]
    u, v = s["u"], s["v"]

    def project(x):
        return (x @ u.conj().T) @ u

    def operator(x):
        r, i = _real_space(x, s["m"], n, vol)
        return kin * x + _sphere_of(r * v, i, n, vol) - eps * x + s["alpha"] * project(x)

    dot = lambda a, b: (a.conj() * b).sum(1).real  # noqa: E731
    r = -(s["w"] - project(s["w"]))
    x, p, rr = torch.zeros_like(r), r.clone(), dot(r, r)
    live = torch.ones_like(rr, dtype=torch.bool)
    iters = np.zeros(len(r), dtype=np.int64)
    for _ in range(1000):
        if not bool(live.any()):
            break
        iters += live.cpu().numpy()
        ap = operator(p)
        al = torch.where(live, rr / dot(p, ap), torch.zeros_like(rr))[:, None]
        x, r = x + al * p, r - al * ap
        new = torch.where(live, dot(r, r), rr)
        p = torch.where(live[:, None], r + (new / rr)[:, None] * p, p)
        rr = new
        live = live & ~(torch.sqrt(rr) < s["tol"])
    return {"g": x, "iters": iters, "resid": torch.sqrt(rr)}


def exact(case, seed):
    kind, cell = case["kind"], _cell(case)
    if work(case)["flops"] > 4.5e12:  # beyond about 20 seconds
        return None
    if kind == "kpoints":
        return _exact_k(case, seed)
    if kind == "sternheimer":
        return _exact_response(case, seed)
    if kind == "batch":
        out = {"vpsi": [], "ex": []}
        for s, (n, L, nb) in enumerate(_systems(case)):
            c = _cell(case, L)
            v, e, _ = _exact_gamma(_orbitals(*_sphere(c, case["ecut"]), nb, seed + 100 * s), np.full(nb, 2.0), c,
                                   case["ecut"], n, case["omega"])
            out["vpsi"].append(v)
            out["ex"].append(e)
        return {"vpsi": out["vpsi"], "ex": np.array(out["ex"])}
    m, g2 = _sphere(cell, case["ecut"])
    psi, occ = _orbitals(m, g2, case["nb"], seed), _occ(case, case["nb"], seed)
    if kind == "grad":
        psi = psi.to(torch.complex64).to(torch.complex128)
    trial = _orbitals(m, g2, case["nt"], seed + 1) if kind == "fixed" else None
    v, e, d = _exact_gamma(psi, occ, cell, case["ecut"], case["N"], case["omega"], trial)
    if kind == "fixed":
        return {"vphi": v}
    if kind == "grad":
        return {"ex": e, "psi_grad": 2 * torch.from_numpy(occ).cuda()[:, None] * v, "omega_grad": d}
    return {"vpsi": v, "ex": e, "dex": d} if case["dex"] else {"vpsi": v, "ex": e}
