"""The workloads by which the speed of the sampler's calls is judged.

A case names one call of the public API (or, where a program makes them
together, a forward and a backward one) with its sizes; :func:`prepare` holds
what a program has in hand before that call (the plan, which every input of a
geometry shares, and inputs drawn from the seed), :func:`run` makes the call,
:func:`work` counts what it cannot do without, and :func:`exact` gives the
same result in plain 64-bit torch.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2306_15511_gb300 as shtg
from paper_2306_15511_gb300 import autograd

# ------------------------------------------------------------------- the cases
# Fields: call; the grid (nside, or nring x nphi of a Gauss-Legendre grid);
# lmax; batch; spin; arith (the transforms' arithmetic: fp64, df64, fp32,
# tc32); geoms (chains): nside:lmax:chains per geometry; the rest belongs to
# single calls.


def listed():
    return [
        # the smallest transform of the test ladder: latency and launches
        dict(name="synth_t_fp64_n32", call="synth", nside=32, nring=0, nphi=0, lmax=64, batch=1, spin=0, arith="fp64"),
        # the full-sky temperature sample in FP64 (closed-form validation runs): a whole small solve
        dict(name="solve_t_fp64_n32", call="solve", nside=32, nring=0, nphi=0, lmax=64, batch=1, ncomp=1, mode="fp64",
             tol=1e-8),
        # forward and backward through the autograd function, one FP32 sky (gradient-based users)
        dict(name="grad_t_fp32_n512", call="grad", nside=512, nring=0, nphi=0, lmax=1024, batch=1, spin=0,
             arith="fp32"),
        # log-posterior with its gradients in alm and in the binned log C_l
        dict(name="logpost_t_n512", call="logpost", nside=512, nring=0, nphi=0, lmax=1024, batch=1, bins=50),
        # the two halves of the mixed solver's operator at the benchmark size, Q/U of 8 realizations
        dict(name="synth_p_tc32_n1024", call="synth", nside=1024, nring=0, nphi=0, lmax=2048, batch=8, spin=2,
             arith="tc32"),
        dict(name="adjoint_p_tc32_n1024", call="adjoint", nside=1024, nring=0, nphi=0, lmax=2048, batch=8, spin=2,
             arith="tc32"),
        # the temperature operator of the chains' largest geometry, odd l_max, 12 chains in a batch
        dict(name="normal_t_tc32_n256", call="normal", nside=256, nring=0, nphi=0, lmax=767, batch=12, spin=0,
             arith="tc32"),
        # the FP64-accurate operator halves of the residual replacements (double-FP32 sums)
        dict(name="normal_p_df64_n512", call="normal", nside=512, nring=0, nphi=0, lmax=1024, batch=4, spin=2,
             arith="df64"),
        # quadrature analysis with one refinement on a Gauss-Legendre grid whose rings are not powers of two
        dict(name="map2alm_t_fp64_gl301", call="map2alm", nside=0, nring=301, nphi=602, lmax=300, batch=3, spin=0,
             arith="fp64", niter=1),
        # one native-FP64 application of the T+E+B operator
        dict(name="operator_teb_fp64_n128", call="operator", nside=128, nring=0, nphi=0, lmax=256, batch=2, ncomp=3),
        # a whole T+E+B sample with uneven noise, tensor-core iterations and residual replacements
        dict(name="solve_teb_tc_n128", call="solve", nside=128, nring=0, nphi=0, lmax=256, batch=4, ncomp=3,
             mode="mixed_tc", tol=1e-11),
        # chains of four geometries under a latitude cut, one call, azimuthal block preconditioner
        dict(name="chains_tc_azim", call="chains", geoms="64:128:10 64:191:5 128:256:8 128:383:4", tol=1e-11),
    ]


#: Largest sizes drawn per call and arithmetic: (nside, batch)
_TOP = {"fp64": (256, 8), "df64": (512, 8), "fp32": (1024, 4), "tc32": (1024, 8)}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["synth", "synth", "adjoint", "adjoint", "grad", "normal", "normal", "map2alm", "operator",
                       "logpost", "solve", "chains"])
    if call == "chains":
        g = [(n, rng.randint(3 * n // 2, 3 * n - 1), rng.randint(1, 8)) for n in rng.sample([16, 24, 32, 48, 64, 96, 128], 3)]
        return dict(call="chains", geoms=" ".join("%d:%d:%d" % t for t in g), tol=1e-11)
    if call == "solve":
        nside = rng.choice([16, 24, 32, 48, 64, 96, 128])
        mode = rng.choice(["fp64", "mixed", "mixed_tc"])
        nc = rng.choice([1, 3])
        nside = min(nside, 48) if mode == "fp64" else nside
        return dict(call="solve", nside=nside, nring=0, nphi=0, lmax=rng.randint(3 * nside // 2, 5 * nside // 2),
                    batch=rng.randint(1, 4), ncomp=nc, mode=mode, tol=1e-8 if mode == "fp64" else 1e-11)
    if call == "operator":
        nside = _log_int(rng, 16, 128)
        return dict(call="operator", nside=nside, nring=0, nphi=0, lmax=rng.randint(3 * nside // 2, 5 * nside // 2),
                    batch=rng.randint(1, 4), ncomp=rng.choice([1, 3]))
    if call == "logpost":
        nside = _log_int(rng, 32, 512)
        return dict(call="logpost", nside=nside, nring=0, nphi=0, lmax=rng.randint(3 * nside // 2, 5 * nside // 2),
                    batch=1, bins=rng.randint(5, 50))
    arith = rng.choice(["fp64", "fp32"]) if call in ("map2alm", "grad") else rng.choice(["fp64", "df64", "fp32", "tc32"])
    top, most = _TOP[arith]
    spin = rng.choice([0, 2])
    c = dict(call=call, nside=0, nring=0, nphi=0, lmax=0, batch=rng.randint(1, most), spin=spin, arith=arith)
    if rng.random() < 0.25 or call == "map2alm":   # a Gauss-Legendre grid, its rings long enough for l_max
        c["lmax"] = _log_int(rng, 24, min(2 * top, 600))
        c["nring"] = c["lmax"] + 1 + rng.randint(0, 9)
        c["nphi"] = 2 * c["lmax"] + 1 + rng.randint(0, 40)
    else:
        c["nside"] = _log_int(rng, 16, top)
        c["lmax"] = rng.randint(3 * c["nside"] // 2, 2 * c["nside"] if c["nside"] > top // 2 else 3 * c["nside"] - 1)
    if call == "map2alm":
        c["niter"] = rng.randint(0, 2)
    while _units(c) * _weight(c) > 1.1e12:
        c["batch"] -= 1
    return c


def _pairs(c):
    nring = c["nring"] or 4 * c["nside"] - 1
    return (nring + 1) // 2


def _weight(c):
    return {"fp64": 8.0, "df64": 4.0, "fp32": 1.0, "tc32": 1.0}[c.get("arith", "fp64")]


def _units(c):
    """Flops of one Legendre stage: per (l, m, ring pair) the recurrence and the maps' multiply-adds."""
    lm = (c["lmax"] + 1) * (c["lmax"] + 2) // 2 * _pairs(c)
    spins = {1: (0,), 3: (0, 2)}[c["ncomp"]] if "ncomp" in c else (c.get("spin", 0),)
    return float(lm) * sum(8 + 16 * c["batch"] if s == 2 else 3 + 4 * c["batch"] for s in spins)


def work(case):
    c = case
    if c["call"] == "chains":
        each = [work(g) for g in _groups(c)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    rows = c["ncomp"] if "ncomp" in c else (2 if c.get("spin") == 2 else 1)
    npix = 12 * c["nside"] ** 2 if c["nside"] else c["nring"] * c["nphi"]
    nalm = (c["lmax"] + 1) * (c["lmax"] + 2) // 2
    real = 4 if c.get("arith") in ("fp32", "tc32") or c["call"] == "logpost" else 8
    maps, alms = real * c["batch"] * rows * npix, 2 * real * c["batch"] * rows * nalm
    ninv = real * npix * (2 if rows == 3 else 1)
    leg = _units(c)
    fft = 2.5 * c["batch"] * rows * npix * math.log2(4 * c["nside"] or c["nphi"])
    one = leg + fft
    call = c["call"]
    if call in ("synth", "adjoint"):
        return {"bytes": maps + alms, "flops": one}
    if call in ("grad", "normal"):
        return {"bytes": 2 * maps + 2 * alms, "flops": 2 * one}
    if call == "map2alm":
        return {"bytes": maps + alms, "flops": (1 + 2 * c["niter"]) * one}
    if call == "operator":
        return {"bytes": 2 * alms + ninv, "flops": 2 * one}
    if call == "logpost":
        return {"bytes": 2 * maps + 2 * alms, "flops": 2 * one}
    # a solve: the right-hand side and ten applications of the operator
    return {"bytes": 2 * maps + 2 * alms + ninv, "flops": 21 * one}


# ------------------------------------------------------------------ the inputs
@functools.lru_cache(maxsize=1)
def _plans(grids):
    """The plans a program makes once per grid and uses for every input."""
    return [shtg.Plan(nside=n, lmax=l, max_batch=b, spin2=s2) if n else
            shtg.Plan(gauss=(r, k), lmax=l, max_batch=b, spin2=s2) for n, r, k, l, b, s2 in grids]


def _groups(c):
    """One temperature problem per geometry of a chains call."""
    return [dict(call="solve", nside=n, nring=0, nphi=0, lmax=l, batch=b, ncomp=1, tol=c["tol"])
            for n, l, b in (map(int, g.split(":")) for g in c["geoms"].split())]


def _grid(c):
    return c["nside"], c["nring"], c["nphi"], c["lmax"], c["batch"], c.get("ncomp", 1) == 3 or c.get("spin") == 2


def _spectra(lmax, ncomp):
    """Flat T spectrum with a damped tail; E, B and T-E as fixed fractions of it; 0 below l = 2."""
    l = np.arange(lmax + 1, dtype=np.float64)
    tt = np.zeros(lmax + 1)
    tt[2:] = 2.0 * math.pi * 1000.0 / (l[2:] * (l[2:] + 1.0)) * np.exp(-l[2:] * (l[2:] + 1.0) / 1500.0 ** 2)
    return tt if ncomp == 1 else np.stack([tt, 0.05 * tt, 5e-5 * tt, 0.3 * math.sqrt(0.05) * tt])


def _beam(lmax):
    """Gaussian beam of FWHM 1.5 times the shortest resolved scale."""
    l = np.arange(lmax + 1, dtype=np.float64)
    sig = 1.5 * math.pi / lmax / math.sqrt(8.0 * math.log(2.0))
    return np.exp(-0.5 * l * (l + 1.0) * sig * sig)


def _lm(lmax):
    l = torch.cat([torch.arange(m, lmax + 1) for m in range(lmax + 1)])
    m = torch.cat([torch.full((lmax + 1 - m,), m) for m in range(lmax + 1)])
    return l, m


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _white_alm(g, lmax, *lead):
    """Unit white noise: variance 1 real at m = 0, 1/2 per part above."""
    _, m = _lm(lmax)
    x = torch.randn(*lead, m.numel(), 2, generator=g, device="cuda", dtype=torch.float64)
    s = torch.where(m == 0, 1.0, math.sqrt(0.5)).double().cuda()
    x = x * s[:, None]
    x[..., (m == 0).cuda(), 1] = 0.0
    return torch.view_as_complex(x)


def _sky(g, lmax, ncomp, *lead):
    """alm of a Gaussian sky: T, or T, E, B with their T-E correlation."""
    cl = torch.as_tensor(_spectra(lmax, 3)).cuda()[:, _lm(lmax)[0].cuda()]
    w = _white_alm(g, lmax, *lead, ncomp)
    t = cl[0].sqrt() * w[..., 0, :]
    if ncomp == 1:
        return t[..., None, :]
    l21 = 0.3 * cl[1].sqrt()
    l22 = (cl[1] * (1.0 - 0.09)).sqrt()
    return torch.stack([t, l21 * w[..., 0, :] + l22 * w[..., 1, :], cl[2].sqrt() * w[..., 2, :]], dim=-2)


def _npix(c):
    return 12 * c["nside"] ** 2 if c["nside"] else c["nring"] * c["nphi"]


def _noise_level(c):
    """Noise variance per pixel: 1 + 4 sin^2 of the angle to a tilted axis scans, 20 uK for one."""
    z, phi = _centres(c)
    s = torch.sqrt(torch.clamp(1.0 - z * z, min=0.0))
    ax = (0.87 * math.cos(1.68), 0.87 * math.sin(1.68), math.sqrt(1.0 - 0.87 ** 2))
    mu = s * torch.cos(phi) * ax[0] + s * torch.sin(phi) * ax[1] + z * ax[2]
    return 400.0 / (1.0 + 4.0 * mu * mu)


def prepare(case, seed):
    c = dict(case)
    if c["call"] == "chains":
        groups = _groups(c)
        plans = _plans(tuple(_grid(g) for g in groups))
        made = [_prepare(g, seed * 16 + k, p, cut=15.0) for k, (g, p) in enumerate(zip(groups, plans))]
        keep = ("plan", "cl", "bl", "ninv", "d", "w1", "w2", "cl_scale")
        return dict(case=c, groups=[{k: m[k] for k in keep} for m in made])
    return _prepare(c, seed, _plans((_grid(c),))[0])


def _prepare(c, seed, plan, cut=0.0):
    g = _generator(seed)
    L, nb, npix = c["lmax"], c["batch"], _npix(c)
    nc = c.get("ncomp", 1)
    spin = c.get("spin", 2 if nc == 3 else 0)
    cx, re = ((torch.complex64, torch.float32) if c.get("arith") in ("fp32", "tc32") or c["call"] == "logpost"
              else (torch.complex128, torch.float64))
    s = dict(case=c, plan=plan)
    call = c["call"]
    rows = (nb, 2) if spin == 2 else (nb,)
    alm = (lambda: (_sky(g, L, 3, nb)[:, 1:] if spin == 2 else _sky(g, L, 1, nb)[:, 0]).to(cx).contiguous())
    noise = (lambda *lead: torch.randn(*lead, npix, generator=g, device="cuda", dtype=torch.float64))
    if call in ("synth", "grad", "normal"):
        s["alm"] = alm()
    if call in ("adjoint", "map2alm"):
        s["map"] = (20.0 * noise(*rows)).to(re)
    if call == "grad":
        s["alm"].requires_grad_()
        s["weight"] = (0.05 * noise(*rows)).to(re)
    if call == "normal":
        s["ninv"] = (1.0 / _noise_level(c)).to(re)
    if call == "operator":
        s["x"] = _sky(g, L, nc, nb).contiguous()
    if call in ("operator", "solve", "logpost"):
        s["cl"], s["bl"] = _spectra(L, nc), _beam(L)
        var = _noise_level(c)
        s["ninv"] = torch.stack([1.0 / var, 0.5 / var]) if nc == 3 else 1.0 / var
    if call in ("solve", "logpost"):
        sky = _sky(g, L, nc, nb)
        bl = torch.as_tensor(s["bl"]).cuda()[_lm(L)[0].cuda()]
        sd = torch.stack([var, 2.0 * var, 2.0 * var]).sqrt() if nc == 3 else var.sqrt()[None]
        s["d"] = sd * noise(nb, nc)
        s["d"][:, 0] += plan.alm2map((sky[:, 0] * bl).contiguous())
        if nc == 3:
            s["d"][:, 1:] += plan.alm2map((sky[:, 1:] * bl).contiguous(), spin=2)
    if call == "solve":
        s["w1"], s["w2"] = _white_alm(g, L, nb, nc), noise(nb, nc)
    if cut:   # chains: a latitude cut, an amplitude of the spectrum per chain (drawn anew, as a sampler's C_l are)
        s["ninv"] = s["ninv"] * (_centres(c)[0].abs() >= math.sin(math.radians(cut)))
        s["cl_scale"] = 0.8 + 0.4 * np.random.default_rng(seed).random(nb)
    if call == "logpost":
        s["alm"] = (sky[0, 0] * 0.9).to(cx)
        s["d"], s["ninv"] = s["d"][0, 0].float().contiguous(), s["ninv"].float()
        w = max(1, (L - 1) // c["bins"])
        s["bins"] = [(2 + k * w, min(L, 2 + (k + 1) * w - 1)) for k in range(c["bins"]) if 2 + k * w <= L]
    return s


# --------------------------------------------------------------------- the call
def run(s):
    c, plan = s["case"], s.get("plan")
    call = c["call"]
    how = dict(tensor_cores=c.get("arith") == "tc32", double_float=c.get("arith") == "df64")
    if call == "synth":
        return plan.alm2map(s["alm"], spin=c["spin"], **how)
    if call == "adjoint":
        return plan.alm2map_adjoint(s["map"], spin=c["spin"], **how)
    if call == "map2alm":
        return plan.map2alm(s["map"], spin=c["spin"], niter=c["niter"])
    if call == "grad":
        s["alm"].grad = None
        m = autograd.alm2map(plan, s["alm"], c["spin"])
        m.backward(s["weight"])
        return m.detach(), s["alm"].grad
    if call == "normal":
        m = plan.alm2map(s["alm"], spin=c["spin"], **how)
        return m, plan.alm2map_adjoint(m * s["ninv"], spin=c["spin"], **how)
    if call == "operator":
        return plan.apply_operator(s["cl"], s["bl"], s["ninv"], s["x"])
    if call == "logpost":
        value, grad, grad_cl = plan.logpost_grad(s["cl"], s["bl"], s["alm"], s["d"], s["ninv"], s["bins"])
        return np.float64(value), grad, grad_cl
    if call == "chains":
        return [x for x, _ in shtg.chains_sample(s["groups"], tol=c["tol"], precond="azim")]
    x, _ = plan.cg_sample(s["cl"], s["bl"], s["ninv"], s["d"], s["w1"], s["w2"], tol=c["tol"], mode=c["mode"])
    return x


# ------------------------------------------------- the same in plain 64-bit torch
def _rings(c):
    """(cos, sin of theta; pixels; phase of the first pixel; quadrature weight) per ring, north to south."""
    if not c["nside"]:
        x, w = np.polynomial.legendre.leggauss(c["nring"])
        x, w = x[::-1].copy(), w[::-1].copy()
        n = np.full(c["nring"], c["nphi"])
        return x, np.sqrt((1 - x) * (1 + x)), n, np.zeros(c["nring"]), w * 2 * np.pi / c["nphi"]
    N = c["nside"]
    i = np.arange(1, 2 * N + 1, dtype=np.float64)
    cap = i < N
    u = np.where(cap, i * i / (3.0 * N * N), 1.0 - (4.0 / 3.0 - 2.0 * i / (3.0 * N)))   # 1 - cos(theta)
    n = np.where(cap, 4 * i, 4.0 * N).astype(int)
    shift = np.where(cap, 1, (i - N) % 2 == 0).astype(float)
    x, s = 1.0 - u, np.sqrt(u * (2.0 - u))
    x[-1] = 0.0 if 2 * N == len(i) else x[-1]
    both = lambda v: np.concatenate([v, v[-2::-1]])  # noqa: E731
    return (np.concatenate([x, -x[-2::-1]]), both(s), both(n), both(shift * np.pi / n),
            np.full(4 * N - 1, 4 * np.pi / (12.0 * N * N)))


def _centres(c):
    x, _, n, p0, _ = _rings(c)
    z = torch.repeat_interleave(torch.as_tensor(x), torch.as_tensor(n))
    j = torch.cat([torch.arange(k, dtype=torch.float64) for k in n])
    per = lambda v: torch.repeat_interleave(torch.as_tensor(v), torch.as_tensor(n))  # noqa: E731
    return z.cuda(), (per(p0) + j * (2 * math.pi / per(n.astype(float)))).cuda()


def _lambda_blocks(c, spins, step=16):
    """Yields (l0, [lambda], or [lw, lx], per spin), each [m, l - l0, ring] on the northern rings and the equator.

    Three-term recurrence in l for all m and rings at once, from sectoral values in base-2 logarithms; values are kept
    as mantissa times 2^(512 e) with e <= 0.  Spin 2 by the spin-raising relations.
    """
    L = c["lmax"]
    x, s, _, _, _ = _rings(c)
    P = (len(x) + 1) // 2
    x, s = torch.as_tensor(x[:P]).cuda(), torch.as_tensor(s[:P]).cuda()
    m = torch.arange(L + 1, dtype=torch.float64, device="cuda")
    lg = torch.cumsum(torch.cat([torch.zeros(1), torch.log2((2 * m[1:] - 1) / (2 * m[1:])).cpu()]).double(), 0).cuda()
    lg = 0.5 * (lg + torch.log2((2 * m + 1) / (4 * math.pi)))
    q = lg[:, None] + m[:, None] * torch.log2(s)[None, :]
    e0 = torch.clamp(torch.ceil(q / 512.0), max=0.0)
    seed = torch.exp2(q - 512.0 * e0) * torch.where(m % 2 == 1, -1.0, 1.0)[:, None]
    cur, prev, ex = torch.zeros_like(q), torch.zeros_like(q), torch.zeros_like(q)
    true_prev = torch.zeros_like(q)
    out = None
    for l in range(L + 1):
        k = l + 1   # rows m <= l
        mm = m[:k]
        if l > 0:
            a = torch.sqrt((4.0 * l * l - 1.0) / torch.clamp(l * l - mm * mm, min=1.0))
            b = torch.sqrt(torch.clamp(((l - 1.0) ** 2 - mm * mm) / (4.0 * (l - 1.0) ** 2 - 1.0), min=0.0)) if l > 1 else 0 * mm
            t = a[:, None] * (x * cur[:k] - b[:, None] * prev[:k])
            prev[:k] = cur[:k]
            cur[:k] = t
            big = (t.abs() > 2.0 ** 200) & (ex[:k] < 0)
            f = torch.exp2(-512.0 * big.double())
            cur[:k] *= f
            prev[:k] *= f
            ex[:k] += big
        cur[l], prev[l], ex[l] = seed[l], 0.0, e0[l]
        lam = torch.where(ex[:k] == 0, cur[:k], 0.0)
        if l % step == 0:
            out = [torch.zeros(L + 1, step, P, device="cuda", dtype=torch.float64)
                   for sp in spins for _ in range(1 if sp == 0 else 2)]
        i = 0
        for sp in spins:
            if sp == 0:
                out[i][:k, l % step] = lam
                i += 1
                continue
            if l >= 2:
                nl = 2.0 / math.sqrt((l + 2.0) * (l + 1.0) * l * (l - 1.0))
                kap = torch.sqrt((2 * l + 1.0) / (2 * l - 1.0) * (l * l - mm * mm))[:, None]
                i2 = 1.0 / (s * s)
                low = kap * true_prev[:k]
                out[i][:k, l % step] = nl * (x * i2 * low - ((l - mm * mm)[:, None] * i2 + 0.5 * l * (l - 1)) * lam)
                out[i + 1][:k, l % step] = nl * i2 * mm[:, None] * (low - (l - 1.0) * x * lam)
            i += 2
        true_prev[:k] = lam
        if l % step == step - 1 or l == L:
            yield l - l % step, out


def _square(alm, L):
    """[..., nalm] -> [m, l, ...] with zeros for l < m."""
    l, m = _lm(L)
    out = torch.zeros(L + 1, L + 1, *alm.shape[:-1], dtype=torch.complex128, device="cuda")
    out[m.cuda(), l.cuda()] = alm.to(torch.complex128).movedim(-1, 0)
    out[0] = out[0].real.to(out.dtype)
    return out


class _Reference:
    """Y and its transpose on rows (maps) of one grid; blocks kept where they fit in memory."""

    def __init__(self, c, spins, keep=False):
        self.c, self.spins, self.L = c, spins, c["lmax"]
        self.n, self.p0, self.w = _rings(c)[2:]
        self.R = len(self.n)
        self.P = (self.R + 1) // 2
        self.kept = [(l0, [b.clone() for b in bl]) for l0, bl in _lambda_blocks(c, spins)] if keep else None

    def blocks(self):
        return self.kept if self.kept is not None else _lambda_blocks(self.c, self.spins)

    def sign(self, l0, k):
        l = torch.arange(l0, l0 + k, device="cuda")[None, :]
        m = torch.arange(self.L + 1, device="cuda")[:, None]
        return torch.where((l + m) % 2 == 0, 1.0, -1.0).double()

    def synth(self, rows):
        """rows: one alm [B, nalm] per spin 0, (E, B) [B, 2, nalm] per spin 2 -> maps [B, npix] / [B, 2, npix]."""
        sq = [_square(a, self.L) for a in rows]
        F = [torch.zeros(self.L + 1, 2, 2 * (a[0, 0].numel()), self.P, device="cuda", dtype=torch.float64) for a in sq]
        for l0, bl in self.blocks():
            k = min(bl[0].shape[1], self.L + 1 - l0)
            sg = self.sign(l0, k)[:, :, None]
            i = 0
            for a, f, sp in zip(sq, F, self.spins):
                v = a[:, l0:l0 + k]
                re = lambda t: torch.view_as_real(t.contiguous()).reshape(self.L + 1, k, -1)  # noqa: E731
                if sp == 0:
                    parts = [(bl[i][:, :k], re(v), 1.0)]
                    i += 1
                else:   # Q = -(E lw + i B lx), U = i E lx - B lw; lx has the opposite parity
                    E, B = v[..., 0], v[..., 1]
                    parts = [(bl[i][:, :k], re(torch.stack([-E, -B], -1)), 1.0),
                             (bl[i + 1][:, :k], re(torch.stack([-1j * B, 1j * E], -1)), -1.0)]
                    i += 2
                for lam, co, par in parts:
                    f[:, 0] += torch.bmm(co.transpose(1, 2), lam)
                    f[:, 1] += torch.bmm((co * sg * par).transpose(1, 2), lam)
        return [self.to_map(f, a.shape[2:]) for f, a in zip(F, sq)]

    def to_map(self, f, lead):
        z = torch.view_as_complex(f.reshape(self.L + 1, 2, -1, 2, self.P).movedim(3, 4).contiguous())
        full = torch.cat([z[:, 0], z[:, 1, :, :self.R - self.P].flip(2)], 2)     # [m, row, ring]
        m = torch.arange(self.L + 1, device="cuda")
        out = [None] * self.R
        for n in np.unique(self.n):
            at = torch.as_tensor(np.nonzero(self.n == n)[0], device="cuda")
            ph = torch.exp(1j * m[:, None] * torch.as_tensor(self.p0, device="cuda")[at][None])
            v = full[:, :, at] * ph[:, None]
            h = torch.zeros(int(n), *v.shape[1:], dtype=v.dtype, device="cuda")
            h.index_add_(0, m % int(n), v)
            mp = 2.0 * torch.fft.ifft(h, dim=0, norm="forward").real - v[0].real
            for j, r in enumerate(at.tolist()):
                out[r] = mp[:, :, j].T
        return torch.cat(out, 1).reshape(*lead, -1)

    def adjoint(self, maps, weighted=False):
        """The transpose: maps per spin -> alm per spin."""
        G = []
        for mp in maps:
            flat = mp.double().reshape(-1, mp.shape[-1])
            g = torch.zeros(self.L + 1, flat.shape[0], self.R, dtype=torch.complex128, device="cuda")
            m = torch.arange(self.L + 1, device="cuda")
            ofs = np.concatenate([[0], np.cumsum(self.n)])
            for n in np.unique(self.n):
                at = np.nonzero(self.n == n)[0]
                v = torch.stack([flat[:, ofs[r]:ofs[r] + n] for r in at], 1)
                if weighted:
                    v = v * torch.as_tensor(self.w[at], device="cuda")[None, :, None]
                h = torch.fft.fft(v, dim=2)[:, :, m % int(n)]
                ph = torch.exp(-1j * m[None, :] * torch.as_tensor(self.p0[at], device="cuda")[:, None])
                g[:, :, torch.as_tensor(at, device="cuda")] = (h * ph[None]).permute(2, 0, 1)
            S = torch.zeros(self.L + 1, flat.shape[0], self.P, dtype=torch.complex128, device="cuda")
            S[:, :, :self.R - self.P] = g[:, :, self.P:].flip(2)
            G.append((g[:, :, :self.P], S, mp.shape[:-1]))
        outs = [torch.zeros(self.L + 1, self.L + 1, *lead, dtype=torch.complex128, device="cuda") for _, _, lead in G]
        for l0, bl in self.blocks():
            k = min(bl[0].shape[1], self.L + 1 - l0)
            even = self.sign(l0, k)[:, None, :] > 0
            i = 0
            for (gn, gs, lead), o, sp in zip(G, outs, self.spins):
                def contract(lam, par):
                    lt = lam[:, :k].transpose(1, 2)
                    both = [torch.bmm(torch.view_as_real(t).movedim(3, 1).reshape(self.L + 1, -1, self.P), lt)
                            for t in (gn + par * gs, gn - par * gs)]
                    v = torch.where(even, both[0], both[1]).reshape(self.L + 1, 2, *lead, k)
                    return torch.complex(v[:, 0], v[:, 1])       # [m, *lead, k]
                if sp == 0:
                    o[:, l0:l0 + k] = contract(bl[i], 1.0).movedim(-1, 1)
                    i += 1
                else:   # E = -lw Q - i lx U, B = i lx Q - lw U
                    w, xx = contract(bl[i], 1.0), contract(bl[i + 1], -1.0)
                    E = -w[..., 0, :] - 1j * xx[..., 1, :]
                    B = 1j * xx[..., 0, :] - w[..., 1, :]
                    o[:, l0:l0 + k] = torch.stack([E, B], -2).movedim(-1, 1)
                    i += 2
        l, m = (t.cuda() for t in _lm(self.L))
        alms = []
        for o in outs:
            o[0] = o[0].real.to(o.dtype)
            alms.append(o[m, l].movedim(0, -1))
        return alms


def _split(a, nc):
    return [a[:, 0]] if nc == 1 else [a[:, 0], a[:, 1:]]


def _join(parts):
    return torch.cat([p.reshape(p.shape[0], -1, p.shape[-1]) for p in parts], 1)


class _Operator:
    """A = S^-1 + B Y^T N^-1 Y B and its right-hand side in 64 bits (multipoles with C_l = 0 held at 0)."""

    def __init__(self, c, s, keep):
        self.nc = c.get("ncomp", 1)
        self.ref = _Reference(c, (0,) if self.nc == 1 else (0, 2), keep)
        L = c["lmax"]
        l = _lm(L)[0]
        cl = torch.as_tensor(s["cl"]).reshape(-1, L + 1)[:, l].cuda()
        self.on = cl[0] > 0
        bl = torch.as_tensor(s["bl"])[l].cuda() * self.on
        self.bl = bl
        one = lambda v: torch.where(self.on, v, torch.ones_like(v))  # noqa: E731
        if self.nc == 1:
            C = one(cl[0])[:, None, None]
        else:
            C = torch.zeros(cl.shape[1], 3, 3, dtype=torch.float64, device="cuda")
            C[:, 0, 0], C[:, 1, 1], C[:, 2, 2] = one(cl[0]), one(cl[1]), one(cl[2])
            C[:, 0, 1] = C[:, 1, 0] = torch.where(self.on, cl[3], torch.zeros_like(cl[3]))
        ev, V = torch.linalg.eigh(C)
        sc = torch.as_tensor(s["cl_scale"], device="cuda") if s.get("cl_scale") is not None else torch.ones(1, device="cuda")
        self.sc = sc.double()[:, None, None]
        self.Si = (V / ev[:, None, :]) @ V.transpose(1, 2)
        self.Sh = (V / ev[:, None, :].sqrt()) @ V.transpose(1, 2)
        self.ninv = s["ninv"].double().reshape(-1, s["ninv"].shape[-1])

    def harm(self, M, a):
        return torch.einsum("nij,bjn->bin", M.to(a.dtype), a)

    def weigh(self, m, w):
        return [m[0] * w[0]] if self.nc == 1 else [m[0] * w[0], m[1] * w[1]]

    def apply(self, a):
        y = self.ref.adjoint(self.weigh(self.ref.synth(_split(a * self.bl, self.nc)), self.ninv))
        return _join(y) * self.bl + self.harm(self.Si, a) / self.sc

    def rhs(self, d, w1, w2):
        y = [p + q for p, q in zip(self.weigh(_split(d, self.nc), self.ninv), self.weigh(_split(w2, self.nc), self.ninv.sqrt()))]
        return _join(self.ref.adjoint(y)) * self.bl + torch.where(self.on, self.harm(self.Sh, w1), 0.0) / self.sc.sqrt()

    def preconditioner(self):
        """T: per m, the inverse of the operator with the noise weight averaged along rings; T+E+B: a scaled diagonal."""
        if self.nc == 3:
            nbar = self.ninv.sum(1) / (4 * math.pi)
            D = self.Si.clone()
            for k in range(3):
                D[:, k, k] += self.bl ** 2 * nbar[min(k, 1)]
            D = torch.linalg.inv(D)
            return lambda r: self.harm(D, r)
        ref, L = self.ref, self.ref.L
        lam = torch.cat([b[0] for _, b in ref.kept], 1)[:, :L + 1]
        ring = torch.stack([t.sum() for t in torch.split(self.ninv[0], [int(k) for k in ref.n])])
        south = torch.zeros(ref.P, dtype=torch.float64, device="cuda")
        south[:ref.R - ref.P] = ring[ref.P:].flip(0)
        l, m = (t.cuda() for t in _lm(L))
        par = (torch.arange(L + 1, device="cuda")[:, None] + torch.arange(L + 1, device="cuda")[None]) % 2 == 0
        b = _square((self.bl + 0j)[None], L)[:, :, 0].real
        d = torch.ones(L + 1, L + 1, dtype=torch.float64, device="cuda")
        d[m, l] = self.Si[:, 0, 0] / self.sc.mean()
        H = torch.where(par, (lam * (ring[:ref.P] + south)) @ lam.transpose(1, 2),
                        (lam * (ring[:ref.P] - south)) @ lam.transpose(1, 2))
        H = torch.linalg.cholesky(H * b[:, :, None] * b[:, None, :] + torch.diag_embed(d))

        def solve(r):
            v = _square(r[:, 0], L)
            z = torch.cholesky_solve(torch.view_as_real(v).reshape(L + 1, L + 1, -1), H)
            return torch.view_as_complex(z.reshape(L + 1, L + 1, -1, 2).contiguous())[m, l].T[:, None]
        return solve


def _dot(a, b, w):
    return (w * (a.conj() * b).real).sum((1, 2))


def _solution(c, s):
    op = _Operator(c, s, keep=True)
    w = torch.where(_lm(c["lmax"])[1] == 0, 1.0, 2.0).cuda()
    b = op.rhs(s["d"], s["w1"], s["w2"])
    M = op.preconditioner()
    x = torch.zeros_like(b)
    r, bb = b, _dot(b, b, w)
    z = M(r)
    p, rz = z, _dot(r, z, w)
    for _ in range(200):
        q = op.apply(p)
        al = (rz / _dot(p, q, w))[:, None, None]
        x, r = x + al * p, r - al * q
        if bool((_dot(r, r, w) <= (1e-14 ** 2) * bb).all()):
            return x
        z = M(r)
        rz, old = _dot(r, z, w), rz
        p = z + (rz / old)[:, None, None] * p
    return None


def exact(case, seed):
    c = dict(case)
    s = prepare(case, seed)
    call = c["call"]
    spin = c.get("spin", 0)
    if call == "chains":
        return [_solution(g, t) for g, t in zip(_groups(c), s["groups"])]
    if call == "solve":
        return _solution(c, s)
    if call == "operator":
        return _Operator(c, s, keep=False).apply(s["x"])
    ref = _Reference(c, (spin,), keep=False)
    if call == "synth":
        return ref.synth([s["alm"]])[0]
    if call == "adjoint":
        return ref.adjoint([s["map"]])[0]
    if call == "normal":
        m = ref.synth([s["alm"]])[0]
        return m, ref.adjoint([m * s["ninv"].double()])[0]
    two = torch.where(_lm(c["lmax"])[1] == 0, 1.0, 2.0).cuda()
    if call == "grad":
        return ref.synth([s["alm"].detach()])[0], two * ref.adjoint([s["weight"]])[0]
    if call == "map2alm":
        a = ref.adjoint([s["map"]], weighted=True)[0]
        for _ in range(c["niter"]):
            a = a + ref.adjoint([s["map"].double() - ref.synth([a])[0]], weighted=True)[0]
        return a
    # the log-posterior and its gradients
    l = _lm(c["lmax"])[0].cuda()
    cl, bl = torch.as_tensor(s["cl"]).cuda(), torch.as_tensor(s["bl"]).cuda()[l]
    on = cl[l] > 0
    bl = bl * on
    icl = torch.where(on, 1.0 / torch.where(on, cl[l], 1.0), 0.0)
    a = s["alm"].to(torch.complex128)
    res = s["d"].double() - ref.synth([(a * bl)[None]])[0][0]
    wres = s["ninv"].double() * res
    power = torch.zeros_like(cl).index_add_(0, l, two * a.abs() ** 2 * icl)
    value = -0.5 * (wres * res).sum() - 0.5 * power.sum()
    grad = (ref.adjoint([wres[None]])[0][0] * bl - a * icl) * on
    gcl = np.array([0.5 * float(power[lo:hi + 1].sum()) for lo, hi in s["bins"]])
    return np.float64(float(value)), grad, gcl
