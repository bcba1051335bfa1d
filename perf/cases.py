"""Workloads that the tracer is timed on: the calls a user's program makes, from a
single evaluation of Hamilton's equations to whole sample -> trace -> bin steps,
images and gradients, over the sizes and stars of the paper's studies.

A case is a dict of plain values.  ``kind`` names the call:

* ``rhs``       rt_hamilton_rhs at given photon points
* ``sample``    rt_sample_batch: conversion-surface samples and weights
* ``bin``       rt_bin_spectrum of traced rays (cube, sky map and spectrum)
* ``forward``   one step of a forward study: rt_sample_batch, rt_trace_batch,
                rt_bin_batch (``precision`` fp64, df or mixed; ``order`` the claim order)
* ``image``     rt_trace_backward of one image plane
* ``uneven``    forward instances and images of different stars in one launch
* ``gradient``  flux.line_flux and its backward pass

Stars are magnetars and pulsars with an aligned or inclined dipole.  ``r_c`` is
the polar conversion radius in stellar radii (it fixes the axion mass); a case
with several stars spreads them from ``r_c`` inwards, as a scan over axion masses
does.  A star whose surface density is below the resonance has no rays: scans
contain such stars, too.
"""
from __future__ import annotations

import math

import torch

from paper_2309_08655_gb300 import flux, rt

F64 = torch.float64
DEV = "cuda"
NTH, NPH, NNU, NU_LO, NU_HI = 64, 32, 128, 0.0, 9.0
PRECISION = {"fp64": rt.PREC_FP64, "df": rt.PREC_DF, "mixed": rt.PREC_MIXED}
RTOL = {"fp64": 1e-10, "df": 1e-10, "mixed": 1e-8}
ORDER = {"index": rt.CLAIM_INDEX, "cost": rt.CLAIM_COST}
PLASMA = {"gj": rt.PLASMA_GJ, "twisted": rt.PLASMA_TWISTED}
# mean attempted steps of a ray (rtol 1e-10; mixed at 1e-8) and the operations of one,
# for work(): six right-hand sides of about 190 and the Runge-Kutta sums
STEPS = {"fp64": 180.0, "df": 180.0, "mixed": 80.0}
STEP_FLOPS = 1600.0


def listed():
    return [
        # a caller that integrates rays itself asks for the right-hand side of a
        # thousand points at a time: one short launch, latency is all there is
        dict(name="rhs_1000", kind="rhs", n=1000, theta=0.0, r_c=20.0, plasma="gj"),
        # the Monte-Carlo samples of the aligned star of the paper's fiducial setup
        dict(name="sample_aligned_4096", kind="sample", n=4096, stars=1, theta=0.0, r_c=20.0,
             span=1.0, plasma="gj", weight=rt.WEIGHT_PAG),
        # the samples of a production step: 16 axion masses of an inclined magnetar
        dict(name="sample_scan_16x65536", kind="sample", n=65536, stars=16, theta=30.0,
             r_c=16.0, span=100.0, plasma="gj", weight=rt.WEIGHT_PAG),
        # sky map, spectrum and cube of a production step's rays
        dict(name="bin_1048576", kind="bin", n=1 << 20, nth=64, nph=32, nnu=128, landed=0.42),
        # the paper's fiducial forward run, double precision, library defaults
        dict(name="forward_fp64_aligned_4096", kind="forward", n=4096, stars=1, theta=0.0,
             r_c=20.0, span=1.0, plasma="gj", rotation=0, precision="fp64", order="index"),
        # magnetar with a twisted field (no null cone): a smooth medium, many even rays
        dict(name="forward_fp64_twisted_16x4093", kind="forward", n=4093, stars=16, theta=30.0,
             r_c=16.0, span=100.0, plasma="twisted", rotation=0, precision="fp64",
             order="index"),
        # the Doppler-broadened line: the magnetosphere turns while the rays fly
        dict(name="forward_fp64_rotating_16x251", kind="forward", n=251, stars=16, theta=30.0,
             r_c=16.0, span=100.0, plasma="gj", rotation=1, precision="fp64", order="index"),
        # production steps: 16 masses in one launch, costly rays first; the accurate
        # path (double-float) and the fast one (mixed)
        dict(name="forward_df_scan_16x8192", kind="forward", n=8192, stars=16, theta=30.0,
             r_c=16.0, span=100.0, plasma="gj", rotation=0, precision="df", order="cost"),
        dict(name="forward_mixed_scan_16x65536", kind="forward", n=65536, stars=16, theta=30.0,
             r_c=16.0, span=100.0, plasma="gj", rotation=0, precision="mixed", order="cost"),
        # the radio image of the fiducial star at 60 degrees, both precisions
        dict(name="image_fp64_255x256", kind="image", nx=255, ny=256, incl=60.0, bmax=50.0,
             theta=0.0, r_c=20.0, precision="fp64"),
        dict(name="uneven_mixed_12", kind="uneven", instances=12, n=60000, side=300, theta=70.0,
             r_c=16.0, span=60.0, precision="mixed"),
        # one step of a fit: the line flux toward the observer and its gradient
        dict(name="gradient_fp64_32768", kind="gradient", n=32768, incl=63.0, theta=30.0,
             r_c=3.7, kappa=415.0, sweep="fp64"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case: kinds as often as a study calls them, sizes over their logarithm."""
    kind = rng.choice(["rhs", "sample", "bin", "forward", "forward", "forward", "image",
                       "uneven", "gradient"])
    theta = rng.choice([0.0, rng.uniform(0.0, 80.0)])
    r_c = _log(rng, 2.0, 16.0)
    if kind == "rhs":
        return dict(kind=kind, n=int(_log(rng, 100, 300000)), theta=theta, r_c=r_c,
                    plasma=rng.choice(["gj", "twisted"]))
    if kind == "sample":
        return dict(kind=kind, n=int(_log(rng, 200, 65536)), stars=rng.randint(1, 16),
                    theta=theta, r_c=r_c, span=_log(rng, 1.0, 100.0),
                    plasma=rng.choice(["gj", "gj", "twisted"]),
                    weight=rng.choice([rt.WEIGHT_PAG, rt.WEIGHT_PAG, rt.WEIGHT_UNIT_P,
                                       rt.WEIGHT_RENORM]))
    if kind == "bin":
        return dict(kind=kind, n=int(_log(rng, 1000, 1 << 20)), nth=rng.choice([18, 33, 64]),
                    nph=rng.choice([1, 31, 32]), nnu=rng.choice([1, 100, 128]),
                    landed=rng.uniform(0.2, 1.0))
    if kind == "forward":
        precision = rng.choice(["fp64", "df", "mixed"])
        plasma = rng.choice(["gj", "gj", "twisted"])
        stars = rng.randint(1, 16)
        rays = int(_log(rng, 500, 500000 if precision == "mixed" else 60000))
        rotation = int(precision == "fp64" and rays < 4000 and rng.random() < 0.5)
        return dict(kind=kind, n=max(1, rays // stars), stars=stars, theta=theta,
                    r_c=r_c if plasma == "gj" else min(r_c, 8.0),
                    span=_log(rng, 1.0, 100.0), plasma=plasma, rotation=rotation,
                    precision=precision, order=rng.choice(["index", "cost"]))
    if kind == "image":
        precision = rng.choice(["fp64", "mixed"])
        most = 256 if precision == "fp64" else 1024
        return dict(kind=kind, nx=int(_log(rng, 24, most)), ny=int(_log(rng, 24, most)),
                    incl=rng.uniform(5.0, 175.0), bmax=r_c * rng.uniform(1.2, 3.0),
                    theta=theta, r_c=r_c, precision=precision)
    if kind == "uneven":
        return dict(kind=kind, instances=rng.randint(2, 12), n=int(_log(rng, 1500, 60000)),
                    side=int(_log(rng, 30, 300)), theta=rng.uniform(0.0, 80.0), r_c=r_c,
                    span=_log(rng, 2.0, 60.0), precision="mixed")
    return dict(kind=kind, n=int(_log(rng, 300, 32768)), incl=rng.uniform(20.0, 160.0),
                theta=rng.uniform(5.0, 60.0), r_c=min(r_c, 4.0), kappa=_log(rng, 4.0, 415.0),
                sweep=rng.choice(["fp64", "fp64", "mixed"]))


# --- stars -------------------------------------------------------------------

def _params(theta, r_c, plasma="gj", rotation=0, weight=rt.WEIGHT_PAG, scale=1.0, phase=1):
    """Star keywords; the axion mass puts omega_p = m_a at r_c / scale^(2/3) radii on the
    axis (Goldreich-Julian), so ``scale`` multiplies the mass of the scan's first star."""
    if theta == 0.0:
        kw = dict(M_sun=1.4, R_km=10.0, B0_G=1e14, P_s=1.0, theta_m=0.0)
        m_a = 1.094e-6 * (20.0 / r_c) ** 1.5
    else:
        kw = dict(M_sun=1.5, R_km=11.0, B0_G=1.6e14, P_s=3.76, theta_m=math.radians(theta))
        m_a = 1.094e-6 * (20.0 / r_c) ** 1.5 * math.sqrt(1.6 / 3.76)
    kw.update(psi=0.0, m_a_eV=m_a * scale, g_GeVinv=1e-12, rho_GeV_cm3=0.45, v0_kms=200.0,
              dispersion=0, resonance=0, fa_model=0, weight_mode=weight, prop_metric=0,
              phase_mode=phase, plasma=PLASMA[plasma], rotation=rotation, plasma_a=0.0)
    if plasma == "twisted":
        kw["plasma_a"] = 4.0            # lambda = 20, psi = 0.2
        kw["m_a_eV"] *= 20.0            # the denser medium converts heavier axions
    return kw


def _scan(case):
    """The scan's stars: masses from that of r_c up to ``span`` times it."""
    n = case["stars"]
    return [_params(case["theta"], case["r_c"], case["plasma"], case.get("rotation", 0),
                    case.get("weight", rt.WEIGHT_PAG),
                    case["span"] ** (i / max(1, n - 1))) for i in range(n)]


def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _uniforms(n, seed):
    u = torch.rand((rt.UNIFORM_ROWS, n), dtype=F64, device=DEV, generator=_generator(seed))
    return u.clamp_(2.0 ** -54, 1.0 - 2.0 ** -53)


def _empty(*shape, dtype=F64):
    return torch.empty(shape, dtype=dtype, device=DEV)


# --- preparing and running ----------------------------------------------------

def prepare(case, seed):
    return globals()["_prepare_" + case["kind"]](case, seed)


def run(state):
    return state["run"](state)


def _points(case, seed):
    """Photon points between the surface and 100 radii, momenta of a few m_a."""
    kw = _params(case["theta"], case["r_c"], case["plasma"])
    n, g = case["n"], _generator(seed)
    d = torch.randn((3, n), dtype=F64, device=DEV, generator=g)
    k = torch.randn((3, n), dtype=F64, device=DEV, generator=g)
    u = torch.rand((3, n), dtype=F64, device=DEV, generator=g)
    st = _empty(rt.STATE_ROWS, n)
    st[:3] = d / d.norm(dim=0) * (kw["R_km"] * 1.3 * (80.0 ** u[0]))
    st[3:6] = k * (0.6 * kw["m_a_eV"])
    st[6] = 2e-7 * (0.1 + u[1])
    st[7] = 2.0 * math.pi * u[2]
    return kw, st


def _prepare_rhs(case, seed):
    kw, st = _points(case, seed)
    n = case["n"]
    return dict(run=_run_rhs, star=rt.Star(rt.make_params(**kw)), n=n, state=st, H=_empty(n),
                dydl=_empty(6, n))


def _run_rhs(s):
    rt.rt_hamilton_rhs(s["star"], s["n"], s["state"], s["H"], s["dydl"])
    return {"H": s["H"], "dydl": s["dydl"]}


def _batch(params, counts, seed):
    stars = [rt.Star(rt.make_params(**kw)) for kw in params]
    N = sum(counts)
    return dict(stars=stars, batch=rt.Batch(stars, counts), u=_uniforms(N, seed),
                state=_empty(rt.STATE_ROWS, N), weight=_empty(N),
                status=_empty(N, dtype=torch.uint8))


def _prepare_sample(case, seed):
    s = _batch(_scan(case), [case["n"]] * case["stars"], seed)
    s["run"] = _run_sample
    return s


def _run_sample(s):
    rt.rt_sample_batch(s["batch"], s["u"], s["state"], s["weight"], s["status"])
    return {"state": s["state"], "weight": s["weight"], "status": s["status"]}


def _rays(case, seed):
    """Rays as a trace leaves them: at 1000 radii, moving outwards, Maxwellian energies,
    weights over several decades, some captured and some without a conversion point."""
    kw = _params(30.0, 16.0)
    n, g = case["n"], _generator(seed)
    d = torch.randn((3, n), dtype=F64, device=DEV, generator=g)
    d /= d.norm(dim=0)
    v = torch.randn((3, n), dtype=F64, device=DEV, generator=g)
    w = torch.randn((2, n), dtype=F64, device=DEV, generator=g)
    u = torch.rand((1, n), dtype=F64, device=DEV, generator=g)
    v0 = 200.0 / 299792.458
    st = _empty(rt.STATE_ROWS, n)
    st[:3] = d * (1000.0 * kw["R_km"])
    st[3:6] = (d + 0.02 * v) * (kw["m_a_eV"] * v0)
    st[6] = 0.25 * v0 * v0 * (v * v).sum(0)
    st[7] = 0.0
    weight = torch.exp(2.0 * w[0]) * 1e6
    status = torch.full((n,), rt.RAY_NO_ROOT, dtype=torch.uint8, device=DEV)
    status[u[0] < case["landed"]] = rt.RAY_ESCAPED
    status[u[0] < 0.01 * case["landed"]] = rt.RAY_CAPTURED
    return kw, st, weight, status


def _prepare_bin(case, seed):
    kw, st, weight, status = _rays(case, seed)
    nth, nph, nnu = case["nth"], case["nph"], case["nnu"]
    return dict(run=_run_bin, star=rt.Star(rt.make_params(**kw)), n=case["n"], state=st,
                weight=weight, status=status, bins=(nth, nph, nnu), hist=_empty(nth, nph, nnu),
                sky=_empty(nth, nph), spec=_empty(nnu), oor=_empty(1))


def _run_bin(s):
    rt.rt_bin_spectrum(s["star"], s["n"], s["state"], s["weight"], s["status"], *s["bins"],
                       NU_LO, NU_HI, s["hist"], s["sky"], s["spec"], s["oor"])
    return {k: s[k] for k in ("hist", "sky", "spec", "oor")}


def _prepare_forward(case, seed):
    s = _batch(_scan(case), [case["n"]] * case["stars"], seed)
    s.update(run=_run_forward, hist=_empty(case["stars"], NTH, NPH, NNU),
             oor=_empty(case["stars"]),
             opts=rt.make_opts(rtol=RTOL[case["precision"]],
                               precision=PRECISION[case["precision"]],
                               claim_order=ORDER[case["order"]]))
    return s


def _run_forward(s):
    rt.rt_sample_batch(s["batch"], s["u"], s["state"], s["weight"], s["status"])
    rt.rt_trace_batch(s["batch"], s["state"], s["status"], opts=s["opts"])
    rt.rt_bin_batch(s["batch"], s["state"], s["weight"], s["status"], NTH, NPH, NNU, NU_LO,
                    NU_HI, s["hist"], s["oor"])
    return {"hist": s["hist"], "oor": s["oor"], "weight": s["weight"], "status": s["status"]}


def _prepare_image(case, seed):
    # the seed turns the observer and the star's phase a little: another image
    kw = _params(case["theta"], case["r_c"], phase=0)
    kw["psi"] = 1e-3 * (seed % 5003)
    nx, ny = case["nx"], case["ny"]
    incl = math.radians(case["incl"]) + 1e-5 * (seed % 4999)
    return dict(run=_run_image, star=rt.Star(rt.make_params(**kw)), nx=nx, ny=ny, incl=incl,
                bmax=case["bmax"], image=_empty(ny, nx), status=_empty(ny, nx, dtype=torch.uint8),
                ncross=_empty(ny, nx, dtype=torch.int32),
                opts=rt.make_opts(rtol=RTOL[case["precision"]],
                                  precision=PRECISION[case["precision"]]))


def _run_image(s):
    rt.rt_trace_backward(s["star"], s["nx"], s["ny"], s["incl"], 1e4, s["bmax"], s["image"],
                         s["status"], s["ncross"], opts=s["opts"])
    return {"image": s["image"], "status": s["status"], "ncross": s["ncross"]}


def _uneven(case):
    """Per instance: star keywords, rays (even instances) or image side (odd ones)."""
    out = []
    k = case["instances"]
    for i in range(k):
        f = ((5 * i + 2) % k) / max(1, k - 1)
        kw = _params(max(0.5, case["theta"] * (i + 1) / k), case["r_c"], phase=1 - i % 2,
                     scale=case["span"] ** f)
        out.append((kw, max(1, int(case["n"] * 60.0 ** -f)),
                    max(1, int(case["side"] * 8.0 ** -f))))
    return out


def _prepare_uneven(case, seed):
    inst = _uneven(case)
    fwd, bwd = inst[0::2], inst[1::2]
    s = _batch([x[0] for x in fwd], [x[1] for x in fwd], seed)
    bstars, descs = [], []
    for j, (kw, _, side) in enumerate(bwd):
        star = rt.Star(rt.make_params(**dict(kw, psi=1e-3 * ((seed + j) % 5003))))
        r_max = max((2.0 * star.info()["wp2_coef"]) ** (1.0 / 3.0), 1.5)
        bstars.append(star)
        descs.append((side, side + j % 2, 0.4 + 0.3 * j, 1e4, 1.3 * r_max, 0.0))
    P = sum(d[0] * d[1] for d in descs)
    s.update(run=_run_uneven, bstars=bstars, image=_empty(P),
             img_status=_empty(P, dtype=torch.uint8), ncross=_empty(P, dtype=torch.int32),
             hist=_empty(len(fwd), NTH, NPH, NNU), oor=_empty(len(fwd)),
             opts=rt.make_opts(rtol=RTOL[case["precision"]],
                               precision=PRECISION[case["precision"]]))
    rt.rt_batch_set_images(s["batch"], bstars, descs, s["image"], s["img_status"], s["ncross"])
    return s


def _run_uneven(s):
    out = _run_forward(s)
    out.update(image=s["image"], img_status=s["img_status"], ncross=s["ncross"])
    return out


def _prepare_gradient(case, seed):
    kw = _params(case["theta"], case["r_c"])
    p = torch.tensor([kw["m_a_eV"], kw["B0_G"], kw["theta_m"], kw["M_sun"], kw["R_km"],
                      math.radians(case["incl"])], dtype=F64)
    return dict(run=_run_gradient, log_p=torch.log(p), base=kw, u=_uniforms(case["n"], seed),
                kappa=case["kappa"], sweep=case["sweep"])


def _run_gradient(s):
    # a fit moves the logarithms of the parameters, whose units span forty decades
    log_p = s["log_p"].clone().requires_grad_(True)
    F = flux.line_flux(torch.exp(log_p), s["base"], s["u"], s["kappa"],
                       grad_precision=s["sweep"])
    F.backward()
    return {"F": F.detach(), "grad": log_p.grad}


# --- what a pass cannot do without ---------------------------------------------

def work(case):
    kind = case["kind"]
    if kind == "rhs":
        return {"bytes": 8.0 * case["n"] * (8 + 7), "flops": 230.0 * case["n"]}
    if kind == "sample":
        N = case["n"] * case["stars"]
        # the speed's inverse distribution and the resonance: two roots of about 60
        # operations for each of a few refinements, and the weight
        return {"bytes": N * (48.0 + 64.0 + 8.0 + 1.0), "flops": 600.0 * N}
    if kind == "bin":
        bins = case["nth"] * case["nph"] * (case["nnu"] + 1.0) + case["nnu"]
        return {"bytes": case["n"] * (1.0 + case["landed"] * 64.0) + 8.0 * bins,
                "flops": 100.0 * case["n"] * case["landed"]}
    if kind == "forward":
        N = case["n"] * case["stars"]
        return {"bytes": N * (48.0 + 8.0 + 1.0) + 8.0 * case["stars"] * NTH * NPH * NNU,
                "flops": N * STEPS[case["precision"]] * STEP_FLOPS}
    if kind == "image":
        N = case["nx"] * case["ny"]
        return {"bytes": 13.0 * N, "flops": N * STEPS[case["precision"]] * STEP_FLOPS}
    if kind == "uneven":
        inst = _uneven(case)
        rays = sum(x[1] for x in inst[0::2])
        pix = sum(x[2] * x[2] for x in inst[1::2])
        return {"bytes": rays * 57.0 + pix * 13.0 + 8.0 * len(inst[0::2]) * NTH * NPH * NNU,
                "flops": (rays + pix) * STEPS[case["precision"]] * STEP_FLOPS}
    # forward, then each step once more with its adjoint (about four times a step)
    return {"bytes": 48.0 * case["n"] + 56.0, "flops": 6.0 * case["n"] * 160.0 * STEP_FLOPS}


# --- values in 64 bits, in plain torch -------------------------------------------

HBARC_EV_KM, HBAR_EV_S, ALPHA = 1.973269804e-10, 6.582119569e-16, 7.2973525693e-3
ME_EV, EV_J, C_KM_S, GM_SUN_KM = 510998.95, 1.602176634e-19, 299792.458, 1.4766250


def exact(case, seed):
    """Right-hand side, samples and histograms from their defining formulas; a traced
    ray has no closed form (None)."""
    fn = globals().get("_exact_" + case["kind"])
    return fn(case, seed) if fn else None


def _constants(kw):
    e = math.sqrt(4.0 * math.pi * ALPHA)
    cm = HBARC_EV_KM * 1e5
    B0 = kw["B0_G"] * math.sqrt((1e-7 / EV_J) * cm ** 3 / (4.0 * math.pi))
    m = kw["m_a_eV"]
    R_eV = kw["R_km"] / HBARC_EV_KM
    if kw["plasma"] == rt.PLASMA_TWISTED:
        cp = e * kw["plasma_a"] * B0 / R_eV / ME_EV / (m * m)
    else:
        cp = e * (HBAR_EV_S * 2.0 * math.pi / kw["P_s"]) * B0 / ME_EV / (m * m)
    return dict(rs=2.0 * kw["M_sun"] * GM_SUN_KM / kw["R_km"], cp=cp, B0=B0, R_eV=R_eV,
                v0=kw["v0_kms"] / C_KM_S, n_inf=kw["rho_GeV_cm3"] * 1e9 * cm ** 3 / m,
                g=kw["g_GeVinv"] * 1e-9, rlc=C_KM_S * kw["P_s"] / (2.0 * math.pi * kw["R_km"]))


def _axis(kw, psi):
    st, ct = math.sin(kw["theta_m"]), math.cos(kw["theta_m"])
    return torch.stack([st * torch.cos(psi), st * torch.sin(psi), torch.full_like(psi, ct)])


def _density(kw, c, r, n, m):
    """omega_p^2 / m_a^2 at radius r along directions n."""
    mu = (m * n).sum(0)
    if kw["plasma"] == rt.PLASMA_TWISTED:
        return c["cp"] * (1.0 - mu * mu) / r ** 4
    return c["cp"] * (3.0 * n[2] * mu - m[2]).abs() / r ** 3


def _hamiltonian(kw, c, x, k, W2, m):
    r = (x * x).sum(0).sqrt()
    n = x / r
    A = 1.0 - c["rs"] / r
    kr, mu = (n * k).sum(0), (m * n).sum(0)
    P = _density(kw, c, r, n, m)
    b = 3.0 * mu * n - m
    ko = k + (A.sqrt() - 1.0) * kr * n
    Kp2 = (ko * b).sum(0) ** 2 / (3.0 * mu * mu + 1.0)
    return -W2 / A + (k * k).sum(0) + (A - 1.0) * kr * kr + P - P * A * Kp2 / W2


def _exact_rhs(case, seed):
    kw, st = _points(case, seed)
    c = _constants(kw)
    x = (st[:3] / kw["R_km"]).requires_grad_(True)
    k = (st[3:6] / kw["m_a_eV"]).requires_grad_(True)
    H = _hamiltonian(kw, c, x, k, (1.0 + st[6]) ** 2, _axis(kw, st[7]))
    gx, gk = torch.autograd.grad(H.sum(), (x, k))
    return {"H": H.detach(), "dydl": torch.cat([gk, -gx])}


def _maxwell_speed(u):
    """x with the speed distribution 4/sqrt(pi) int_0^x t^2 exp(-t^2) dt = u."""
    up = u > 0.5
    v = torch.where(up, 1.0 - u, u)
    a = 2.0 / math.sqrt(math.pi)
    lo, hi = torch.zeros_like(u), torch.full_like(u, 30.0)
    x = torch.full_like(u, 1.0876520317)
    for _ in range(90):
        e = torch.exp(-x * x)
        # below 0.1 the alternating series: erf(x) and its partner cancel there
        y = x * x
        ser = 2.0 * a * x * y * (1.0 / 3.0 - y * (1.0 / 5.0 - y * (1.0 / 14.0 - y * (
            1.0 / 54.0 - y * (1.0 / 264.0 - y * (1.0 / 1560.0 - y / 10800.0))))))
        low = torch.where(x < 0.1, ser, torch.erf(x) - a * x * e)
        q = torch.where(up, torch.erfc(x) + a * x * e, low)
        below = torch.where(up, q > v, q < v)
        lo, hi = torch.where(below, x, lo), torch.where(below, hi, x)
        step = (q - v) / (2.0 * a * y * e) * torch.where(up, -1.0, 1.0)
        new = x - step
        x = torch.where((new > lo) & (new < hi), new, 0.5 * (lo + hi))
    return x


def _exact_sample_star(kw, u):
    c = _constants(kw)
    n_s = u.shape[1]

    def direction(a, b):
        z = 1.0 - 2.0 * a
        s = ((1.0 - z) * (1.0 + z)).clamp(min=0.0).sqrt()
        return torch.stack([s * torch.cos(2.0 * math.pi * b), s * torch.sin(2.0 * math.pi * b), z])

    n, q = direction(u[0], u[1]), direction(u[2], u[3])
    kinf = _maxwell_speed(u[4]) * c["v0"]
    delta = kinf * kinf / ((1.0 + kinf * kinf).sqrt() + 1.0)
    W2 = (1.0 + delta) ** 2
    psi = 2.0 * math.pi * u[5]
    m = _axis(kw, psi)
    mu = (m * n).sum(0)
    bb = 3.0 * mu * mu + 1.0
    c2 = (q * (3.0 * mu * n - m)).sum(0) ** 2 / bb
    s2 = 1.0 - c2

    def G(r):
        K2 = W2 / (1.0 - c["rs"] / r) - 1.0
        return _density(kw, c, r, n, m) * (1.0 + K2 * s2) - (1.0 + K2)

    one = torch.ones_like(mu)
    ok = G(one) > 0.0
    lo, hi = one.clone(), torch.full_like(one, 4096.0)
    for _ in range(70):                      # the root by bisection, to rounding
        mid = 0.5 * (lo + hi)
        pos = G(mid) > 0.0
        lo, hi = torch.where(pos, mid, lo), torch.where(pos, hi, mid)
    r = 0.5 * (lo + hi)
    if kw["plasma"] == rt.PLASMA_TWISTED:
        ok = ok & (r < c["rlc"] * (1.0 - mu * mu))
    A = 1.0 - c["rs"] / r
    K2 = W2 / A - 1.0
    E2 = 1.0 + K2
    E = E2.sqrt()
    P = _density(kw, c, r, n, m)
    dP = -(4.0 if kw["plasma"] == rt.PLASMA_TWISTED else 3.0) * P / r
    dK2 = -W2 * c["rs"] / (r * r * A * A)
    dG = dP * (1.0 + K2 * s2) + P * s2 * dK2 - dK2
    hden = 2.0 * E * (E2 - K2 * P * c2 / E2)
    kloc = K2.sqrt()
    ma = kw["m_a_eV"]
    dh = (dG / hden).abs() * ma / c["R_eV"]
    W1 = 4.0 * math.pi * (r * c["R_eV"]) ** 2 * (kloc / kinf) * c["n_inf"] / (A * dh)
    W1 = W1 / n_s * (EV_J / HBAR_EV_S)
    if kw["weight_mode"] == rt.WEIGHT_PAG:
        D = c2 * P * (P - 2.0 * E2) + E2 * E2
        B = 0.5 * c["B0"] * bb.sqrt() / r ** 3
        w = W1 * 0.5 * math.pi * c["g"] ** 2 * B * B * (E2 * E2 * s2 / D) * (E * ma)
    else:
        # the resonance function's gradient at the conversion point, its leaf fixed
        X = (r * n).requires_grad_(True)
        R = (X * X).sum(0).sqrt()
        N = X / R
        MU = (m * N).sum(0)
        S2 = 1.0 - (q * (3.0 * MU * N - m)).sum(0) ** 2 / (3.0 * MU * MU + 1.0)
        KK = W2 / (1.0 - c["rs"] / R) - 1.0
        g = torch.autograd.grad((_density(kw, c, R, N, m) * (1.0 + KK * S2) - KK).sum(), X)[0]
        kg = (q * g).sum(0) + (A.sqrt() - 1.0) * (g * n).sum(0) * (q * n).sum(0)
        w = W1 * kloc * ma * (kg / hden).abs() * ma / c["R_eV"]
        if kw["weight_mode"] == rt.WEIGHT_RENORM:
            kc = (c["v0"] ** 2 + c["rs"] / r).sqrt() / c["v0"]
            per_cm3 = (HBARC_EV_KM * 1e5) ** 3
            w = w * (per_cm3 / (c["n_inf"] * kc)) / kloc / A.sqrt()
    nko = kloc * (n * q).sum(0)
    k = kloc * q + (1.0 / A.sqrt() - 1.0) * nko * n
    zero = torch.zeros_like(r)
    x = torch.where(ok, r * n, zero) * kw["R_km"]
    k = torch.where(ok, k, zero) * ma
    state = torch.cat([x, k, delta[None], psi[None]])
    status = torch.where(ok, rt.RAY_READY, rt.RAY_NO_ROOT).to(torch.uint8)
    return state.detach(), torch.where(ok, w, zero).detach(), status


def _exact_sample(case, seed):
    n, stars = case["n"], _scan(case)
    u = _uniforms(n * len(stars), seed)
    got = [_exact_sample_star(kw, u[:, i * n:(i + 1) * n]) for i, kw in enumerate(stars)]
    return {"state": torch.cat([g[0] for g in got], 1), "weight": torch.cat([g[1] for g in got]),
            "status": torch.cat([g[2] for g in got])}


def _exact_bin(case, seed):
    kw, st, weight, status = _rays(case, seed)
    c = _constants(kw)
    nth, nph, nnu = case["nth"], case["nph"], case["nnu"]
    x, k = st[:3] / kw["R_km"], st[3:6]
    r = (x * x).sum(0).sqrt()
    n = x / r
    o = k + ((1.0 - c["rs"] / r).sqrt() - 1.0) * (n * k).sum(0) * n
    th = torch.acos((o[2] / (o * o).sum(0).sqrt()).clamp(-1.0, 1.0))
    ph = torch.atan2(o[1], o[0])
    ph = torch.where(ph < 0.0, ph + 2.0 * math.pi, ph)
    y = st[6] / (0.5 * c["v0"] ** 2)
    esc = status == rt.RAY_ESCAPED
    inside = esc & (y >= NU_LO) & (y < NU_HI)
    i = (th / (math.pi / nth)).floor().long().clamp(max=nth - 1)
    j = (ph / (2.0 * math.pi / nph)).floor().long() % nph
    f = ((y - NU_LO) / ((NU_HI - NU_LO) / nnu)).floor().long().clamp(0, nnu - 1)
    flat = (i * nph + j) * nnu + f
    hist = torch.zeros(nth * nph * nnu, dtype=F64, device=st.device)
    hist.index_add_(0, flat[inside], weight[inside])
    hist = hist.reshape(nth, nph, nnu)
    return {"hist": hist, "sky": hist.sum(2), "spec": hist.sum((0, 1)),
            "oor": weight[esc & ~inside].sum().reshape(1)}
