"""The calls that a user of the light-curve library makes, as measurable cases.

A case is a dict of plain values.  ``listed()`` gives the fixed ones, ``draw(rng)`` one more of the
same ranges, ``prepare(case, seed)`` what a program holds before the call (a built model, times,
parameters, a cotangent), ``run(state)`` one pass through the public entry points, ``work(case)``
the bytes and operations that a pass cannot do without, and ``exact(case, seed)`` the outputs in
64 bits from plain torch: the same radial and (k, g) grids, orbit, area and averages, gradients by
autograd, none of the library's code.

Fields of a case
  mode       flux: Model.evaluate; fit: Model.flux and its backward pass; both: Model.prepare and
             Model.evaluate_both; host: Model.evaluate_host on pinned buffers, with the gradient
  npv, npt   parameter vectors and times (all passbands together)
  law        limb-darkening law
  precision  mixed or fp64
  npb        passbands; chromatic: one radius ratio per passband
  ss, cad    sub-exposures and exposure length (minutes) per passband, cycled over the passbands
  direct, shared  the direct model; one weight array per parameter vector
  params     prior: every vector another planet; posterior: vectors scattered about one planet
  times      sorted: uniform over 27.5 days; cadence: each passband at its own cadence, merged;
             transits: stretches about five transits; linear: one transit at a constant step;
             channels: every sorted time once per passband
"""
import math

import numpy as np
import torch

MINUTE = 1.0 / 1440.0
BJD = 2459000.5
NZIN, NZLIMB, ZCUT, NG, NK, K0, K1 = 200, 300, 0.7, 200, 60, 0.005, 0.3
NLDC = {"quadratic": 2, "quadratic_tri": 2, "nonlinear": 4, "tabulated": 0}


def _case(name, mode, npv, npt, law="quadratic_tri", precision="mixed", npb=1, chromatic=False, ss="1", cad="2",
          direct=False, shared=False, params="prior", times="sorted"):
    return dict(name=name, mode=mode, npv=npv, npt=npt, law=law, precision=precision, npb=npb, chromatic=chromatic,
                ss=ss, cad=cad, direct=direct, shared=shared, params=params, times=times)


def listed():
    return [
        # one light curve of one transit in FP64: a least-squares fit's function call, the smallest use
        _case("single_fp64", "flux", 1, 2000, law="quadratic", precision="fp64", params="circular", times="linear"),
        # one eccentric planet, 27 days at 2-minute cadence, 10 sub-exposures: a survey target's curve
        _case("single_ss10", "flux", 1, 19440, law="nonlinear", ss="10", times="cadence", params="posterior"),
        # a gradient-based sampler's step (a few chains) through autograd
        _case("sampler_grad", "fit", 16, 2000, params="posterior", times="transits"),
        # an ensemble sampler's likelihood: 200 walkers over five observed transits, a ragged length
        _case("ensemble", "flux", 200, 3001, params="posterior", times="transits"),
        # the same over a quarter of 30-minute exposures, 10 sub-exposures each
        _case("long_cadence", "flux", 100, 4407, law="quadratic", ss="10", cad="29.4", params="posterior",
              times="cadence"),
        # three bands with a radius ratio and coefficients each and mixed exposures: a joint fit's gradient
        _case("joint_fit", "fit", 256, 9001, law="nonlinear", npb=3, chromatic=True, ss="1,5,10", cad="2,5,10",
              params="posterior", times="cadence"),
        # a population drawn over the prior, light curves and gradients
        _case("population", "both", 4096, 20000),
        # the heterogeneous series: eight bands of numerical profiles, 1, 10 and 30 sub-exposures
        _case("heterogeneous", "flux", 2048, 60000, law="tabulated", npb=8, ss="1,10,30", cad="2,10,30",
              times="cadence"),
        # transmission spectroscopy: eight channels, the direct model with one weight array per vector
        _case("transmission", "both", 2048, 20000, law="quadratic", npb=8, chromatic=True, direct=True, shared=True,
              times="channels"),
        # the direct model (weights at each vector's own radius ratio) on one band
        _case("direct", "flux", 1000, 4999, law="quadratic", direct=True),
        # the FP64 form with its gradient, where ppm-level differences matter
        _case("population_fp64", "both", 512, 10007, law="quadratic", precision="fp64"),
        # data that live in host memory: pinned arrays in and out, with the gradient
        _case("host", "host", 512, 20000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    case = _drawn(rng)
    del case["name"]
    return case


def _drawn(rng):
    kind = rng.choice(["single", "ensemble", "sampler", "population", "heterogeneous", "joint", "transmission",
                       "direct", "fp64", "host"])
    law = rng.choice(["quadratic", "quadratic_tri", "nonlinear", "tabulated"])
    ss, cad = rng.choice([("1", "2"), ("1", "2"), ("5", "10"), ("10", "29.4")])
    if kind == "single":
        return _case("", "flux", 1, _log_int(rng, 200, 100000), law=law, ss=ss, cad=cad, params="posterior",
                     precision=rng.choice(["mixed", "mixed", "fp64"]), times=rng.choice(["cadence", "transits"]))
    if kind == "ensemble":
        return _case("", "flux", _log_int(rng, 8, 1000), _log_int(rng, 300, 20000), law=law, ss=ss, cad=cad,
                     params="posterior", times=rng.choice(["cadence", "transits"]))
    if kind == "sampler":
        return _case("", "fit", _log_int(rng, 1, 128), _log_int(rng, 300, 20000), law=law, ss=ss, cad=cad,
                     params="posterior", times=rng.choice(["cadence", "transits"]))
    if kind == "population":
        return _case("", rng.choice(["flux", "both"]), _log_int(rng, 256, 4096), _log_int(rng, 1500, 20000), law=law)
    if kind in ("heterogeneous", "joint"):
        s, c = rng.choice([("1,10,30", "2,10,30"), ("1,5,10", "2,5,10"), ("1", "2")])
        het = kind == "heterogeneous"
        return _case("", "flux" if het else "fit", _log_int(rng, 32, 1024), _log_int(rng, 2000, 40000),
                     law="tabulated" if het else rng.choice(["quadratic", "nonlinear"]), npb=rng.randint(2, 8),
                     chromatic=not het, ss=s, cad=c, params="prior" if het else "posterior", times="cadence")
    if kind == "transmission":
        npb = rng.randint(2, 8)
        return _case("", rng.choice(["flux", "both"]), _log_int(rng, 64, 1024), npb * _log_int(rng, 300, 2500),
                     law="quadratic", npb=npb, chromatic=True, direct=True, shared=True, times="channels")
    if kind == "direct":
        return _case("", rng.choice(["flux", "both"]), _log_int(rng, 16, 1500), _log_int(rng, 500, 10000), law=law,
                     direct=True)
    if kind == "fp64":
        return _case("", rng.choice(["flux", "both"]), _log_int(rng, 4, 512), _log_int(rng, 500, 10007), law=law,
                     precision="fp64", params=rng.choice(["prior", "posterior"]))
    return _case("", "host", _log_int(rng, 16, 512), _log_int(rng, 500, 20000), law=law, params="prior")


# ---- inputs ------------------------------------------------------------------


def _bernstein(beta, x):
    n = len(beta) - 1
    return sum(beta[m] * math.comb(n, m) * x ** m * (1.0 - x) ** (n - m) for m in range(n + 1))


def _coefficients(rng, law, n):
    """Limb-darkening coefficients (n, nldc) of positive, limb-darkened profiles."""
    if law == "quadratic":
        return np.stack([rng.uniform(0.1, 0.5, n), rng.uniform(0.0, 0.3, n)], axis=1)
    if law == "quadratic_tri":
        return np.stack([rng.uniform(0.05, 1.0, n), rng.uniform(0.0, 1.0, n)], axis=1)
    if law == "nonlinear":
        # ascending Bernstein coefficients in sqrt(mu), ending at 1, in powers of sqrt(mu)
        b0 = rng.uniform(0.05, 0.6, (n, 1))
        beta = np.concatenate([b0, np.sort(rng.uniform(0.0, 1.0, (n, 3)), axis=1) * (1.0 - b0) + b0,
                               np.ones((n, 1))], axis=1)
        p = np.zeros((n, 5))
        for m in range(5):
            for j in range(m, 5):
                p[:, j] += beta[:, m] * math.comb(4, m) * math.comb(4 - m, j - m) * (-1.0) ** (j - m)
        return p[:, 1:]
    return np.zeros((n, 0))


def _inputs(case, seed):
    """Host inputs of a case, from the seed alone."""
    rng = np.random.Generator(np.random.PCG64(seed))
    npv, npt, npb, law = case["npv"], case["npt"], case["npb"], case["law"]
    sss = [int(x) for x in case["ss"].split(",")]
    cads = [float(x) * MINUTE for x in case["cad"].split(",")]
    ss = np.array([sss[j % len(sss)] for j in range(npb)], np.int32)
    ex = np.array([cads[j % len(cads)] for j in range(npb)], np.float64)
    nkp, nldc = (npb if case["chromatic"] else 1), NLDC[law]
    if case["params"] == "prior":
        k = rng.uniform(0.01, 0.25, npv)
        a = rng.uniform(3.0, 30.0, npv)
        b = rng.uniform(0.0, 1.0, npv) * (1.0 + k)
        P = rng.uniform(1.0, 10.0, npv)
        e = rng.uniform(0.0, 1.0, npv) * np.minimum(0.5, 1.0 - (1.5 + k) / a)
        w = rng.uniform(0.0, 2.0 * np.pi, npv)
        t0 = rng.uniform(0.0, 1.0, npv) * P
        start = 0.0
        spread = 0.03
    else:
        # one planet; its vectors scatter as a posterior does
        one = npv == 1
        tk, ta, tb, tP = rng.uniform(0.05, 0.15), rng.uniform(6.0, 16.0), rng.uniform(0.0, 0.6), rng.uniform(2.0, 6.0)
        circ = case["params"] == "circular"
        te, tw = (0.0, 0.0) if circ else (rng.uniform(0.05, 0.35), rng.uniform(0.0, 2.0 * np.pi))
        s = 0.0 if one else 1.0
        start = 0.0 if circ else BJD

        def scat(x, sd):
            return x + s * sd * rng.standard_normal(npv)
        tt0 = 0.0 if circ else start + rng.uniform(0.0, tP)
        k, a, b, P = scat(tk, 0.005 * tk), scat(ta, 0.01 * ta), np.abs(scat(tb, 0.02)), scat(tP, 1e-5)
        e, w, t0 = np.clip(scat(te, 0.01), 0.0, 0.45), scat(tw, 0.02), scat(tt0, 2e-4)
        spread = 0.02
    cols = [t0, P, a, b, e, w]
    if case["chromatic"]:
        cols += [k * (1.0 + spread * rng.uniform(-1.0, 1.0, npv)) for _ in range(npb)]
    else:
        cols += [k]
    for _ in range(npb):
        if case["params"] == "prior":
            c = _coefficients(rng, law, npv)
        else:
            c = _coefficients(rng, law, 1) * (1.0 + (0.02 if npv > 1 else 0.0) * rng.uniform(-1.0, 1.0, (npv, nldc)))
            if law == "quadratic_tri":
                c = np.clip(c, 0.02, 0.98)
        cols += list(c.T)
    params = np.stack(cols, axis=1)
    pb = np.zeros(npt, np.int32)
    if case["times"] == "linear":
        times = np.linspace(-0.15, 0.15, npt)
    elif case["times"] == "transits":
        half = 2.5 * tP * (1.0 + tk) / (np.pi * ta)
        times = np.sort(tt0 + tP * rng.integers(0, 5, npt) + half * rng.uniform(-1.0, 1.0, npt))
    elif case["times"] == "cadence":
        pb = (np.arange(npt) % npb).astype(np.int32)
        times = start + ex[pb] * (np.arange(npt) // npb)
        order = np.argsort(times, kind="stable")
        times, pb = times[order], pb[order]
    elif case["times"] == "channels":
        base = np.sort(rng.uniform(0.0, 27.5, npt // npb))
        times, pb = np.repeat(base, npb), np.tile(np.arange(npb, dtype=np.int32), npt // npb)
    else:
        times = np.sort(start + rng.uniform(0.0, 27.5, npt))
    profiles = None
    if law == "tabulated":
        mu = np.linspace(0.0, 1.0, 500)
        profiles = []
        for _ in range(npb):
            b0 = rng.uniform(0.05, 0.4)
            profiles.append((mu, _bernstein(np.concatenate([[b0], np.sort(rng.uniform(b0, 1.0, 5)), [1.0]]), mu)))
    gbar = rng.standard_normal((npv, npt), dtype=np.float32) if case["mode"] != "flux" else None
    return dict(times=times, pb=pb, params=params, ss=ss, ex=ex, profiles=profiles, gbar=gbar, nkp=nkp, nldc=nldc)


def prepare(case, seed):
    from paper_2009_08500_gb300 import rr
    inp = _inputs(case, seed)
    m = rr.Model(case["law"], case["npb"], case["chromatic"], case["precision"],
                 dict(zcut=ZCUT, nzin=NZIN, nzlimb=NZLIMB, ng=NG, nk=NK, k0=K0, k1=K1), direct=case["direct"],
                 shared_weights=case["shared"])
    if inp["profiles"]:
        for j, (mu, it) in enumerate(inp["profiles"]):
            m.set_ld_profile(j, mu, it)
    m.build()
    st = dict(mode=case["mode"], model=m, ss=inp["ss"], ex=inp["ex"])
    multi = case["npb"] > 1
    if case["mode"] == "host":
        def pin(x):
            return torch.from_numpy(np.ascontiguousarray(x)).pin_memory()
        npv, npt = case["npv"], case["npt"]
        st.update(times=pin(inp["times"]), params=pin(inp["params"]), pb=pin(inp["pb"]) if multi else None,
                  gbar=pin(inp["gbar"]).to(m.dtype),
                  out=torch.empty((npv, npt), dtype=m.dtype, pin_memory=True),
                  grad_out=torch.empty((npv, m.nparam), dtype=torch.float64, pin_memory=True),
                  status_out=torch.empty((npv,), dtype=torch.int32, pin_memory=True))
        return st
    st.update(times=torch.as_tensor(inp["times"], device=m.device), params=torch.as_tensor(inp["params"], device=m.device),
              pb=torch.as_tensor(inp["pb"], device=m.device) if multi else None)
    if inp["gbar"] is not None:
        st["gbar"] = torch.as_tensor(inp["gbar"], device=m.device).to(m.dtype)
    if case["mode"] == "fit":
        st["params"].requires_grad_(True)
    return st


def run(state):
    m, t, p, pb, ss, ex = (state[x] for x in ("model", "times", "params", "pb", "ss", "ex"))
    if state["mode"] == "flux":
        return m.evaluate(t, p, pb, ss, ex)
    if state["mode"] == "fit":
        f = m.flux(t, p, pb, ss, ex)
        g, = torch.autograd.grad(f, p, state["gbar"])
        return f.detach(), g
    if state["mode"] == "both":
        ws = m.prepare(t, p, pb, ss, ex)
        return m.evaluate_both(t, p, state["gbar"], ws, pb, ss, ex)
    return m.evaluate_host(t, p, pb, ss, ex, grad_flux=state["gbar"], out=state["out"], grad_out=state["grad_out"],
                           status_out=state["status_out"])


def work(case):
    """Bytes: every input read and every output written once.  Operations: the exposure samples inside
    a transit (about 3%, and 20% of the times about transits) at about 120 operations forward and 260 with
    the gradient, and a lens area of 80 operations per covered annulus edge
    (about 100) and g node of a direct model's row."""
    npv, npt, npb = case["npv"], case["npt"], case["npb"]
    elem = 8 if case["precision"] == "fp64" else 4
    grad = case["mode"] != "flux"
    nkp, nldc = (npb if case["chromatic"] else 1), NLDC[case["law"]]
    nparam = 6 + nkp + npb * nldc
    nbytes = npt * (8 + (4 if npb > 1 else 0)) + npv * nparam * 8 + npv * npt * elem
    if grad:
        nbytes += npv * npt * elem + npv * nparam * 8
    sss = [int(x) for x in case["ss"].split(",")]
    mean_ss = sum(sss[j % len(sss)] for j in range(npb)) / npb
    duty = 0.2 if case["times"] in ("transits", "linear") else 0.03
    flops = npv * npt * mean_ss * duty * (260 if grad else 120)
    if case["direct"]:
        flops += npv * (1 if case["shared"] else nkp) * NG * 100 * 80
    return {"bytes": float(nbytes), "flops": float(flops)}


# ---- the same outputs in 64 bits ----------------------------------------------


def _grid():
    ze = np.empty(NZIN + NZLIMB + 1)
    ze[:NZIN + 1] = np.arange(NZIN + 1) * ZCUT / NZIN
    m = np.sqrt(1.0 - ZCUT ** 2) * (1.0 - np.arange(1, NZLIMB + 1) / NZLIMB)
    ze[NZIN + 1:] = np.sqrt(1.0 - m * m)
    zm = 0.5 * (ze[1:] + ze[:-1])
    return ze, np.sqrt(1.0 - zm * zm)


def _bases(case, inp, mu):
    """Profile bases at the bin means (nb, nz) and their disk integrals."""
    law = case["law"]
    if law == "tabulated":
        B = np.stack([np.interp(mu, m, i) for m, i in inp["profiles"]])
        I = []
        for m, i in inp["profiles"]:
            d = np.diff(m)
            I.append(2 * np.pi * np.sum(d / 6 * (i[:-1] * (2 * m[:-1] + m[1:]) + i[1:] * (m[:-1] + 2 * m[1:]))))
        return B, np.array(I)
    one = np.ones_like(mu)
    if law == "nonlinear":
        return (np.stack([one] + [-(1.0 - mu ** (0.5 * n)) for n in range(1, 5)]),
                np.array([np.pi] + [-np.pi * n / (n + 4.0) for n in range(1, 5)]))
    return np.stack([one, -(1 - mu), -(1 - mu) ** 2]), np.array([np.pi, -np.pi / 3, -np.pi / 6])


def _lens(r, k, c):
    """Area common to disks of radii r and k at distance c (differentiable away from the contacts)."""
    h = (r + k - c) * (c + (r - k)) * (c - (r - k)) * (c + (r + k))
    ins = (c < r + k) & (c > (r - k).abs()) & (h > 0)
    K = torch.where(ins, h, torch.ones_like(h)).sqrt()
    lens = r * r * torch.atan2(K, c * c + (r * r - k * k)) + k * k * torch.atan2(K, c * c + (k * k - r * r)) - 0.5 * K
    small = torch.where(r < k, r.expand_as(h), k.expand_as(h))
    return torch.where(ins, lens, torch.where(c >= r + k, torch.zeros_like(h), math.pi * small * small))


def _projections(kv, B, ze):
    """Rows (n, nb, NG) of the weights at radius ratios kv, projected onto the bases B."""
    g = torch.arange(NG, dtype=torch.float64, device=kv.device) * (1.0 / (NG - 1))
    k = kv[:, None, None]
    c = g[None, :-1, None] * (1.0 + k)
    a = _lens(ze[None, None, :], k, c)
    w = (a[:, :, 1:] - a[:, :, :-1]) / a[:, :, -1:]
    T = torch.einsum("ngz,bz->nbg", w, B)
    return torch.cat([T, B[None, :, -1:].expand(T.shape[0], -1, 1)], dim=2)


def exact(case, seed):
    inp = _inputs(case, seed)
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")

    def dv(x, dt=torch.float64):
        return torch.as_tensor(x, dtype=dt, device=dev)
    ze_h, mu_h = _grid()
    B_h, I_h = _bases(case, inp, mu_h)
    ze, B, Istar = dv(ze_h), dv(B_h), dv(I_h)
    npv, npt, npb, nkp, nldc = case["npv"], case["npt"], case["npb"], inp["nkp"], inp["nldc"]
    tab, grad = case["law"] == "tabulated", case["mode"] != "flux"
    kgrid = K0 + (K1 - K0) / (NK - 1) * dv(np.arange(NK))
    T = None if case["direct"] else _projections(kgrid, B, ze)       # (NK, nb, NG)
    # every exposure sample: time, its index, passband, share of the mean
    ssn, times, pb = inp["ss"], inp["times"], inp["pb"]
    n_of = ssn[pb]
    idx = np.repeat(np.arange(npt), n_of)
    sub = np.arange(idx.size) - np.repeat(np.cumsum(n_of) - n_of, n_of)
    s_pb = pb[idx]
    off = np.where(ssn[s_pb] > 1, inp["ex"][s_pb] * ((sub + 0.5) / ssn[s_pb] - 0.5), 0.0)
    s_t, s_i, s_pb, s_w = dv(times[idx] + off), dv(idx, torch.int64), dv(s_pb, torch.int64), dv(1.0 / n_of[idx])
    params = dv(inp["params"])
    flux = torch.ones((npv, npt), dtype=torch.float64, device=dev)
    gout = torch.zeros((npv, params.shape[1]), dtype=torch.float64, device=dev)
    step = max(1, min(npv, 30_000_000 // max(1, s_t.numel()), 128 if case["direct"] else npv))
    for p0 in range(0, npv, step):
        P_ = params[p0:p0 + step].clone().requires_grad_(grad)
        n = P_.shape[0]
        with torch.no_grad():
            # samples within a generous window of a conjunction
            T0, P, a, b, e, w = (P_[:, j] for j in range(6))
            kmax = P_[:, 6:6 + nkp].max(dim=1).values
            d = torch.asin(((1 + kmax) / (a * (1 - e))).clamp(max=1.0))
            f0 = 0.5 * math.pi - w

            def M_of(f):
                E = torch.atan2((1 - e * e).sqrt() * torch.sin(f), e + torch.cos(f))
                return E - e * torch.sin(E)
            M0 = M_of(f0)
            tp = 2 * math.pi
            win = torch.maximum(torch.remainder(M_of(f0 + d) - M0, tp), torch.remainder(M0 - M_of(f0 - d), tp))
            win = win * 1.001 + 1e-6
            ph = (s_t[None, :] - T0[:, None]) / P[:, None]
            vi, si = (tp * (ph - ph.round()).abs() <= win[:, None]).nonzero(as_tuple=True)
            del ph
        with torch.enable_grad() if grad else torch.no_grad():
            rows = P_[vi]
            T0, P, a, b, e, w = (rows[:, j] for j in range(6))
            q = s_pb[si]
            kcol = P_[:, 6:6 + nkp]
            k = kcol[vi, q if case["chromatic"] else torch.zeros_like(q)]
            dt = s_t[si] - T0
            m = (dt / P).detach().round()
            tau = dt - m * P
            f0 = 0.5 * math.pi - w
            sq = (1 - e * e).sqrt()
            E0 = torch.atan2(sq * torch.sin(f0), e + torch.cos(f0))
            M = E0 - e * torch.sin(E0) + 2 * math.pi * tau / P
            with torch.no_grad():
                E = M + e * torch.sin(M)
                for _ in range(14):
                    E = E - (E - e * torch.sin(E) - M) / (1 - e * torch.cos(E))
            E = E - (E - e * torch.sin(E) - M) / (1 - e * torch.cos(E)).detach()
            X, Y = torch.cos(E) - e, sq * torch.sin(E)
            cw, sw = torch.cos(w), torch.sin(w)
            Px, Py = X * cw - Y * sw, X * sw + Y * cw
            z = ((a * Px) ** 2 + (b * Py) ** 2).sqrt()
            hit = ((Py > 0) & (z < 1 + k)).nonzero(as_tuple=True)[0]
            vi, si, q, k, z = vi[hit], si[hit], q[hit], k[hit], z[hit]
            A = _lens(torch.ones_like(k), k, z)
            x = z / (1 + k) * (NG - 1)
            ig = x.detach().floor().long().clamp(0, NG - 2)
            al = x - ig
            # the projections of each sample's row at its two g nodes
            if case["direct"]:
                kr = kcol.mean(dim=1) if case["shared"] else kcol.reshape(-1)
                R = _projections(kr, B, ze)
                row = vi if (case["shared"] or not case["chromatic"]) else vi * nkp + q

                def at(bb, i):
                    return R[row, bb, i]
            else:
                kw = kcol.mean(dim=1)[vi] if case["shared"] else k
                xk = (kw - K0) / ((K1 - K0) / (NK - 1))
                ik = xk.detach().floor().long().clamp(0, NK - 2)
                ak = xk - ik

                def at(bb, i):
                    return (1 - ak) * T[ik, bb, i] + ak * T[ik + 1, bb, i]

            def lerp(bb):
                lo = at(bb, ig)
                return lo + al * (at(bb, ig + 1) - lo)
            if tab:
                Ib = lerp(q) / Istar[q]
            else:
                base = 6 + nkp + q * nldc
                u = [P_[vi, base + j] for j in range(nldc)]
                if case["law"] == "quadratic_tri":
                    u = [2 * u[0].sqrt() * u[1], u[0].sqrt() * (1 - 2 * u[1])]
                zero = torch.zeros_like(q)
                num, den = lerp(zero), Istar[0]
                for j in range(nldc):
                    num = num + u[j] * lerp(zero + 1 + j)
                    den = den + u[j] * Istar[1 + j]
                Ib = num / den
            delta = A * Ib * s_w[si]
            out = torch.ones(n * npt, dtype=torch.float64, device=dev)
            out.index_add_(0, vi * npt + s_i[si], -delta.detach())
            flux[p0:p0 + n] = out.view(n, npt)
            if grad:
                gb = dv(inp["gbar"][p0:p0 + n])
                gout[p0:p0 + n], = torch.autograd.grad(-(delta * gb[vi, s_i[si]]).sum(), P_)
    if not grad:
        return flux
    if case["mode"] == "host":
        return flux.cpu(), gout.cpu(), None
    return flux, gout
