"""Cases that the library's speed is measured on.

One case is one call pattern of a solver on the seeded 9/21, 53/325 and 160/900
mechanisms: how many states it has in hand, which outputs it asks for and in which
precision.  ``listed`` names fixed ones, ``draw`` gives others of the same ranges.

States are the workload's (T uniform, p log-uniform or one atmosphere, Y Dirichlet).  Cases
that return rates draw T from 700 K up: below that the synthetic equilibrium constants push
single reverse rates beyond 1e150, and the 2-norm of an output would overflow float64.
Transport alone takes the full range from 300 K.
"""
import math
import os

import numpy as np
import torch

from paper_2411_02640_gb300 import kx, synth

H2, GRI, LARGE = "h2o2_9_21", "gri_53_325", "large_160_900"
N_S = {H2: 9, GRI: 53, LARGE: 160}
N_R = {H2: 21, GRI: 325, LARGE: 900}

# The most states that a drawn case of a call has, for 53/325 (about 10 ms a pass); the other
# mechanisms' limits follow from their size.
MOST = {"step": 1 << 19, "rates": 1 << 20, "transport": 1 << 20, "vjp": 1 << 18, "rop": 1 << 17, "host": 1 << 18}
SHARE = {H2: 1.0, GRI: 1.0, LARGE: 1.0 / 16}


def listed():
    def case(name, call, mech, n, precision="fp64"):
        return {"name": name, "call": call, "mech": mech, "n": n, "precision": precision}

    return [
        # Everything that one time step of a reacting-flow solver needs, on a small hydrogen
        # problem: a handful of microseconds of work, where launches and latency count.
        case("step_h2_4096", "step", H2, 4096),
        # The same on one small block of a methane flame, a ragged number of cells.
        case("step_gri_997", "step", GRI, 997),
        # A rank's ordinary share of a mesh, mixed precision, one cell short of a power of two.
        case("step_gri_mixed_16383", "step", GRI, 16383, "mixed"),
        # The source terms of a large mesh (the benchmark's size).
        case("rates_gri_1m", "rates", GRI, 1 << 20),
        # Its transport coefficients.
        case("transport_gri_1m", "transport", GRI, 1 << 20),
        # The two in mixed precision, on an odd number of cells.
        case("rates_gri_mixed_300001", "rates", GRI, 300001, "mixed"),
        case("transport_gri_mixed_300001", "transport", GRI, 300001, "mixed"),
        # A large hydrocarbon mechanism's source terms.
        case("rates_large_200003", "rates", LARGE, 200003),
        # One vector-Jacobian product of an implicit integrator's Newton step: a block of cells
        # that is still igniting, and a whole mesh.
        case("vjp_gri_4095", "vjp", GRI, 4095),
        case("vjp_gri_262144", "vjp", GRI, 1 << 18),
        # Rates of progress of every reaction, for a reaction-path analysis of a snapshot.
        case("rop_gri_20001", "rop", GRI, 20001),
        # A solver whose state lives in host memory: all outputs, through the pipelined host call.
        case("host_gri_200000", "host", GRI, 200000),
    ]


def draw(rng):
    call = rng.choice(("step", "step", "rates", "rates", "transport", "transport", "vjp", "rop", "host"))
    mech = rng.choice((H2, GRI, GRI, GRI, LARGE))
    if call in ("rop", "host") and mech == LARGE:
        mech = GRI
    precision = "fp64" if call == "vjp" else rng.choice(("fp64", "fp64", "mixed"))
    least = 4096 if call == "host" else 64
    n = int(round(math.exp(rng.uniform(math.log(least), math.log(MOST[call] * SHARE[mech])))))
    if rng.random() < 0.5:
        n |= 1
    return {"call": call, "mech": mech, "n": n, "precision": precision}


# ------------------------------------------------------------------ what a program has in hand

_handles = {}


def _handle(mech):
    """A program loads a mechanism once and keeps it."""
    if mech not in _handles:
        path = synth.mechanism_file(mech, os.path.join(".kxcache", "mech"))
        _handles[mech] = kx.Mechanism(path, cache_dir=os.path.join(".kxcache", "kernels"))
    return _handles[mech]


def _states(case, seed):
    spec = synth.STATE_SPECS[case["mech"]]
    if case["call"] != "transport":
        spec = synth.StateSpec((700.0, spec.T_range[1]), spec.p_atm_range, spec.alpha, spec.seed)
    return synth.make_states_torch(N_S[case["mech"]], spec, case["n"], seed)


def prepare(case, seed):
    h = _handle(case["mech"])
    T, p, Y = _states(case, seed)
    state = {"case": case, "h": h, "T": T, "p": p, "Y": Y}
    n, ns = case["n"], N_S[case["mech"]]
    if case["call"] == "vjp":
        g = torch.Generator(device="cuda")
        g.manual_seed(seed + 1)
        state["v"] = torch.randn((ns, n), dtype=torch.float64, device="cuda", generator=g)
    elif case["call"] == "host":
        for k in ("T", "p", "Y"):
            host = torch.empty(state[k].shape, dtype=torch.float64, pin_memory=True)
            host.copy_(state[k])
            state[k] = host
        state["out"] = {k: torch.empty((ns, n) if k in ("wdot", "Dk") else (n,), dtype=torch.float64, pin_memory=True)
                        for k in ("wdot", "cp", "h", "mu", "lam", "Dk")}
        chunk = min(n, 1 << 17)
        state["ws"] = torch.empty(2 * chunk * h.evaluate_host_bytes_per_state(7) + 4096, dtype=torch.uint8, device="cuda")
        state["streams"] = (torch.cuda.Stream(), torch.cuda.Stream())
    return state


def run(state):
    case, h = state["case"], state["h"]
    T, p, Y, prec, call = state["T"], state["p"], state["Y"], case["precision"], case["call"]
    if call == "rates":
        return {"wdot": h.production_rates(T, p, Y, precision=prec)}
    if call == "transport":
        mu, lam, Dk = h.transport(T, p, Y, precision=prec)
        return {"mu": mu, "lam": lam, "Dk": Dk}
    if call == "step":
        wdot = h.production_rates(T, p, Y, precision=prec)
        cp, hm = h.thermo(T, p, Y)
        mu, lam, Dk = h.transport(T, p, Y, precision=prec)
        return {"wdot": wdot, "cp": cp, "h": hm, "mu": mu, "lam": lam, "Dk": Dk}
    if call == "vjp":
        gT, gY = h.production_rates_vjp(T, p, Y, state["v"])
        return {"gT": gT, "gY": gY}
    if call == "rop":
        return {"q": h.rates_of_progress(T, p, Y, precision=prec)}
    h.evaluate_host(T, p, Y, state["out"], outputs=7, precision=prec, workspace=state["ws"], streams=state["streams"])
    for s in state["streams"]:   # the outputs are read by the host
        s.synchronize()
    return state["out"]


# ------------------------------------------------------------------ what a pass cannot do without

def work(case):
    """Bytes: T, p, Y (and the cotangents) once, each output once.  Operations: one per plain
    operation of the formulas, 20 for an exponential, a logarithm or a power."""
    ns, nr, n, call = N_S[case["mech"]], N_R[case["mech"]], case["n"], case["call"]
    rates = nr * (2 * 20 + 20) + ns * (2 * 20 + 12)
    thermo = ns * 22
    # degree-4 fits; Wilke's sums over all pairs; D_kj once for each unordered pair
    transport = ns * (2 * (8 + 20) + 40) + ns * ns * 6 + ns * (ns + 1) // 2 * (8 + 20 + 4)
    words, flops = {"rates": (ns, rates), "thermo": (2, thermo), "transport": (ns + 2, transport),
                    "step": (2 * ns + 4, rates + thermo + transport), "host": (2 * ns + 4, rates + thermo + transport),
                    "vjp": (2 * ns + 1, 3 * rates), "rop": (nr, rates)}[call]
    return {"bytes": 8.0 * n * (ns + 2 + words), "flops": float(flops) * n}


def tolerance(case):
    """About four times the error against 64 bits that the outputs show.  Transport is relative to
    each value (2e-14 in float pairs, 1.7e-7 in float32).  Rates, their products and the adjoint
    carry the rounding of logarithms of size ~100-1000 (up to 2e-12 in float pairs, 2e-5 mixed), and
    the 2-norm lies in the few coldest states: a small net rate of such a state is off by that
    share of the state's largest rate, which may be 1e4 times the root mean square."""
    if case["call"] == "transport":
        return {"rel": 1e-6, "max": 1e-5} if case["precision"] == "mixed" else {"rel": 1e-13, "max": 2e-12}
    return {"rel": 1e-4, "max": 0.5} if case["precision"] == "mixed" else {"rel": 1e-11, "max": 1e-7}


# ------------------------------------------------------------------ the same in 64 bits, in plain torch

R_U, P_ATM = synth.R_U, synth.P_ATM


def _dev(a):
    return torch.tensor(np.asarray(a, dtype=np.float64), device="cuda")


def _powers(T, k):
    return torch.stack([T ** i for i in range(k)])


def _nasa(m, T):
    """cp/R, H/RT, S/R [N_s, n] (NASA-7, the low block below T_mid)."""
    lo, hi, mid = _dev(m.nasa_lo), _dev(m.nasa_hi), _dev(m.nasa_T)[:, 1]
    low = T[None, :] < mid[:, None]
    a = [torch.where(low, lo[:, i:i + 1], hi[:, i:i + 1]) for i in range(7)]
    cp = a[0] + T * (a[1] + T * (a[2] + T * (a[3] + T * a[4])))
    h = a[0] + T * (a[1] / 2 + T * (a[2] / 3 + T * (a[3] / 4 + T * a[4] / 5))) + a[5] / T
    s = a[0] * torch.log(T) + T * (a[1] + T * (a[2] / 2 + T * (a[3] / 3 + T * a[4] / 4))) + a[6]
    return cp, h, s


def _arr(r, T):
    return r[0] * T ** r[1] * torch.exp(-r[2] / T)


def _progress(m, T, p, Y):
    """q_i of every reaction, one at a time, and its net stoichiometry."""
    W = _dev(m.W)
    sigma = (Y / W[:, None]).sum(0)
    C = list((p / (R_U * T * sigma))[None, :] * (Y / W[:, None]))
    _, h, s = _nasa(m, T)
    G = list(h - s)
    Call = torch.stack(C)
    log10 = math.log(10.0)
    for r in m.reactions:
        X = None
        if r.uses_third_body():
            if r.collider is not None:
                X = C[r.collider]
            else:
                eff = np.full(m.n_species, float(r.default_eff))
                for k, e in r.efficiencies.items():
                    eff[k] = e
                X = (_dev(eff)[:, None] * Call).sum(0)
        kf = _arr(r.rate, T)
        if r.kind == "falloff":
            pr = torch.clamp(_arr(r.rate_low, T) * X / kf, min=1e-300)
            blend = pr / (1 + pr)
            if r.troe is not None:
                al, t3, t1, t2 = r.troe
                lfc = torch.log10((1 - al) * torch.exp(-T / t3) + al * torch.exp(-T / t1) + torch.exp(-t2 / T))
                c, nn, lp = -0.4 - 0.67 * lfc, 0.75 - 1.27 * lfc, torch.log10(pr)
                f = (lp + c) / (nn - 0.14 * (lp + c))
                blend = blend * torch.exp(log10 * lfc / (1 + f * f))
            kf = kf * blend
        elif r.kind not in ("elementary", "three_body"):
            raise ValueError(r.kind)
        fwd = kf
        for k, nu in r.reactants:
            fwd = fwd * (C[k] if nu == 1 else C[k] ** nu)
        q = fwd
        if r.reversible:
            sg, sn = 0.0, 0
            for k, nu in r.products:
                sg, sn = sg + nu * G[k], sn + nu
            for k, nu in r.reactants:
                sg, sn = sg - nu * G[k], sn - nu
            rev = kf * torch.exp(sg) * (P_ATM / (R_U * T)) ** (-sn)
            for k, nu in r.products:
                rev = rev * (C[k] if nu == 1 else C[k] ** nu)
            q = fwd - rev
        if r.kind == "three_body":
            q = q * X
        yield r, q


def _wdot(m, T, p, Y):
    w = [None] * m.n_species
    for r, q in _progress(m, T, p, Y):
        for side, sign in ((r.reactants, -1), (r.products, 1)):
            for k, nu in side:
                w[k] = sign * nu * q if w[k] is None else w[k] + sign * nu * q
    return torch.stack([torch.zeros_like(T) if x is None else x for x in w])


def _thermo(m, T, Y):
    cp, h, _ = _nasa(m, T)
    y = Y * (R_U / _dev(m.W))[:, None]
    return (y * cp).sum(0), (y * h).sum(0) * T


def _transport(m, T, p, Y):
    W = _dev(m.W)
    L = torch.log(T)
    Lp = _powers(L, 5)
    X = Y / W[:, None]
    X = X / X.sum(0)
    eta, lam = torch.exp(_dev(m.eta_fit) @ Lp), torch.exp(_dev(m.lam_fit) @ Lp)
    mu = torch.zeros_like(T)
    for k in range(m.n_species):
        phi = (8.0 ** -0.5 * (1 + W[k] / W) ** -0.5)[:, None] * (1 + (eta[k] / eta) ** 0.5 * ((W / W[k]) ** 0.25)[:, None]) ** 2
        mu += X[k] * eta[k] / (X * phi).sum(0)
    lam = 0.5 * ((X * lam).sum(0) + 1 / (X / lam).sum(0))
    Wx = X * W[:, None]
    wbar = Wx.sum(0)
    dif, D = _dev(m.diff_fit), []
    for k in range(m.n_species):
        x = X * torch.exp(-(dif[k] @ Lp))
        x[k] = 0.0
        wx = Wx.clone()
        wx[k] = 0.0
        D.append(wx.sum(0) / wbar / x.sum(0) * (P_ATM / p))
    return mu, lam, torch.stack(D)


def exact(case, seed):
    m = synth.mechanism(case["mech"])
    T, p, Y = _states(case, seed)
    call, n = case["call"], case["n"]
    v = prepare(case, seed)["v"] if call == "vjp" else None
    got = {}
    step = 1 << (13 if call == "vjp" else 15 if case["mech"] == LARGE else 16)
    for a in range(0, n, step):
        t, q, y = T[a:a + step], p[a:a + step], Y[:, a:a + step].contiguous()
        part = {}
        if call in ("rates", "step", "host"):
            part["wdot"] = _wdot(m, t, q, y)
        if call in ("step", "host"):
            part["cp"], part["h"] = _thermo(m, t, y)
        if call in ("transport", "step", "host"):
            part["mu"], part["lam"], part["Dk"] = _transport(m, t, q, y)
        if call == "rop":
            part["q"] = torch.stack([x for _, x in _progress(m, t, q, y)])
        if call == "vjp":
            t, y = t.clone().requires_grad_(True), y.requires_grad_(True)
            with torch.enable_grad():
                part["gT"], part["gY"] = torch.autograd.grad((_wdot(m, t, q, y) * v[:, a:a + step]).sum(), (t, y))
        for k, x in part.items():
            got.setdefault(k, []).append(x.detach())
    return {k: torch.cat(x, dim=-1) for k, x in got.items()}
