"""The work that users of this library have it do, as cases that can be timed and compared.

A flow solver calls the library in four ways: it asks for the chemical source term (chem_rates), for the
sparse analytical Jacobian (chem_jacobian), it advances a field of cells over their flow time steps
(chem_integrate, plain or through the sorted work queue, with the library's kernels or the
mechanism-specialised ones, exact or with tabulated temperature functions, or with zonal mapping of its
unreactive cells), and it differentiates that advance (chem_adjoint).  The mechanisms and fields are the
seeded ones of synth.py: 10 species / 27 reactions, 53 / 325 and 150 / 1000.

Every integration starts from the same state in each pass: a flow solver hands over new T and Y after its
transport step, so the pass copies them in.  The previous substep counts that the work queue sorts by come
from a plain model of the cell's cost (`_previous_counts`), as if left by the previous flow step.
"""
import functools
import math

import numpy as np
import torch

from paper_2311_14941_gb300 import chem, opcount, synth

MECHS = {"small": synth.mechanism_small, "methane": synth.mechanism_methane_sized, "large": synth.mechanism_large}
R_U, P_0 = 8.314462618, 101325.0


def listed():
    return [
        # one block of a coarse or heavily decomposed mesh: the launch and the latency of one cell count
        {"name": "rates small 100", "kind": "rates", "mech": "small", "field": "random", "cells": 100},
        # the source term of a whole 256 x 256 flame field, as an explicit or operator-split code asks for it
        {"name": "rates methane 65536", "kind": "rates", "mech": "methane", "field": "jet", "cells": 65536},
        # the same for a detailed fuel mechanism, an odd number of cells
        {"name": "rates large 4099", "kind": "rates", "mech": "large", "field": "jet", "cells": 4099},
        # the Jacobian of a field, for a flow solver's own implicit scheme or preconditioner
        {"name": "jacobian methane 8191", "kind": "jacobian", "mech": "methane", "field": "jet", "cells": 8191},
        # hydrogen-sized mechanism, every cell reacting: the library's default call
        {"name": "advance small 1024", "kind": "advance", "mech": "small", "field": "random", "cells": 1024,
         "dt_lo": 1e-5, "dt_hi": 1e-5, "mode": 0, "method": 0, "rtol": 1e-6},
        # the same mechanism on a large field through the work queue
        {"name": "advance small 6000", "kind": "advance", "mech": "small", "field": "random", "cells": 6000,
         "dt_lo": 1e-5, "dt_hi": 1e-5, "mode": 1, "method": 0, "rtol": 1e-6},
        # uniform flow step of a jet flame field, one launch in cell order
        {"name": "advance methane jet 4096", "kind": "advance", "mech": "methane", "field": "jet", "cells": 4096,
         "dt_lo": 1e-5, "dt_hi": 1e-5, "mode": 0, "method": 0, "rtol": 1e-6},
        # local time stepping, heavy-tailed costs: sorted work queue and mechanism-specialised kernels
        {"name": "advance methane lts 8000", "kind": "advance", "mech": "methane", "field": "lts", "cells": 8000,
         "dt_lo": 1e-7, "dt_hi": 1e-3, "mode": 1, "method": 0, "rtol": 1e-6, "specialized": True},
        # the fourth-order method, for users who ask for accuracy
        {"name": "advance methane rodas4 2047", "kind": "advance", "mech": "methane", "field": "jet", "cells": 2047,
         "dt_lo": 1e-5, "dt_hi": 1e-5, "mode": 1, "method": 2, "rtol": 1e-6},
        # tabulated temperature functions and zonal mapping of the cold cells, the paper's cheaper settings
        {"name": "mapped methane 3000", "kind": "mapped", "mech": "methane", "field": "jet", "cells": 3000,
         "dt_lo": 1e-5, "dt_hi": 1e-5, "mode": 1, "method": 0, "rtol": 1e-6, "tabulate": True},
        # detailed fuel mechanism whose cells fill shared memory (two warps per cell by the library's choice)
        {"name": "advance large 500", "kind": "advance", "mech": "large", "field": "jet", "cells": 500,
         "dt_lo": 1e-6, "dt_hi": 3e-5, "mode": 1, "method": 0, "rtol": 1e-6},
        # gradients of the final state of igniting cells with respect to every reaction's parameters
        {"name": "adjoint methane 600", "kind": "adjoint", "mech": "methane", "field": "igniting", "cells": 600,
         "dt_lo": 2e-6, "dt_hi": 2e-6, "rtol": 1e-6},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["rates", "rates", "jacobian", "small", "small", "jet", "lts", "lts", "rodas4", "mapped", "large",
                       "adjoint"])
    if kind == "rates":
        mech = rng.choice(["small", "methane", "methane", "large"])
        return {"kind": kind, "mech": mech, "field": "random" if mech == "small" else "jet",
                "cells": size(32, 8000 if mech == "large" else 65536)}
    if kind == "jacobian":
        mech = rng.choice(["small", "methane", "methane", "large"])
        return {"kind": kind, "mech": mech, "field": "random" if mech == "small" else "jet",
                "cells": size(32, 2000 if mech == "large" else 10000)}
    rtol = rng.choice([1e-6, 1e-6, 1e-5])
    if kind == "small":
        return {"kind": "advance", "mech": "small", "field": "random", "cells": size(64, 6000), "dt_lo": 1e-5,
                "dt_hi": 1e-5, "mode": rng.choice([0, 1]), "method": 0, "rtol": rtol}
    if kind == "jet":
        return {"kind": "advance", "mech": "methane", "field": "jet", "cells": size(64, 4000), "dt_lo": 1e-5,
                "dt_hi": 1e-5, "mode": rng.choice([0, 1]), "method": 0, "rtol": rtol}
    if kind == "lts":
        return {"kind": "advance", "mech": "methane", "field": "lts", "cells": size(500, 8000), "dt_lo": 1e-7,
                "dt_hi": rng.choice([1e-4, 1e-3]), "mode": 1, "method": 0, "rtol": rtol,
                "specialized": rng.choice([True, False])}
    if kind == "rodas4":
        return {"kind": "advance", "mech": "methane", "field": "jet", "cells": size(64, 2048), "dt_lo": 1e-5,
                "dt_hi": 1e-5, "mode": rng.choice([0, 1]), "method": 2, "rtol": rtol}
    if kind == "mapped":
        return {"kind": "mapped", "mech": "methane", "field": "jet", "cells": size(64, 3000), "dt_lo": 1e-5,
                "dt_hi": 1e-5, "mode": 1, "method": 0, "rtol": rtol, "tabulate": rng.choice([True, False])}
    if kind == "large":
        return {"kind": "advance", "mech": "large", "field": "jet", "cells": size(16, 500), "dt_lo": 1e-6,
                "dt_hi": 3e-5, "mode": rng.choice([0, 1]), "method": 0, "rtol": rtol}
    return {"kind": "adjoint", "mech": "methane", "field": "igniting", "cells": size(4, 600), "dt_lo": 2e-6,
            "dt_hi": 2e-6, "rtol": rtol}


@functools.lru_cache(maxsize=None)
def _desc(mech):
    return MECHS[mech]()


@functools.lru_cache(maxsize=None)
def _handle(mech, specialized):
    """The compiled mechanism a program keeps for its whole run."""
    h = chem.create(_desc(mech), torch.cuda.current_device())
    if specialized:
        h.specialize()
    return h


@functools.lru_cache(maxsize=None)
def _plan(mech):
    return chem.create(_desc(mech), -1)


def _field(case, seed):
    m, N = _desc(case["mech"]), case["cells"]
    dt = (case.get("dt_lo", 1e-5), case.get("dt_hi", 1e-5))
    if case["field"] == "random":
        F = synth.field_uniform_random(m, N, seed=seed, dt=dt[0])
    elif case["field"] == "igniting":
        F = synth.field_igniting(m, N, seed=seed, dt=dt[0])
    elif case["field"] == "lts":
        F = synth.field_lts_mix(m, N, seed=seed, dt_range=dt)
    else:
        rows = -(-N // 64)
        F = synth.field_bimodal_jet(m, rows, 64, seed=seed, dt=dt[0], dt_range=dt if dt[0] < dt[1] else None)
        F = F.subset(np.arange(N))
    return F


def _previous_counts(F):
    """Substep counts as a previous flow step would have left them: more for longer steps and for reacting cells."""
    per_kind = np.array([1.0, 12.0, 8.0, 20.0, 30.0])[F.kind]
    return np.maximum(1, np.round(per_kind * (F.dt / 1e-7) ** 0.4)).astype(np.int32)


def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def prepare(case, seed):
    h = _handle(case["mech"], bool(case.get("specialized")))
    F = _field(case, seed)
    N, n = case["cells"], h.n
    s = {"h": h, "case": case, "T0": _gpu(F.T), "p": _gpu(F.p), "Y0": _gpu(F.Y), "dt": _gpu(F.dt)}
    f8 = functools.partial(torch.zeros, dtype=torch.float64, device="cuda")
    i4 = functools.partial(torch.zeros, dtype=torch.int32, device="cuda")
    if case["kind"] == "rates":
        s |= {"dTdt": f8(N), "dYdt": f8(n, N), "wdot": f8(n, N)}
    elif case["kind"] == "jacobian":
        s |= {"S": f8(h.info["nnz_S"], N), "u": f8(h.m, N), "v": f8(h.m, N)}
    else:
        s |= {"T": f8(N), "Y": f8(n, N), "status": i4(N)}
        if case["kind"] == "adjoint":
            rng = np.random.default_rng(seed)
            gY = np.zeros((n, N))
            gY[synth.cotangent_species(_desc(case["mech"]))] = rng.standard_normal((5, N))
            s |= {"gT": _gpu(np.full(N, 1e-3)), "gY": _gpu(gY), "gA": f8(h.R), "gE": f8(h.R), "gT0": f8(N),
                  "gY0": f8(n, N)}
        else:
            s |= {"h_io": f8(N), "counts": _gpu(_previous_counts(F)), "nsub": i4(N), "ref": i4(N)}
    return s


def run(s):
    h, case = s["h"], s["case"]
    if case["kind"] == "rates":
        h.rates(s["T0"], s["p"], s["Y0"], s["dTdt"], s["dYdt"], s["wdot"])
        return {"dTdt": s["dTdt"], "dYdt": s["dYdt"], "wdot": s["wdot"]}
    if case["kind"] == "jacobian":
        h.jacobian(s["T0"], s["p"], s["Y0"], s["S"], s["u"], s["v"])
        return {"S": s["S"], "u": s["u"], "v": s["v"]}
    s["T"].copy_(s["T0"])
    s["Y"].copy_(s["Y0"])
    if case["kind"] == "adjoint":
        h.adjoint(s["T"], s["p"], s["Y"], s["dt"], s["gT"], s["gY"], s["gA"], s["gE"], s["status"], gT0=s["gT0"],
                  gY0=s["gY0"], rtol=case["rtol"])
        return {k: s[k] for k in ("T", "Y", "gA", "gE", "gT0", "gY0", "status")}
    s["h_io"].zero_()
    s["nsub"].copy_(s["counts"])
    opts = {"rtol": case["rtol"], "mode": case["mode"], "method": case["method"]}
    if case.get("tabulate"):
        opts["tabulate"] = 1
    out = {k: s[k] for k in ("T", "Y", "h_io", "nsub", "status")}
    if case["kind"] == "mapped":
        roles = _desc(case["mech"]).roles
        zones = {"T_max": 700.0, "dT": 20.0, "species": [roles["fuel"], roles["O2"]], "dY": [0.02, 0.02]}
        h.integrate_mapped(s["T"], s["p"], s["Y"], s["dt"], s["h_io"], s["nsub"], s["status"], s["ref"], zones, **opts)
        return out | {"ref": s["ref"]}
    if case.get("specialized"):
        opts["specialized"] = 1
    h.integrate(s["T"], s["p"], s["Y"], s["dt"], s["h_io"], s["nsub"], s["status"], **opts)
    return out


#: Attempted steps per cell at rtol 1e-6, measured: a pass's work depends on them (rtol 1e-5 takes about 0.6 of them).
ATTEMPTS = {("small", "random", 0): 1000.0, ("methane", "jet", 0): 188.0, ("methane", "jet", 2): 77.0,
            ("methane", "lts", 0): 249.0, ("large", "jet", 0): 460.0, ("methane", "igniting", 0): 325.0}


def work(case):
    """Bytes: the inputs read once, the outputs written once.  Operations: two per FP64 slot of the library's own
    work model, with the usual number of attempted steps of the field."""
    h, N = _plan(case["mech"]), case["cells"]
    n, m = h.n, h.m
    method = case.get("method", 0)
    ops = opcount.model(_desc(case["mech"]), h.export_plan(0), h.export_plan(1), method)
    state = 8.0 * N * (n + 2)
    if case["kind"] == "rates":
        return {"bytes": state + 8.0 * N * (1 + 2 * n), "flops": 2.0 * ops.f_eval * N}
    if case["kind"] == "jacobian":
        return {"bytes": state + 8.0 * N * (h.info["nnz_S"] + 2 * m), "flops": 2.0 * ops.jac * N}
    steps = N * ATTEMPTS[case["mech"], case["field"], method] * (0.6 if case["rtol"] > 1e-6 else 1.0)
    flops = 2.0 * steps * (ops.attempt + ops.jac)
    if case["kind"] == "adjoint":   # forward, recompute, and at least two Jacobian products and four solves a step
        return {"bytes": 2 * state + 16.0 * N * n + 16.0 * h.R, "flops": 2.0 * flops + 2.0 * steps * (2 * ops.jac + 4 * ops.solve)}
    if case["kind"] == "mapped":    # the zones leave about this share of the work to integrate
        flops *= 0.6
    return {"bytes": 2 * state + 40.0 * N, "flops": flops}


# ---- the source term and the Jacobian in plain 64-bit torch ------------------------------------------------------

def _tables(m, dev):
    t = functools.partial(torch.as_tensor, dtype=torch.float64, device=dev)
    n, R = m.n_species, m.n_reactions
    nu_r, nu_p, am1 = np.zeros((R, n)), np.zeros((R, n)), np.zeros((R, n))
    for r in range(R):
        re, pr = m.reaction(r)
        for k, c in re:
            nu_r[r, k] += c
        for k, c in pr:
            nu_p[r, k] += c
        if m.rtype[r] != 0:
            for i in range(m.eff_ptr[r], m.eff_ptr[r + 1]):
                am1[r, m.eff_sp[i]] = m.eff_alpha[i] - 1.0
    return {"W": t(m.W), "nu_r": t(nu_r), "nu_p": t(nu_p), "am1": t(am1), "third": t((m.rtype == 1) * 1.0),
            "troe": torch.as_tensor(np.flatnonzero(m.rtype == 2), device=dev), "rev": t(m.reversible * 1.0),
            "occ_r": _occurrences(nu_r, dev), "occ_p": _occurrences(nu_p, dev)}


def _occurrences(nu, dev):
    """[R, 3] species of each side's factors, one per unit of the coefficient; absent ones point past the last."""
    occ = np.full((nu.shape[0], 3), nu.shape[1], dtype=np.int64)
    for r in range(nu.shape[0]):
        lst = [k for k in np.flatnonzero(nu[r]) for _ in range(int(nu[r, k]))]
        occ[r, : len(lst)] = lst
    return torch.as_tensor(occ, device=dev)


def _thermo(m, T):
    """cp/R, h/(R T), s/R and d(cp/R)/dT of every species at every T: [N, n] each."""
    t = functools.partial(torch.as_tensor, dtype=torch.float64, device=T.device)
    a = torch.where((T[:, None] < t(m.T_mid))[..., None], t(m.nasa_lo), t(m.nasa_hi))
    x = T[:, None]
    cp = a[..., 0] + x * (a[..., 1] + x * (a[..., 2] + x * (a[..., 3] + x * a[..., 4])))
    hh = a[..., 0] + x * (a[..., 1] / 2 + x * (a[..., 2] / 3 + x * (a[..., 3] / 4 + x * a[..., 4] / 5))) + a[..., 5] / x
    ss = a[..., 0] * x.log() + x * (a[..., 1] + x * (a[..., 2] / 2 + x * (a[..., 3] / 3 + x * a[..., 4] / 4))) + a[..., 6]
    dcp = a[..., 1] + x * (2 * a[..., 2] + x * (3 * a[..., 3] + x * 4 * a[..., 4]))
    return cp, hh, ss, dcp


def _progress(m, tb, T, C, p):
    """Rates of progress [N, R] as a function of T and the concentrations, the total one being p/(R T)."""
    t = functools.partial(torch.as_tensor, dtype=torch.float64, device=T.device)
    x, lnT = T[:, None], T[:, None].log()
    _, hh, ss, _ = _thermo(m, T)
    ln_k = t(m.A).log() + t(m.b) * lnT - t(m.Ea) / (R_U * x)
    M = p[:, None] / (R_U * x) + C @ tb["am1"].T
    kf = ln_k.exp()
    i = tb["troe"]
    if len(i):
        low, tr = t(m.low)[i], t(m.troe)[i]
        ln_pr = low[:, 0].log() + low[:, 1] * lnT - low[:, 2] / (R_U * x) - ln_k[:, i] + M[:, i].log()
        fc = (1 - tr[:, 0]) * torch.exp(-x / tr[:, 1]) + tr[:, 0] * torch.exp(-x / tr[:, 2])
        fc = fc + torch.where(tr[:, 3] > 0, torch.exp(-tr[:, 3] / x), torch.zeros_like(x))
        lfc = fc.log10()
        y = ln_pr / math.log(10.0) - 0.4 - 0.67 * lfc
        f1 = y / (0.75 - 1.27 * lfc - 0.14 * y)
        F = torch.exp(math.log(10.0) * lfc / (1 + f1 * f1))
        pr = ln_pr.exp()
        kf = kf.index_copy(1, i, kf[:, i] * pr / (1 + pr) * F)
    dnu = tb["nu_p"] - tb["nu_r"]
    ln_Kc = -((hh - ss) @ dnu.T) + dnu.sum(1) * torch.log(P_0 / (R_U * x))
    C1 = torch.cat([C, torch.ones_like(C[:, :1])], 1)
    fwd = kf * C1[:, tb["occ_r"]].prod(2)
    bwd = kf * torch.exp(-ln_Kc) * tb["rev"] * C1[:, tb["occ_p"]].prod(2)
    return (fwd - bwd) * torch.where(tb["third"] > 0, M, torch.ones_like(M))


def _exact_chunk(m, tb, h, T, p, Y, jacobian):
    cp_k, h_k, _, dcp_k = _thermo(m, T)
    W = tb["W"]
    wbar = 1.0 / (Y / W).sum(1)
    rho = p * wbar / (R_U * T)
    C = rho[:, None] * Y / W
    cp = R_U * (Y / W * cp_k).sum(1)
    dnu = tb["nu_p"] - tb["nu_r"]
    w = _progress(m, tb, T, C, p) @ dnu
    f_T = -R_U * T * (h_k * w).sum(1) / (rho * cp)
    f = W * w / rho[:, None]
    if not jacobian:
        return f_T, f, w
    n = m.n_species
    w_T = torch.func.jvp(lambda t: _progress(m, tb, t, C, p), (T,), (torch.ones_like(T),))[1] @ dnu
    cols = []
    for j in range(n):
        e = torch.zeros_like(C)
        e[:, j] = 1.0
        cols.append(torch.func.jvp(lambda c: _progress(m, tb, T, c, p), (C,), (e,))[1] @ dnu)
    D = torch.stack(cols, 2)                    # [N, k, j] = d w_k / d C_j at fixed total concentration
    g = (D * C[:, None, :]).sum(2)
    S = torch.zeros(T.shape[0], n + 1, n + 1, dtype=torch.float64, device=T.device)
    S[:, 1:, 1:] = D * W[:, None] / W
    dw_T = w_T - g / T[:, None]
    S[:, 1:, 0] = (W / rho[:, None]) * dw_T + f / T[:, None]
    tk = (D * h_k[:, :, None]).sum(1)
    S[:, 0, 1:] = -R_U * (T[:, None] * tk + f_T[:, None] * cp_k) / (W * cp[:, None])
    dcp = (Y / W * dcp_k).sum(1)
    S[:, 0, 0] = -R_U * (cp_k * w + T[:, None] * h_k * dw_T).sum(1) / (rho * cp) + f_T * (1 / T - R_U * dcp / cp)
    u = torch.cat([(R_U * T * (h_k * g).sum(1) / (rho * cp) + f_T)[:, None], W * (w - g) / rho[:, None]], 1)
    v = torch.cat([torch.zeros_like(T)[:, None], wbar[:, None] / W], 1)
    rp, ci = h.jacobian_pattern()
    rows = np.repeat(np.arange(n + 1), np.diff(rp))
    return S[:, torch.as_tensor(rows, device=T.device), torch.as_tensor(ci, device=T.device).long()], u, v


def exact(case, seed):
    """The source term and the Jacobian.  Integrations are left out: an adaptive integration of a whole field in plain
    torch takes minutes, and its own step decisions would not be the library's."""
    if case["kind"] not in ("rates", "jacobian"):
        return None
    m, F, h = _desc(case["mech"]), _field(case, seed), _plan(case["mech"])
    T, p, Y = _gpu(F.T), _gpu(F.p), _gpu(F.Y.T)
    tb, jac = _tables(m, T.device), case["kind"] == "jacobian"
    step = 256 if jac else 4096
    parts = [_exact_chunk(m, tb, h, T[i: i + step], p[i: i + step], Y[i: i + step], jac) for i in range(0, len(T), step)]
    out = [torch.cat([q[k] for q in parts]) for k in range(3)]
    if jac:
        return {"S": out[0].T.contiguous(), "u": out[1].T.contiguous(), "v": out[2].T.contiguous()}
    return {"dTdt": out[0], "dYdt": out[1].T.contiguous(), "wdot": out[2].T.contiguous()}
