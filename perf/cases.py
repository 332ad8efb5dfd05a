"""The calls whose speed is tracked, through the public entry points of
paper_1309_2710_gb300.kin, and what they should return.

A case names a mechanism (a key of MECHS), an entry point and its options:

  entry      "integrate"  kin.integrate on device tensors
             "batch"      kin.integrate_batch, several instances in one launch
             "host"       kin.integrate_host on pinned host tensors, and the wait for its result
             "rates"      kin.rates, the source term alone
  cells      cells of the call (of all instances together for "batch")
  dt         flow step [s]; the instances of a batch alternate dt and 10 dt
  precision  "fp64" or "mixed"
  energy     True: the constant-pressure energy equation is integrated too
  occupancy  "default" or "high", the register budget of the call
  instances  instances of a batch

Mechanisms, temperature, pressure and composition ranges, spectral-radius
estimators and tolerances are those of the workloads in synth.py. An
integration starts from the caller's transported state, which is copied over
the call's in/out buffers first, as in an operator-split flow solver.
"""
from __future__ import annotations

import dataclasses
import functools
import math

import numpy as np
import torch

from paper_1309_2710_gb300 import kin, synth

# mechanism -> workload of synth.py; the case's "energy" adds the thermochemistry
MECHS = {"h2": "h2_9sp_rkck", "h2co": "h2co_13sp_rkc", "ch4": "ch4_53sp_rkc_mixed",
         "c2h4": "c2h4_111sp_rkc_batched"}
# Mean f evaluations per cell at dt, and the exponent of their growth with dt,
# counted by a plain C integrator on 64 cells of each workload.
EVALS = {"h2": (66, 1e-7, 0.63), "h2co": (370, 1e-6, 0.45), "ch4": (691, 1e-6, 0.29),
         "c2h4": (3830, 1e-6, 0.53)}


def _case(name, mech, entry, cells, dt=0.0, precision="fp64", energy=False, occupancy="default",
          instances=1):
    return dict(name=name, mech=mech, entry=entry, cells=cells, dt=dt, precision=precision,
                energy=energy, occupancy=occupancy, instances=instances)


def listed():
    return [
        # one small block of a nonstiff flow domain: launch and latency of a single call
        _case("h2_rkck_64", "h2", "integrate", 64, 1e-7),
        # the nonstiff workload
        _case("h2_rkck_4096", "h2", "integrate", 4096, 1e-7),
        # a ragged subdomain of a moderately stiff flow, too small to fill the GPU
        _case("h2co_rkc_1000", "h2co", "integrate", 1000, 1e-6),
        # a mid-sized subdomain (one lane per cell, table-driven f)
        _case("h2co_rkc_30011", "h2co", "integrate", 30011, 1e-6),
        # the headline workload: a whole flow domain of the CO/H2 mechanism
        _case("h2co_rkc_262144", "h2co", "integrate", 262144, 1e-6),
        # the same chemistry with the energy equation
        _case("h2co_energy_20000", "h2co", "integrate", 20000, 1e-6, energy=True),
        # a subdomain whose state lives in host memory: copies in and out counted
        _case("h2co_host_65536", "h2co", "host", 65536, 1e-6),
        # the smallest serving request of the methane mechanism, mixed precision
        _case("ch4_mixed_1024", "ch4", "integrate", 1024, 1e-6, "mixed"),
        # the largest serving request, at the register budget its workload uses
        _case("ch4_mixed_65536", "ch4", "integrate", 65536, 1e-6, "mixed", occupancy="high"),
        # the methane mechanism in full FP64
        _case("ch4_fp64_4096", "ch4", "integrate", 4096, 1e-6),
        # several uneven subdomains of the ethylene mechanism in one launch
        _case("c2h4_batch_2000", "c2h4", "batch", 2000, 1e-7, instances=16),
        # the source term alone, for a caller with its own integrator
        _case("rates_ch4_50000", "ch4", "rates", 50000),
    ]


def draw(rng):
    log = lambda lo, hi: math.exp(rng.uniform(math.log(lo), math.log(hi)))
    kind = rng.choice(["h2", "h2co", "h2co", "h2co_energy", "host", "ch4_mixed", "ch4_mixed", "ch4_fp64",
                       "ch4_energy", "c2h4", "rates"])
    if kind == "h2":
        c = _case("", "h2", "integrate", int(log(33, 60000)), log(3e-8, 3e-7))
    elif kind == "h2co":
        c = _case("", "h2co", "integrate", int(log(97, 200000)), log(1e-7, 1e-6),
                  occupancy=rng.choice(["default", "high"]))
    elif kind == "h2co_energy":
        c = _case("", "h2co", "integrate", int(log(97, 60000)), log(1e-7, 1e-6), energy=True)
    elif kind == "host":
        c = _case("", "h2co", "host", int(log(1024, 100000)), log(1e-7, 1e-6))
    elif kind == "ch4_mixed":
        c = _case("", "ch4", "integrate", int(log(65, 60000)), log(1e-7, 1e-6), "mixed",
                  occupancy=rng.choice(["default", "high"]))
    elif kind == "ch4_fp64":
        c = _case("", "ch4", "integrate", int(log(65, 6000)), log(1e-7, 1e-6))
    elif kind == "ch4_energy":
        c = _case("", "ch4", "integrate", int(log(65, 12000)), log(1e-7, 1e-6), "mixed", energy=True)
    elif kind == "c2h4":
        n = rng.randint(1, 32)
        c = _case("", "c2h4", "batch", max(n, int(log(100, 3000))), log(3e-8, 1e-7), instances=n)
    else:
        m = rng.choice(["h2", "h2co", "ch4", "c2h4"])
        top = {"h2": 800000, "h2co": 500000, "ch4": 60000, "c2h4": 20000}[m]
        c = _case("", m, "rates", int(log(100, top)), precision=rng.choice(["fp64", "mixed"]))
    del c["name"]
    return c


# ------------------------------------------------------------- a call's state
@functools.lru_cache(maxsize=None)
def _tables(mech, energy):
    return synth.workload_mechanism(MECHS[mech] + ("_energy" if energy else ""))


@functools.lru_cache(maxsize=None)
def _mechanism(mech, energy):
    """The device-resident mechanism, which a program creates once."""
    return kin.Mechanism(_tables(mech, energy))


def _states(case, seed):
    return synth.workload_states(MECHS[case["mech"]], _tables(case["mech"], case["energy"]),
                                 cells=case["cells"], seed_offset=10000 + seed)


def _parts(case):
    """(first cell, cells, dt) of each instance; sizes log-uniform over a factor of 64."""
    n, cells = case["instances"], case["cells"]
    w = np.exp(np.random.default_rng(n).uniform(0.0, math.log(64.0), n))
    sizes = 1 + np.floor(w / w.sum() * (cells - n)).astype(int)
    sizes[-1] += cells - sizes.sum()
    first = np.concatenate([[0], np.cumsum(sizes)])
    return [(int(first[i]), int(sizes[i]), case["dt"] * (10.0 if i % 2 else 1.0)) for i in range(n)]


def _options(case):
    w = synth.WORKLOADS[MECHS[case["mech"]]]
    sigma = kin.SIGMA_POWER if case["energy"] else w["sigma"]
    return dict(method=w["method"], precision=kin.MIXED if case["precision"] == "mixed" else kin.FP64,
                sigma=sigma, energy=int(case["energy"]),
                occupancy=kin.OCC_HIGH if case["occupancy"] == "high" else kin.OCC_DEFAULT)


def prepare(case, seed):
    T, p, Y = (torch.as_tensor(a) for a in _states(case, seed))
    mech = _mechanism(case["mech"], case["energy"])
    s = dict(case=case, mech=mech, opts=_options(case))
    w = synth.WORKLOADS[MECHS[case["mech"]]]
    s["rtol"], s["atol"] = w["rtol"], w["atol"]
    if case["entry"] == "host":
        s["T"], s["p"], s["Y0"] = T.pin_memory(), p.pin_memory(), Y.pin_memory()
        s["Y"] = torch.empty_like(Y).pin_memory()
        s["status"] = torch.empty(case["cells"], dtype=torch.uint8).pin_memory()
        s["buffer"] = kin.host_buffer(mech, case["cells"], **s["opts"])
        return s
    s["T0"], s["p"], s["Y0"] = T.cuda(), p.cuda(), Y.cuda()
    if case["entry"] == "rates":
        s["out"] = torch.empty_like(s["Y0"])
        s["workspace"] = mech.workspace(kin.RKC, s["opts"]["precision"], case["cells"],
                                        layout=kin.LAYOUT_LANE)
        return s
    o = s["opts"]
    s["workspace"] = mech.workspace(o["method"], o["precision"], case["cells"], occupancy=o["occupancy"],
                                    sigma=o["sigma"], energy=o["energy"])
    s["T"] = torch.empty_like(s["T0"]) if case["energy"] else s["T0"]
    s["status"] = torch.empty(case["cells"], dtype=torch.uint8, device="cuda")
    if case["entry"] == "batch":  # each instance owns its species-major block
        s["inst"] = []
        for a, n, dt in _parts(case):
            cut = slice(a, a + n)
            s["inst"].append((s["Y0"][:, cut].contiguous(),
                              kin.Cells(s["T0"][cut].clone(), s["p"][cut].clone(),
                                        torch.empty(Y.shape[0], n, dtype=torch.float64, device="cuda"),
                                        dt, s["rtol"], s["atol"], s["status"][cut])))
        return s
    s["Y"] = torch.empty_like(s["Y0"])
    return s


def run(s):
    entry, dt = s["case"]["entry"], s["case"]["dt"]
    if entry == "rates":
        kin.rates(s["mech"], s["T0"], s["p"], s["Y0"], s["opts"]["precision"], out=s["out"],
                  workspace=s["workspace"])
        return {"dYdt": s["out"]}
    if entry == "host":
        s["Y"].copy_(s["Y0"])
        kin.integrate_host(s["mech"], s["T"], s["p"], s["Y"], dt, s["rtol"], s["atol"],
                           status=s["status"], buffer=s["buffer"], **s["opts"])
        torch.cuda.current_stream().synchronize()  # the caller reads the host result
        return {"Y": s["Y"], "status": s["status"]}
    if entry == "batch":
        for Y0, c in s["inst"]:
            c.Y.copy_(Y0)
        kin.integrate_batch(s["mech"], [c for _, c in s["inst"]], workspace=s["workspace"], **s["opts"])
        return {"Y": [c.Y for _, c in s["inst"]], "status": s["status"]}
    s["Y"].copy_(s["Y0"])
    if s["case"]["energy"]:
        s["T"].copy_(s["T0"])
    kin.integrate(s["mech"], s["T"], s["p"], s["Y"], dt, s["rtol"], s["atol"], status=s["status"],
                  workspace=s["workspace"], **s["opts"])
    out = {"Y": s["Y"], "status": s["status"]}
    if s["case"]["energy"]:
        out["T"] = s["T"]
    return out


def work(case):
    m = _tables(case["mech"], case["energy"])
    nS, nR, n = m.n_species, m.n_reactions, case["cells"]
    rows, fall = m.n_third_body_rows, int(np.count_nonzero(m.rtype == synth.FALLOFF))
    # one evaluation of f, an FMA as two: mixture and concentrations, rates of
    # progress, third-body sums, falloff, four net coefficients a reaction
    f = 4 * nS + 2 * nR + 2 * nS * rows + 6 * fall + 8 * nR + 2 * nS
    if case["entry"] == "rates":
        return {"bytes": 8 * n * (2 + 2 * nS), "flops": n * (f + 6 * nR)}
    at, dt0, power = EVALS[case["mech"]]
    per = n / len(_parts(case)) if case["entry"] == "batch" else n
    dts = [dt for _, _, dt in _parts(case)] if case["entry"] == "batch" else [case["dt"]]
    evals = sum(per * at * (dt / dt0) ** power for dt in dts)
    t = 8 if case["energy"] else 0
    return {"bytes": n * (16 + 16 * nS + 1 + t), "flops": evals * (f + 10 * nS)}


# ------------------------------------------------------- the results in FP64
class _Source:
    """dY/dt (and dT/dt) of a set of cells in plain torch, FP64."""

    def __init__(self, m, T, p, energy):
        t = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float64), device="cuda")
        self.m, self.energy, self.T, self.p = m, energy, T, p
        self.W, self.iW = t(m.W)[:, None], t(1.0 / m.W)[:, None]
        self.lnA, self.beta = t(m.lnA)[:, None], t(m.beta)[:, None]
        self.EaR = t(m.Ea / synth.R_GAS)[:, None]
        self.fo = torch.as_tensor(np.flatnonzero(m.rtype == synth.FALLOFF), device="cuda")
        self.tb = torch.as_tensor(np.flatnonzero(m.rtype == synth.THIRD_BODY), device="cuda")
        non = np.flatnonzero(m.rtype != synth.PLAIN)  # efficiency rows, in reaction order
        eff = np.asarray(m.eff).reshape(len(non), m.n_species)
        self.eff_tb = t(eff[m.rtype[non] == synth.THIRD_BODY])
        self.eff_fo = t(eff[m.rtype[non] == synth.FALLOFF])
        low = m.rtype == synth.FALLOFF
        self.lnA0, self.beta0 = t(m.lnA0[low])[:, None], t(m.beta0[low])[:, None]
        self.Ea0R = t(m.Ea0[low] / synth.R_GAS)[:, None]
        nu = np.zeros((m.n_species, m.n_reactions))
        for j in range(m.n_reactions):
            for k in range(2):
                if m.prod[j, k] >= 0:
                    nu[m.prod[j, k], j] += 1.0
                if m.reac[j, k] >= 0:
                    nu[m.reac[j, k], j] -= 1.0
        self.nu = t(nu)
        one = m.n_species  # an empty slot reads a concentration of 1
        self.r = [torch.as_tensor(np.where(m.reac[:, k] >= 0, m.reac[:, k], one), device="cuda")
                  for k in range(2)]
        if energy:
            self.cp, self.Hf = t(m.cp)[:, None], t(m.Hf)[:, None]
        else:
            self.k, self.k0 = self._constants(T)

    def _constants(self, T):
        a = self.lnA + self.beta * torch.log(T) - self.EaR / T
        a0 = self.lnA0 + self.beta0 * torch.log(T) - self.Ea0R / T
        return torch.exp(a), torch.exp(a0 - a[self.fo])  # k, k0/kinf

    def __call__(self, y, cells):
        nS = self.m.n_species
        Y, p = y[:nS], self.p[cells]
        T = y[nS] if self.energy else self.T[cells]
        k, k0 = self._constants(T) if self.energy else (self.k[:, cells], self.k0[:, cells])
        rho = p * 1e-6 / (synth.R_GAS * T * (Y * self.iW).sum(0))
        C = torch.cat([rho * Y * self.iW, torch.ones_like(rho)[None]])
        q = k * C[self.r[0]] * C[self.r[1]]
        if len(self.tb):
            q[self.tb] *= self.eff_tb @ C[:nS]
        if len(self.fo):
            pr = k0 * (self.eff_fo @ C[:nS])
            q[self.fo] *= pr / (1.0 + pr)
        om = self.nu @ q
        d = om * (self.W / rho)
        if not self.energy:
            return d
        h = ((self.Hf + self.cp * (T - 298.15)) * om).sum(0)
        cp = (Y * self.cp * self.iW).sum(0)
        return torch.cat([d, (-h / (rho * cp))[None]])


def _rkck(f, y, dt, rtol, atol):
    """Cash-Karp 5(4) of every cell over dt [cells]."""
    b = [[], [1 / 5], [3 / 40, 9 / 40], [3 / 10, -9 / 10, 6 / 5], [-11 / 54, 5 / 2, -70 / 27, 35 / 27],
         [1631 / 55296, 175 / 512, 575 / 13824, 44275 / 110592, 253 / 4096]]
    c5 = [37 / 378, 0, 250 / 621, 125 / 594, 0, 512 / 1771]
    c4 = [2825 / 27648, 0, 18575 / 48384, 13525 / 55296, 277 / 14336, 1 / 4]
    t, h, left = torch.zeros_like(dt), dt.clone(), torch.arange(y.shape[1], device=y.device)
    f0 = f(y, left)
    while len(left):
        rest = dt[left] - t[left]
        last = h[left] >= rest
        hh = torch.where(last, rest, h[left])
        yl = y[:, left]
        k = [f0[:, left]]
        for st in range(1, 6):
            k.append(f(yl + hh * sum(w * ki for w, ki in zip(b[st], k)), left))
        y5 = yl + hh * sum(w * ki for w, ki in zip(c5, k))
        e = hh * sum((u - v) * ki for u, v, ki in zip(c5, c4, k))
        err = (e.abs() / (rtol * (yl.abs() + (hh * k[0]).abs()) + atol)).amax(0)
        ok = err <= 1.0
        h[left] = torch.where(ok, torch.minimum(0.9 * hh * err ** -0.2, 5.0 * hh),
                              torch.maximum(0.9 * hh * err ** -0.25, 0.1 * hh))
        acc = left[ok]
        y[:, acc] = y5[:, ok]
        t[acc] += hh[ok]
        go = left[ok & ~last]
        if len(go):
            f0[:, go] = f(y[:, go], go)
        left = left[~(ok & last)]
    return y


@functools.lru_cache(maxsize=None)
def _rkc_table():
    """mu, nu, mu~, gamma~ of every stage j of every stage count s <= 250."""
    tab = np.zeros((251, 251, 4))
    for s in range(2, 251):
        w0 = 1.0 + (2.0 / 13.0) / s ** 2
        T, d, dd = [1.0, w0], [0.0, 1.0], [0.0, 0.0]
        for j in range(2, s + 1):
            T.append(2 * w0 * T[-1] - T[-2])
            d.append(2 * T[j - 1] + 2 * w0 * d[-1] - d[-2])
            dd.append(4 * d[j - 1] + 2 * w0 * dd[-1] - dd[-2])
        w1 = d[s] / dd[s]
        bb = [0.0, 0.0] + [dd[j] / d[j] ** 2 for j in range(2, s + 1)]
        bb[0] = bb[1] = bb[2]
        tab[s, 1, 2] = bb[1] * w1
        for j in range(2, s + 1):
            mt = 2 * bb[j] * w1 / bb[j - 1]
            tab[s, j] = (2 * bb[j] * w0 / bb[j - 1], -bb[j] / bb[j - 2], mt, -(1 - bb[j - 1] * T[j - 1]) * mt)
    return torch.as_tensor(tab, device="cuda")


@dataclasses.dataclass
class _Norm:
    rtol: float
    atol: float

    def __call__(self, d, a, b):
        return torch.sqrt(((d / (self.atol + self.rtol * torch.maximum(a.abs(), b.abs()))) ** 2).mean(0))


def _radius(f, y, f0, v, cells, atol, power):
    """Spectral radius of the Jacobian at y and the power method's last direction."""
    u = math.sqrt(2.0 ** -52)
    if not power:
        rows = torch.zeros_like(y)
        for k in range(y.shape[0]):
            eps = u * y[k].abs().clamp(min=atol)
            x = y.clone()
            x[k] += eps
            rows += ((f(x, cells) - f0) / eps).abs()
        return rows.amax(0), v
    size = u * y.norm(dim=0)
    v = v * (size / v.norm(dim=0))
    sig, going = torch.zeros_like(size), torch.ones_like(size, dtype=torch.bool)
    for k in range(1, 21):
        g = going.nonzero()[:, 0]
        if not len(g):
            break
        w = f(y[:, g] + v[:, g], cells[g]) - f0[:, g]
        wn = w.norm(dim=0)
        new = wn / size[g]
        v[:, g] = w * (size[g] / wn)
        if k >= 2:
            going[g] = (new - sig[g]).abs() > 0.01 * new
        sig[g] = new
    return 1.2 * sig, v


def _rkc(f, y, dt, rtol, atol, power):
    """Runge-Kutta-Chebyshev of every cell over dt [cells]."""
    norm, tab = _Norm(rtol, atol), _rkc_table()
    left = torch.arange(y.shape[1], device=y.device)
    f0 = f(y, left)
    sig, ev = _radius(f, y, f0, f0.clone(), left, atol, power)
    h = torch.minimum(1.0 / sig, dt)
    e0 = norm(h * (f(y + h * f0, left) - f0), y, y)
    h = torch.minimum(0.1 * h / torch.sqrt(e0), dt)
    t, hprev, eprev = torch.zeros_like(dt), torch.ones_like(dt), torch.zeros_like(dt)
    since = torch.zeros_like(left)
    here, rejected = torch.ones_like(dt, dtype=torch.bool), torch.zeros_like(dt, dtype=torch.bool)
    while len(left):
        stale = left[(since[left] >= 25) | (rejected[left] & ~here[left])]
        if len(stale):
            sig[stale], ev[:, stale] = _radius(f, y[:, stale], f0[:, stale], ev[:, stale], stale, atol, power)
            since[stale], here[stale] = 0, True
        rest = dt[left] - t[left]
        last = h[left] >= rest
        hh = torch.where(last, rest, h[left])
        s = torch.floor(1.0 + torch.sqrt(1.0 + 1.54 * hh * sig[left]))
        cap = s > 250
        hh = torch.where(cap, (249.0 ** 2 - 1.0) / (1.54 * sig[left]), hh)
        last &= ~cap
        s = s.clamp(2, 250).long()
        yl, fl = y[:, left], f0[:, left]
        w2, w1 = yl.clone(), yl + tab[s, 1, 2] * hh * fl
        for j in range(2, int(s.max()) + 1):
            g = (s >= j).nonzero()[:, 0]
            mu, nu, mt, gt = tab[s[g], j].unbind(1)
            new = ((1.0 - mu - nu) * yl[:, g] + mu * w1[:, g] + nu * w2[:, g]
                   + mt * hh[g] * f(w1[:, g], left[g]) + gt * hh[g] * fl[:, g])
            w2[:, g] = w1[:, g]
            w1[:, g] = new
        fs = f(w1, left)
        err = norm(0.8 * (yl - w1) + 0.4 * hh * (fl + fs), yl, w1)
        ok = err <= 1.0
        first = (eprev[left] == 0.0) | rejected[left]
        fac = torch.where(first | ~ok, 0.8 * err ** (-1 / 3),
                          0.8 * hh / hprev[left] * eprev[left] ** (1 / 3) * err ** (-2 / 3))
        fac = torch.where(ok, fac.clamp(0.1, 10.0), fac.clamp(min=0.1))
        h[left] = fac * hh
        acc = left[ok]
        y[:, acc], f0[:, acc] = w1[:, ok], fs[:, ok]
        t[acc] += hh[ok]
        hprev[acc], eprev[acc], here[acc] = hh[ok], err[ok], False
        since[acc] += 1
        rejected[left] = ~ok
        left = left[~(ok & last)]
    return y


def exact(case, seed):
    m = _tables(case["mech"], case["energy"])
    if case["entry"] == "batch" and case["cells"] * case["dt"] > 400 * 1e-7:
        return None  # thousands of steps of the stiffest cells: too long in plain torch
    T, p, Y = (torch.as_tensor(a).cuda() for a in _states(case, seed))
    f = _Source(m, T, p, case["energy"])
    cells = torch.arange(case["cells"], device="cuda")
    if case["entry"] == "rates":
        return {"dYdt": torch.cat([f(Y[:, c], c) for c in cells.split(20000)], 1)}
    o, w = _options(case), synth.WORKLOADS[MECHS[case["mech"]]]
    dt = torch.full_like(T, case["dt"])
    if case["entry"] == "batch":
        for a, n, d in _parts(case):
            dt[a:a + n] = d
    y = torch.cat([Y, T[None]]) if case["energy"] else Y
    step = _rkck if o["method"] == kin.RKCK else functools.partial(_rkc, power=o["sigma"] == kin.SIGMA_POWER)
    y = step(f, y, dt, w["rtol"], w["atol"])
    nS = m.n_species
    if case["entry"] == "batch":
        return {"Y": [y[:, a:a + n].contiguous() for a, n, _ in _parts(case)], "status": None}
    out = {"Y": y[:nS].contiguous(), "status": None}
    if case["energy"]:
        out["T"] = y[nS]
    return out
