"""The work a user of this library has it do: zone burns, their gradients and
the predicted costs, through the package's public calls, on the networks of
``gen`` and over the sizes between one hydro tile and a full grid.

Each case is a dict of plain values.  ``kind`` names the call:

* ``burn``: ``burn`` with its default launch, as the README calls it;
* ``graph``: a captured ``BurnGraph`` replayed (a time-stepping loop);
* ``host``: ``burn_host`` from and to pinned host arrays;
* ``coop``: ``burn`` with the cooperative launch the autotuner picks for
  large networks;
* ``autograd``: ``Burn.apply`` and the backward pass of a scalar loss;
* ``adjoint``: a taped burn and ``adjoint`` with several cotangent sets;
* ``multi``: ``burn_multi``, the same zones burned with several networks;
* ``costs``: ``zone_costs``, before zones are dealt out to ranks.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import gen
import paper_2312_02836_gb300 as nb

DEV = "cuda"

CHAINS = ("chain13", "chain13_literal", "chain13_heat", "chain13_heat_ap", "chain13_heat_scr",
          "chain13_heat_tab")

# Mean algorithmic flops of one zone's burn to the workload's end time
# (net128_heat: to a tenth of it), from its event counters (adds and multiplies; exp, log and divisions apart)
FLOPS = {"chain13": 6.3e5, "chain13_literal": 7.5e5, "chain13_heat": 1.55e6,
         "chain13_heat_ap": 2.1e6, "chain13_heat_scr": 1.6e6, "chain13_heat_tab": 1.6e6,
         "net48": 5.1e6, "net48_adjoint": 5.1e6, "net128_heat": 3.0e7}

# net128_heat zones here keep to the paper's temperatures and to densities up
# to 1e6: beyond, a fifth of them run away to T9 of 13-17, where rounding
# decides their outcome
LIMITS = {"net128_heat": dict(T9=(0.3, 3.0), rho=(1e4, 1e6))}


def listed():
    return [
        # one small hydro tile (4 x 4 x 4 zones), the smallest call of a
        # time step: the latency of the longest zone
        dict(name="tile_64", kind="burn", workload="chain13_heat", Z=64),
        # the fixed-temperature chain at its configured size
        dict(name="chain_4096", kind="burn", workload="chain13", Z=4096),
        # the self-heating chain at its configured size: a full grid per call
        dict(name="heat_65536", kind="burn", workload="chain13_heat", Z=65536),
        # an operator-split step of a screened network: every zone its own
        # end time, plasma parameter and set of rate multipliers (a
        # sensitivity ensemble), an odd number of zones
        dict(name="split_scr_12345", kind="burn", workload="chain13_heat_scr", Z=12345,
             split=True, mult="zone"),
        # a time-stepping loop on one 16^3 tile, replaying its captured graph
        # (tabulated weak rates)
        dict(name="graph_tab_4096", kind="graph", workload="chain13_heat_tab", Z=4096),
        # a host code's own arrays in and out, effective (alpha,p)(p,gamma)
        # rates with shared multipliers
        dict(name="host_ap_10007", kind="host", workload="chain13_heat_ap", Z=10007,
             mult="shared"),
        # the 48-species network in the launch the autotuner picks for it
        dict(name="net48_16384", kind="coop", workload="net48", Z=16384, threads_per_block=128,
             blocks_per_sm=3, warps_per_zone=0),
        # the 128-species network, two warps per zone as the autotuner picks,
        # one tenth of its configured time (a hydro step)
        dict(name="net128_304", kind="coop", workload="net128_heat", Z=304, t_end=1e-2,
             threads_per_block=0, blocks_per_sm=0, warps_per_zone=2),
        # gradients of a scalar loss in a training loop, through autograd
        dict(name="autograd_256", kind="autograd", workload="chain13_heat", Z=256),
        # the sensitivity study: energy and the five largest abundances of
        # every zone by all 180 rates
        dict(name="adjoint48_1024", kind="adjoint", workload="net48_adjoint", Z=1024, K=6,
             max_steps=4000),
        # the paper's comparison: the same zones with three networks
        dict(name="multi_3x2048", kind="multi",
             workload="chain13_heat,chain13_heat_ap,chain13_literal", Z=2048),
        # predicted costs of a full grid, before it is dealt out to ranks
        dict(name="costs_262144", kind="costs", workload="net48", Z=262144),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["burn", "burn", "burn", "graph", "host", "coop", "coop", "autograd",
                       "adjoint", "multi", "costs"])
    if kind in ("burn", "graph", "host"):
        c = dict(kind=kind, workload=rng.choice(CHAINS), Z=_log_int(rng, 1, 40000))
        if kind == "burn" and rng.random() < 0.5:
            c["split"] = True
        if rng.random() < 0.5:
            c["mult"] = rng.choice(["shared", "zone"])
        return c
    if kind == "coop":
        if rng.random() < 0.7:
            tpb, bps, wpz = rng.choice([(128, 3, 0), (128, 3, 0), (0, 0, 0), (0, 0, 2)])
            return dict(kind=kind, workload="net48", Z=_log_int(rng, 16, 12000),
                        threads_per_block=tpb, blocks_per_sm=bps, warps_per_zone=wpz)
        return dict(kind=kind, workload="net128_heat", Z=_log_int(rng, 8, 300), t_end=1e-2,
                    threads_per_block=0, blocks_per_sm=0, warps_per_zone=rng.choice([2, 2, 4]))
    if kind == "autograd":
        return dict(kind=kind, workload=rng.choice(["chain13", "chain13_heat"]),
                    Z=_log_int(rng, 16, 1000))
    if kind == "adjoint":
        return dict(kind=kind, workload="net48_adjoint", Z=_log_int(rng, 32, 1500),
                    K=rng.choice([1, 2, 6]), max_steps=4000)
    if kind == "multi":
        return dict(kind=kind, workload=",".join(rng.sample(CHAINS, rng.choice([2, 3]))),
                    Z=_log_int(rng, 64, 4000))
    return dict(kind=kind, workload=rng.choice(["net48", "chain13_heat"]),
                Z=_log_int(rng, 1000, 262144))


# ---------------------------------------------------------------- inputs

@functools.lru_cache(maxsize=None)
def _spec(workload):
    return gen.network(workload)


@functools.lru_cache(maxsize=None)
def _net(workload):
    """One compiled network per workload, kept as a program keeps it."""
    return nb.Network(_spec(workload))


def _inputs(case, seed):
    """Host arrays of a case: its zones, drawn from the workload's own ranges
    (log-uniform T9 and density), and what its options add."""
    names = case["workload"].split(",")
    cfg, spec, Z = gen.CONFIGS[names[0]], _spec(names[0]), case["Z"]
    rng = np.random.default_rng([seed, Z])
    lim = dict(T9=cfg["T9"], rho=cfg["rho"]) | LIMITS.get(names[0], {})
    log_u = lambda lo, hi: np.exp(rng.uniform(np.log(lo), np.log(hi), Z))
    a = dict(T9=log_u(*lim["T9"]), rho=log_u(*lim["rho"]), Y=np.zeros((Z, spec.N)))
    if cfg["kind"] == "chain":
        a["Y"][:, 0] = 0.25
    else:
        X = rng.dirichlet([0.3] * 4, Z)
        a["Y"][:, :4] = X / X.sum(1, keepdims=True) / np.arange(1, 5)
    a["zeta"] = None
    if any(gen.CONFIGS[n].get("zeta") for n in names):
        a["zeta"] = rng.uniform(1.0, 2.0, Z)
    a["t_end"] = case.get("t_end", cfg["t_end"])
    if case.get("split"):
        a["t_end"] = cfg["t_end"] * np.exp(rng.uniform(np.log(0.1), 0.0, Z))
    mult = case.get("mult")
    a["lnm"] = (None if mult is None else rng.normal(0.0, 0.1, spec.R) if mult == "shared"
                else rng.normal(0.0, 0.1, (Z, spec.R)))
    if case["kind"] == "autograd":
        a["lnm"] = np.zeros(spec.R)
        a["wY"] = rng.uniform(0.0, 1.0, (Z, spec.N))
    if case["kind"] == "adjoint":
        a["gY"] = rng.uniform(0.0, 1.0, (case["K"], Z, spec.N))
        a["gE"] = rng.uniform(0.0, 1.0, (case["K"], Z))
    return a


def prepare(case, seed):
    names = case["workload"].split(",")
    cfg = gen.CONFIGS[names[0]]
    a = _inputs(case, seed)
    s = dict(case=case, nets=[_net(n) for n in names], rtol=cfg["rtol"], atol=cfg["atol"])
    if case["kind"] == "host":
        for k in ("Y", "T9", "rho"):
            a[k] = torch.from_numpy(a[k]).pin_memory().numpy()
        s.update(a)
        if a["zeta"] is not None:
            s["zeta"] = torch.from_numpy(a["zeta"]).to(DEV)
        pin = lambda *sh, dt=torch.float64: torch.empty(sh, dtype=dt, pin_memory=True).numpy()
        Z = case["Z"]
        s["out"] = dict(Y=pin(Z, a["Y"].shape[1]), T9=pin(Z), E=pin(Z),
                        counters=pin(Z, nb.NCOUNT, dt=torch.int32), status=pin(Z, dt=torch.int32))
        return s
    s.update({k: torch.from_numpy(v).to(DEV) if isinstance(v, np.ndarray) else v
              for k, v in a.items()})
    if case["kind"] == "graph":
        s["graph"] = nb.BurnGraph(s["nets"][0], s["Y"], s["T9"], s["rho"], s["t_end"], s["rtol"],
                                  s["atol"], s["lnm"], zeta=s["zeta"])
    if case["kind"] == "autograd":
        for k in ("Y", "T9", "lnm"):
            s[k].requires_grad_()
    if case["kind"] == "adjoint":
        s["tape"] = nb.Tape(s["nets"][0], case["Z"], case["max_steps"])
    return s


# ---------------------------------------------------------------- one pass

def run(s):
    case, net = s["case"], s["nets"][0]
    kind = case["kind"]
    tol = (s["t_end"], s["rtol"], s["atol"])
    if kind == "burn":
        return nb.burn(net, s["Y"], s["T9"], s["rho"], *tol, s["lnm"], zeta=s["zeta"])._asdict()
    if kind == "graph":
        return s["graph"].replay()._asdict()
    if kind == "host":
        return nb.burn_host(net, s["Y"], s["T9"], s["rho"], *tol, s["lnm"], zeta=s["zeta"],
                            out=s["out"])
    if kind == "coop":
        return nb.burn(net, s["Y"], s["T9"], s["rho"], *tol, kernel="coop",
                       threads_per_block=case["threads_per_block"],
                       blocks_per_sm=case["blocks_per_sm"],
                       warps_per_zone=case["warps_per_zone"])._asdict()
    if kind == "autograd":
        Y, T9, E, counters, status = nb.Burn.apply(s["Y"], s["T9"], s["rho"], s["lnm"], net, *tol)
        loss = (s["wY"] * Y).sum() + (0.0 if not net.has_energy else E.sum())
        gY, gT, gl = torch.autograd.grad(loss, (s["Y"], s["T9"], s["lnm"]))
        return dict(Y=Y.detach(), T9=T9.detach(), E=E.detach(), counters=counters, status=status,
                    gY=gY, gT9=gT, glnm=gl)
    if kind == "adjoint":
        out = nb.burn(net, s["Y"], s["T9"], s["rho"], *tol, kernel="coop", tape=s["tape"])
        dl, dY0, dT0 = nb.adjoint(net, s["tape"], s["gY"], s["gE"])
        return dict(out._asdict(), dl=dl, dY0=dY0, dT0=dT0)
    if kind == "multi":
        sets = [dict(net=m, Y0=s["Y"], T9=s["T9"], rho=s["rho"],
                     **({} if s["zeta"] is None else {"zeta": s["zeta"]})) for m in s["nets"]]
        return [o._asdict() for o in nb.burn_multi(sets, *tol)]
    return nb.zone_costs(net, s["Y"], s["T9"], s["rho"], *tol)


def work(case):
    """Inputs read and outputs written once; algorithmic flops at the
    workloads' mean per zone."""
    Z, K = case["Z"], case.get("K", 1)
    by, fl = 0.0, 0.0
    for name in case["workload"].split(","):
        sp = _spec(name)
        if case["kind"] == "costs":
            # start-up: two right-hand sides and, where T moves, two sets of rates
            by += Z * 8.0 * (sp.N + 3)
            fl += Z * (2.0 * 14 * sp.R + 2 * 6.0 * sp.R)
            continue
        by += Z * (16.0 * sp.N + 8 * 4 + 9 * 4 + 4)
        by += Z * 8.0 * ((sp.R if case.get("mult") == "zone" else 0) + bool(case.get("split")))
        fl += Z * FLOPS[name]
        if case["kind"] in ("autograd", "adjoint"):
            # cotangents in, gradients out; one transposed solve per step and set
            by += Z * K * 8.0 * (2 * sp.N + sp.R + 2)
            fl += Z * FLOPS[name] * (0.5 + 0.15 * K)
    return dict(bytes=by, flops=fl)


# ---------------------------------------------------------------- 64-bit values

class _Ode:
    """Right-hand side and Jacobian of a network on torch float64 tensors,
    state [Y_0.., T9, E]: the rate fits, tables and screening as published,
    written out here without the library.  Complex states and multipliers
    carry a derivative in their imaginary part."""

    def __init__(self, spec, T9, rho, Y, zeta, lnm, dev):
        t = lambda v, dt=T9.dtype: torch.as_tensor(np.asarray(v), dtype=dt, device=dev)
        self.spec, self.N, self.R = spec, spec.N, spec.R
        self.rho, self.lnm, self.T0 = rho, lnm, T9
        self.re = t(spec.reactants, torch.int64)
        nre = (self.re >= 0).sum(1)
        self.pre = rho[:, None] ** (nre - 1)[None, :]
        self.real = not T9.is_complex()
        if spec.scale is not None:
            self.pre = self.pre * t(spec.scale)
        S = np.zeros((spec.N, spec.R))
        for r in range(spec.R):
            for v in spec.reactants[r]:
                if v >= 0:
                    S[v, r] -= 1
            for v in spec.products[r]:
                if v >= 0:
                    S[v, r] += 1
        self.S, self.co = t(S), t(spec.coeffs)
        self.Q = t(np.zeros(spec.R) if spec.Q is None else spec.Q)
        self.h = None
        if spec.screen is not None and zeta is not None:
            self.h = t(spec.screen)[None, :] * (torch.sqrt(rho * zeta) * 10 ** -4.5)[:, None]
        self.ap = None if spec.ap_pg is None else t(spec.ap_pg, torch.bool)
        self.apc = None if spec.ap_pg is None else t(spec.ap_coeffs)
        self.tab = None
        if spec.tab_of is not None:
            d, u = t(spec.tab_dens), torch.log10(rho * (Y @ t(spec.charge)))
            i = torch.clamp(torch.searchsorted(d, u.contiguous()) - 1, 0, d.numel() - 2)
            w = torch.clamp((u - d[i]) / (d[i + 1] - d[i]), 0.0, 1.0)
            L = t(spec.tab_lnl)
            self.tab = ((1 - w)[:, None, None] * L[:, i].transpose(0, 1)
                        + w[:, None, None] * L[:, i + 1].transpose(0, 1))
            self.tab_r = [r for r in range(spec.R) if spec.tab_of[r] >= 0]
            self.tab_m = [int(spec.tab_of[r]) for r in self.tab_r]
            self.tT = t(spec.tab_t9)
        if not spec.self_heating:
            self.k0 = self.rates(T9)

    def take(self, m):
        """The zones of mask m."""
        o = object.__new__(_Ode)
        o.__dict__.update(self.__dict__)
        for k in ("rho", "T0", "pre", "h", "tab", "k0"):
            v = getattr(self, k, None)
            if v is not None:
                setattr(o, k, v[m])
        if self.lnm is not None and self.lnm.dim() == 2:
            o.lnm = self.lnm[m]
        return o

    def rates(self, T):
        c = (torch.clamp(T, min=1e-3) if self.real else T)[:, None]
        ph = torch.cat([torch.ones_like(c), 1 / c, c ** (-1 / 3), c ** (1 / 3), c, c ** (5 / 3),
                        torch.log(c)], 1)
        e = ph @ self.co.T
        if self.tab is not None:
            j = torch.clamp(torch.searchsorted(self.tT, T.contiguous()) - 1, 0,
                            self.tT.numel() - 2)
            v = torch.clamp((T - self.tT[j]) / (self.tT[j + 1] - self.tT[j]), 0.0, 1.0)[:, None]
            z = torch.arange(T.numel(), device=T.device)
            e = e.clone()
            e[:, self.tab_r] = ((1 - v) * self.tab[z, :, j] + v * self.tab[z, :, j + 1])[:, self.tab_m]
        add = torch.zeros_like(e) if self.lnm is None else self.lnm.expand_as(e)
        if self.h is not None:
            add = add + self.h * c ** -1.5
        lam = torch.exp(e + add)
        if self.ap is not None:
            x = torch.einsum("zk,rck->zrc", ph, self.apc)
            eff = lam + torch.exp(x[..., 0] + add) * torch.sigmoid(x[..., 1] - x[..., 2])
            lam = torch.where(self.ap[None, :], eff, lam)
        return lam * self.pre

    def k(self, x):
        return self.rates(x[:, self.N]) if self.spec.self_heating else self.k0

    def flow(self, k, x):
        y = torch.cat([x[:, :self.N], torch.ones_like(x[:, :1])], 1)   # index -1: one
        return k * y[:, self.re[:, 0]] * y[:, self.re[:, 1]] * y[:, self.re[:, 2]]

    def f(self, x, k=None):
        k = self.k(x) if k is None else k
        R = self.flow(k, x)
        ed = R @ self.Q
        dT = torch.zeros_like(ed)
        if self.spec.self_heating:
            dT = ed / (1.5 * x[:, :self.N].sum(1) + 1e-3 * x[:, self.N] ** 3)
        return torch.cat([R @ self.S.T, dT[:, None], ed[:, None]], 1)

    def jac(self, x):
        N, Z = self.N, x.shape[0]
        k = self.k(x)
        y = torch.cat([x[:, :N], torch.ones_like(x[:, :1])], 1)
        dR = torch.zeros(Z, self.R, N + 1, dtype=x.dtype, device=x.device)
        for a in range(3):
            b, c = (a + 1) % 3, (a + 2) % 3
            v = k * y[:, self.re[:, b]] * y[:, self.re[:, c]]
            idx = torch.where(self.re[:, a] >= 0, self.re[:, a], torch.full_like(self.re[:, a], N))
            dR.scatter_add_(2, idx[None, :, None].expand(Z, -1, 1), v[:, :, None])
        dR = dR[:, :, :N]
        J = torch.zeros(Z, N + 2, N + 2, dtype=x.dtype, device=x.device)
        J[:, :N, :N] = torch.einsum("ir,zrj->zij", self.S, dR)
        J[:, N + 1, :N] = torch.einsum("r,zrj->zj", self.Q, dR)
        if self.spec.self_heating:
            T, R = x[:, N], self.flow(k, x)
            g = (torch.log(self.rates(T * (1 + 1e-6))) - torch.log(self.rates(T * (1 - 1e-6)))) \
                / (2e-6 * T)[:, None]
            RT = torch.nan_to_num(R * g)
            J[:, :N, N] = RT @ self.S.T
            J[:, N + 1, N] = RT @ self.Q
            cv = 1.5 * x[:, :N].sum(1) + 1e-3 * T ** 3
            ed = R @ self.Q
            J[:, N, :N + 1] = J[:, N + 1, :N + 1] / cv[:, None]
            J[:, N, :N] -= (1.5 * ed / cv ** 2)[:, None]
            J[:, N, N] -= 3e-3 * T ** 2 * ed / cv ** 2
        return J


def _integrate(ode, x, t_end, h0, rtol=1e-11, atol=1e-16, cols=8):
    """Final states of every zone by extrapolated linearly implicit Euler
    steps (Deuflhard's harmonic sequence, ``cols`` columns), each zone its
    own step size."""
    out = x.clone()
    live = torch.arange(x.shape[0], device=x.device)
    t, h = torch.zeros_like(t_end), torch.minimum(h0, t_end)
    n = x.shape[1]
    eye = torch.eye(n, dtype=x.dtype, device=x.device)
    for it in range(20000):
        J = ode.jac(x)
        k0 = None if ode.spec.self_heating else ode.k0
        prev = []
        for j in range(1, cols + 1):
            A, hj = eye / (h / j)[:, None, None] - J, None
            LU, piv, _ = torch.linalg.lu_factor_ex(A)
            y = x
            for _ in range(j):
                y = y + torch.linalg.lu_solve(LU, piv, ode.f(y, k0)[:, :, None])[:, :, 0]
            row = [y]
            for m in range(1, j):
                row.append(row[m - 1] + (row[m - 1] - prev[m - 1]) / (j / (j - m) - 1.0))
            prev = row
        err = ((row[-1] - row[-2]).abs()
               / (atol + rtol * torch.maximum(x.abs(), row[-1].abs()))).amax(1)
        err = torch.nan_to_num(err, nan=1e30, posinf=1e30)
        ok = err <= 1.0
        x = torch.where(ok[:, None], row[-1], x)
        last = t + h >= t_end * (1 - 1e-14)
        t = torch.where(ok, t + h, t)
        done = ok & last
        h = h * torch.clamp(0.8 * torch.clamp(err, min=1e-30) ** (-1.0 / cols), 0.1, 4.0)
        h = torch.minimum(h, t_end - t)
        if it % 8 == 0 or bool(done.any()):
            if bool(done.any()):
                out[live[done]] = x[done]
                keep = ~done
                live, x, t, h, t_end = live[keep], x[keep], t[keep], h[keep], t_end[keep]
                ode = ode.take(keep)
            if live.numel() == 0:
                return out
    raise RuntimeError("the reference integration did not finish")


def _exact_burn(spec, a, lnm, dev):
    t = lambda v: torch.as_tensor(v, dtype=torch.float64, device=dev)
    Y, T9, rho = (torch.as_tensor(a[k], device=dev) for k in ("Y", "T9", "rho"))
    zeta = None if a["zeta"] is None else t(a["zeta"])
    ode = _Ode(spec, T9, rho, Y, zeta,
               None if lnm is None else torch.as_tensor(lnm, device=dev), dev)
    x = torch.cat([Y, T9[:, None], torch.zeros_like(T9[:, None])], 1)
    te = t(a["t_end"]).expand(T9.shape[0]).clone()
    f = ode.f(x)
    h0 = 1e-6 * torch.clamp(1.0 / (f.abs() / (1e-12 + x.abs())).amax(1), max=1.0)
    x = _integrate(ode, x, te, torch.clamp(h0, min=1e-30))
    N = spec.N
    E = x[:, N + 1] if spec.Q is not None else torch.zeros_like(T9)
    return dict(Y=x[:, :N], T9=x[:, N] if spec.self_heating else T9, E=E, counters=None,
                status=None)


def _exact_costs(spec, cfg, a, dev):
    """(1 + ln(t_end / h0))^2 with the starting step of Hairer, Norsett and
    Wanner, Solving ODEs I, II.4."""
    t = lambda v: torch.as_tensor(v, dtype=torch.float64, device=dev)
    Y, T9, rho = t(a["Y"]), t(a["T9"]), t(a["rho"])
    ode = _Ode(spec, T9, rho, Y, None, None, dev)
    n = spec.N + int(spec.self_heating)
    x = torch.cat([Y, T9[:, None], torch.zeros_like(T9[:, None])], 1)
    f0 = ode.f(x)
    w = 1.0 / (cfg["atol"] + cfg["rtol"] * x.abs())
    rms = lambda v: torch.sqrt((v * w)[:, :n].square().mean(1))
    d0, d1, te = rms(x), rms(f0), float(cfg["t_end"])
    hp = torch.where((d0 < 1e-5) | (d1 < 1e-5), torch.full_like(d0, 1e-6), 0.01 * d0 / d1)
    hp = torch.clamp(hp, max=te)
    x1 = x + hp[:, None] * f0
    x1[:, spec.N + 1] = 0.0
    if not spec.self_heating:
        x1[:, spec.N] = T9
    d2 = rms((ode.f(x1) - f0) / hp[:, None])
    dm = torch.maximum(d1, d2)
    h1 = torch.where(dm <= 1e-15, torch.clamp(hp * 1e-3, min=1e-6), torch.sqrt(0.01 / dm))
    h = torch.clamp(torch.minimum(100.0 * hp, h1), max=te)
    h = torch.clamp(h, min=1e-30 * te)
    return (1.0 + torch.clamp(torch.log(te / h), min=0.0)) ** 2


def exact(case, seed):
    names = case["workload"].split(",")
    cfg, kind = gen.CONFIGS[names[0]], case["kind"]
    dev = DEV if torch.cuda.is_available() else "cpu"
    a = _inputs(case, seed)
    if kind == "costs":
        return _exact_costs(_spec(names[0]), cfg, a, dev)
    if kind in ("coop", "adjoint") or case["Z"] > 13000:
        return None      # minutes in this form
    if kind == "multi":
        return [_exact_burn(_spec(n), a, None, dev) for n in names]
    base = _exact_burn(_spec(names[0]), a, a["lnm"], dev)
    if kind != "autograd":
        return base
    if case["Z"] > 256:
        return dict(base, gY=None, gT9=None, glnm=None)
    # the loss's derivatives by every multiplier, initial abundance and initial
    # temperature, each the imaginary part of a burn perturbed along it
    spec, Z, eps = _spec(names[0]), case["Z"], 1e-30
    P = spec.R + spec.N + 1
    b = dict(Y=np.concatenate([a["Y"]] * P) + 0j, T9=np.concatenate([a["T9"]] * P) + 0j,
             rho=np.concatenate([a["rho"]] * P), zeta=None, t_end=a["t_end"])
    lnm = np.zeros((P, Z, spec.R), complex)
    for r in range(spec.R):
        lnm[r, :, r] = 1j * eps
    for i in range(spec.N):
        b["Y"][(spec.R + i) * Z:(spec.R + i + 1) * Z, i] += 1j * eps
    b["T9"][(P - 1) * Z:] += 1j * eps
    o = _exact_burn(spec, b, lnm.reshape(P * Z, spec.R), dev)
    wY = torch.as_tensor(np.tile(a["wY"], (P, 1)), device=dev)
    g = (((wY * o["Y"].imag).sum(1) + o["E"].imag) / eps).reshape(P, Z)
    return dict(base, gY=g[spec.R:spec.R + spec.N].T.contiguous(), gT9=g[-1],
                glnm=g[:spec.R].sum(1))
