"""The work whose speed counts: Newton power-flow solves through the package's entry points.

Every case solves load scenarios of a seeded grid to a power mismatch of 1e-8 pu, as a user of the
library does: a study of many load scenarios of one grid (device buffers, pinned or pageable host
buffers), a single solve inside somebody's loop, a handful of served requests of different grids.
Grids are those of the benchmark and the tests (14, 2,000 and 10,000 buses, the 8,000-node feeder)
and grids of the same generator at other, odd sizes.

A case is a dict:
  call       "device": pf_solve_batch_device on device buffers; "pinned": pf_solve_batch on pinned
             host buffers; "host": pf_solve_batch on pageable host buffers; "serve": pf_submit of
             requests of several grids, pf_drain, pf_poll of each result
  kind       "mesh" (single phase) or "feeder" (three phase)
  n, topo    buses or nodes, and the seed of the topology ("serve": the largest grid's buses)
  angle      meshes: the loading, as the DC angle across the most loaded branch (rad)
  B          scenarios ("serve": grids, each with two requests)
  precision, method, qlim, tuned   options of the solve; tuned: pf_autotune ran once on the handle

Voltages are returned whole, and the status of every solve.  The final mismatch is not: below the
stop test it is rounding noise.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1711_10579_gb300 import cases as grids
from paper_1711_10579_gb300 import pf

DEV = "cuda:0"
SIGMA = 0.2  # spread of the lognormal load multipliers of a scenario


def _case(name, call, kind, n, B, precision="mixed", method="nr", topo=0, angle=0.1, qlim=False,
          tuned=False):
    return {"name": name, "call": call, "kind": kind, "n": n, "B": B, "precision": precision,
            "method": method, "topo": topo, "angle": angle, "qlim": qlim, "tuned": tuned}


def listed():
    return [
        # the smallest call: one 14-bus solve between host arrays, where a program solves small
        # grids one after another and latency is all
        _case("mesh14_x1_host", "host", "mesh", 14, 1, angle=0.3),
        # one FP64 solve of a mid-size grid of odd size: the plain double-precision Newton
        _case("mesh2749_x1_fp64", "device", "mesh", 2749, 1, precision="fp64", topo=3),
        # one mixed-precision solve of a large grid, as inside a control loop
        _case("mesh10000_x1_mixed", "device", "mesh", 10_000, 1, angle=0.3),
        # one three-phase solve of the 8,000-node feeder in double precision
        _case("feeder8000_x1_fp64", "device", "feeder", 8_000, 1, precision="fp64"),
        # load profiles of one distribution feeder (an hour by the minute), host buffers
        _case("feeder1000_x61_pinned", "pinned", "feeder", 1_000, 61),
        # very many scenarios of a tiny grid: a Monte Carlo study
        _case("mesh14_x9728_mixed", "device", "mesh", 14, 9_728, angle=0.3, tuned=True),
        # the batched configuration of the tests: 2,000 buses x 512 scenarios
        _case("mesh2000_x512_mixed", "device", "mesh", 2_000, 512, angle=0.3),
        # the benchmark's step: 10,000 buses x 9,728 scenarios, autotuned
        _case("mesh10000_x9728_mixed", "device", "mesh", 10_000, 9_728, angle=0.3, tuned=True),
        # the same grid in double precision, 4 scenarios per SM, library defaults
        _case("mesh10000_x608_fp64", "device", "mesh", 10_000, 608, precision="fp64", angle=0.3),
        # Newton-Krylov (GMRES with ILU(0)) on the 2,000-bus grid
        _case("mesh2000_x1_nk", "device", "mesh", 2_000, 1, method="nk", angle=0.3),
        # reactive limits of generators enforced over a batch, pageable host buffers
        _case("mesh500_x255_qlim_host", "host", "mesh", 500, 255, topo=2, qlim=True),
        # a burst of requests of twelve grids of different sizes through the serving runtime
        _case("serve_12grids_x2", "serve", "mesh", 10_000, 12),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: any size from 14 to 10,000 buses (12 to 8,000 nodes), any
    batch whose scenarios x buses the benchmark's step is not below.  Loading 0.06 rad: every grid
    the generator draws at it has a solution that flat start reaches."""
    kind = rng.choice(["mesh1", "feeder1", "mesh", "mesh", "mesh", "small", "feeder", "nk", "qlim",
                       "serve"])
    prec = rng.choice(["mixed", "mixed", "fp64"])
    c = _case("", "device", "mesh", 0, 1, precision=prec, topo=rng.randrange(200), angle=0.06)
    if kind == "mesh1":
        c.update(call=rng.choice(["device", "host"]), n=_log(rng, 14, 10_000))
    elif kind == "feeder1":
        c.update(call=rng.choice(["device", "host"]), kind="feeder", n=_log(rng, 12, 8_000))
    elif kind == "mesh":
        n = _log(rng, 300, 10_000)
        cap = 9_728 * 10_000 // 8 if prec == "fp64" else 9_728 * 10_000 // 2
        c.update(call=rng.choice(["device", "device", "pinned"]), n=n,
                 B=_log(rng, 17, min(9_728, cap // n)))
    elif kind == "small":
        c.update(n=_log(rng, 14, 300), B=_log(rng, 500, 9_728))
    elif kind == "feeder":
        c.update(call=rng.choice(["device", "pinned"]), kind="feeder", n=_log(rng, 100, 4_000))
        c["B"] = _log(rng, 5, max(6, min(500, 400_000 // c["n"])))
    elif kind == "nk":
        c.update(method="nk", n=_log(rng, 100, 2_000))
    elif kind == "qlim":
        c.update(call="host", qlim=True, n=_log(rng, 50, 600), B=_log(rng, 17, 300))
    else:
        c.update(call="serve", precision="mixed", n=_log(rng, 2_000, 10_000),
                 B=rng.randrange(3, 14))
    return {k: v for k, v in c.items() if k != "name"}


# ---------------------------------------------------------------------------
# grids, handles and inputs
# ---------------------------------------------------------------------------

@functools.lru_cache(maxsize=32)
def _grid(kind, n, topo, angle, qlim):
    """The seeded grid (numbers only)."""
    if kind == "feeder":
        return grids.feeder_case(n, topo)
    m, pv = (20, 4) if n == 14 else (int(round(1.35 * n)), n // 5)
    g = grids.transmission_case(n, m, pv, topo, max_angle=angle)
    return grids.with_q_limits(g, topo + 1) if qlim else g


def _grids(case):
    """The case's grids: one, or the pool of a serving case (two meshes to one feeder, sizes
    spread over the logarithm up to n buses)."""
    if case["call"] != "serve":
        return [_grid(case["kind"], case["n"], case["topo"], case["angle"], case["qlim"])]
    out = []
    for k in range(case["B"]):
        n = int(round(500 * (case["n"] / 500) ** ((k + 1) / case["B"])))
        out.append(_grid("feeder", max(12, n // 2), case["topo"] + k, 0.0, False) if k % 3 == 1
                   else _grid("mesh", n, case["topo"] + k, case["angle"], False))
    return out


class _Handle:
    """Created cases of a context, as a program keeps them from call to call."""

    def __init__(self, case):
        self.cases = [pf.pf_create_case(_ctx(), g) for g in _grids(case)]
        if case["tuned"]:
            pf.pf_autotune(self.cases[0], case["B"], _opts(case))

    def __del__(self):
        for c in self.cases:
            pf.pf_destroy_case(c)


@functools.lru_cache(maxsize=1)
def _ctx():
    return pf.pf_ctx_create(0)


@functools.lru_cache(maxsize=1)  # the newest only: a batch's workspace takes tens of GB
def _handle(key):
    return _Handle(dict(key))


def _opts(case):
    return pf.make_opts(method=pf.PF_NK if case["method"] == "nk" else pf.PF_NR,
                        precision=pf.PF_FP64 if case["precision"] == "fp64" else pf.PF_MIXED,
                        q_limits=int(case["qlim"]))


def _loads(g, B, seed):
    """Loads [B, slots] of B scenarios on the GPU: every bus (node) load x lognormal(0, 0.2),
    generation rescaled to 1.05 x the scenario's load (None for a feeder)."""
    rng = torch.Generator(device=DEV).manual_seed(int(seed))
    feeder = isinstance(g, grids.ThreePhaseCase)
    n = g.n_node if feeder else g.n_bus
    mult = torch.exp(SIGMA * torch.randn((B, n), generator=rng, device=DEV, dtype=torch.float64))
    p, q = (torch.tensor(np.asarray(a), device=DEV) for a in (g.p_load, g.q_load))
    if feeder:
        return (p * mult[:, :, None]).reshape(B, -1), (q * mult[:, :, None]).reshape(B, -1), None
    pl, ql = p * mult, q * mult
    w = torch.tensor(np.where(g.bus_type == grids.PV, g.p_gen, 0.0), device=DEV)
    return pl, ql, 1.05 * pl.sum(1, keepdim=True) * (w / w.sum())


def _host(t, pinned):
    if t is None:
        return None
    return t.cpu().pin_memory().numpy() if pinned else t.cpu().numpy()


def prepare(case, seed):
    h = _handle(tuple((k, v) for k, v in sorted(case.items()) if k != "name"))
    s = {"call": case["call"], "handle": h, "case": h.cases[0], "opts": _opts(case),
         "B": case["B"]}
    if case["call"] == "serve":
        s["requests"] = []
        for k, (c, g) in enumerate(zip(h.cases, _grids(case))):
            ld = [None if a is None else a.cpu().numpy() for a in _loads(g, 2, seed * 64 + k)]
            for r in range(2):
                s["requests"].append((c, *[None if a is None else a[r] for a in ld]))
        return s
    loads = _loads(_grids(case)[0], case["B"], seed)
    shape = tuple(loads[0].shape)
    if case["call"] == "device":
        s["in"] = loads
        s["vm"], s["va"] = (torch.zeros(shape, dtype=torch.float64, device=DEV) for _ in range(2))
        s["info"] = torch.zeros((case["B"], pf.INFO_DTYPE.itemsize // 4), dtype=torch.int32,
                                device=DEV)
    else:
        pin = case["call"] == "pinned"
        s["in"] = tuple(_host(a, pin) for a in loads)
        vm, va = (_host(torch.zeros(shape, dtype=torch.float64), pin) for _ in range(2))
        info = _host(torch.zeros(case["B"] * pf.INFO_DTYPE.itemsize, dtype=torch.uint8), pin)
        s["out"] = (vm, va, info.view(pf.INFO_DTYPE))
    return s


def run(s):
    if s["call"] == "device":
        pl, ql, pg = s["in"]
        pf.pf_solve_batch_device(s["case"], s["B"], pl, ql, pg, s["opts"], s["vm"], s["va"],
                                 s["info"], torch.cuda.current_stream().cuda_stream)
        return {"vm": s["vm"], "va": s["va"], "status": s["info"][:, 0]}
    if s["call"] == "serve":
        ctx = _ctx()
        tickets = [pf.pf_submit(ctx, c, pl, ql, pg, s["opts"]) for c, pl, ql, pg in s["requests"]]
        pf.pf_drain(ctx)
        got = [pf.pf_poll(ctx, t, r[0].slots) for t, r in zip(tickets, s["requests"])]
        return {"vm": [g[0] for g in got], "va": [g[1] for g in got],
                "status": np.array([g[2]["status"] for g in got])}
    pl, ql, pg = s["in"]
    vm, va, info = pf.pf_solve_batch(s["case"], pl, ql, pg, s["opts"], out=s["out"])
    return {"vm": vm, "va": va, "status": info["status"]}


# ---------------------------------------------------------------------------
# what a pass cannot do without, and how exact it is
# ---------------------------------------------------------------------------

def work(case):
    """Bytes: loads (and generation) in, voltages out, the branch data once.  Flops: Newton steps x
    what one takes on such a sparse grid (mismatch and Jacobian over 3.7 entries per bus, a block
    factorisation of about 5 entries and 6.6 block updates per bus, two triangular solves; three
    phase 3 entries and one update of 6x6 blocks per node), the Krylov solver's about 150 products
    and preconditioner solves per Newton step."""
    nbytes = flops = 0
    each = 2 if case["call"] == "serve" else case["B"]
    for g in _grids(case):
        if isinstance(g, grids.ThreePhaseCase):
            nbytes += g.n_node * (each * 3 * 8 * 4 + 9 * 16)
            flops += 2 * each * g.n_node * 2_400
        else:
            nbytes += g.n_bus * (each * 8 * 5 + 60)
            steps = 8 if case["qlim"] else 4
            per = 350 if case["method"] == "nr" else 150 * 200
            flops += steps * each * g.n_bus * per
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Every solve ends at a power mismatch of at most 1e-8 pu, wherever in that interval its last
    step leaves it: against exact() up to 1.4e-8 (a mixed-precision feeder; most grids 1e-9 and
    less), and four times that is stated."""
    return {"rel": 6e-8, "max": 4e-6, "differ": 0.0}


# ---------------------------------------------------------------------------
# the same solutions in plain torch, 64 bits
# ---------------------------------------------------------------------------

def _current(g, V):
    """I = Y V of [n, B] voltages, branch by branch (pi model)."""
    f, t = (torch.tensor(a, device=DEV, dtype=torch.int64) for a in (g.br_from, g.br_to))
    y = torch.tensor(1.0 / (g.br_r + 1j * g.br_x), device=DEV)[:, None]
    sh = torch.tensor(0.5j * g.br_b, device=DEV)[:, None]
    Vf, Vt = V[f], V[t]
    flow = y * (Vf - Vt)
    I = torch.zeros_like(V)
    I.index_add_(0, f, flow + sh * Vf)
    I.index_add_(0, t, sh * Vt - flow)
    return I


def _ybus(g):
    return _current(g, torch.eye(g.n_bus, device=DEV, dtype=torch.complex128))


def _jacobian(Y, V):
    """[[dP/d delta, dP/d|V|], [dQ/d delta, dQ/d|V|]] at V [n] (constant-power loads)."""
    I = Y @ V
    U = V / V.abs()
    dd = -1j * V[:, None] * (Y * V[None, :]).conj()
    dd.diagonal().add_(1j * V * I.conj())
    dm = V[:, None] * (Y * U[None, :]).conj()
    dm.diagonal().add_(U * I.conj())
    return torch.cat([torch.cat([dd.real, dm.real], 1), torch.cat([dd.imag, dm.imag], 1)], 0)


def _exact_mesh(g, pl, ql, pg):
    """Polar Newton with a Jacobian frozen at the grid's own solution (its inverse in 32 bits; the
    mismatch in 64): converges to the accuracy of the mismatch."""
    n, B = g.n_bus, pl.shape[0]
    bt = torch.tensor(np.asarray(g.bus_type), device=DEV)
    P = (pg - pl).T
    Q = torch.tensor(g.q_gen, device=DEV)[:, None] - ql.T
    free = torch.cat([torch.nonzero(bt != 0)[:, 0], n + torch.nonzero(bt == 2)[:, 0]])
    Y = _ybus(g)

    def mismatch(vm, va, P, Q):
        V = torch.polar(vm, va)
        S = V * _current(g, V).conj()
        return torch.cat([P - S.real, Q - S.imag])[free]

    def add(vm, va, dx):
        x = torch.cat([va, vm])
        x.index_add_(0, free, dx)
        return x[n:], x[:n]

    vm0 = torch.where(bt == 2, 1.0, torch.tensor(g.v_set, device=DEV))[:, None]
    vm, va = vm0.clone(), torch.zeros_like(vm0)
    own = [torch.tensor(a, device=DEV)[:, None] for a in (g.p_gen - g.p_load, g.q_gen - g.q_load)]
    for _ in range(8):
        J = _jacobian(Y, torch.polar(vm, va)[:, 0])[free][:, free].float()
        d = torch.linalg.solve(J, mismatch(vm, va, *own).float())
        vm, va = add(vm, va, d.double())
        if d.abs().max() < 1e-5:
            break
    inv = torch.linalg.inv(J)
    out_m, out_a = (torch.empty((B, n), dtype=torch.float64, device=DEV) for _ in range(2))
    step = max(1, (1 << 24) // n)
    for b in range(0, B, step):
        e = min(B, b + step)
        m, a = vm.expand(n, e - b).contiguous(), va.expand(n, e - b).contiguous()
        last = math.inf
        for _ in range(80):
            f = mismatch(m, a, P[:, b:e], Q[:, b:e])
            r = float(f.abs().max())
            if not r < 1e4 or r < 1e-14 or (r < 1e-11 and r > 0.5 * last):
                break
            last = r
            m, a = add(m, a, (inv @ f.float()).double())
        out_m[b:e], out_a[b:e] = m.T, a.T
    return out_m, out_a


def _exact_qlim(g, pl, ql, pg):
    """Rounds of full Newton solves, all scenarios at once; after each, every PV bus outside its
    reactive limits becomes PQ at the limit."""
    n, B = g.n_bus, pl.shape[0]
    bt = torch.tensor(np.asarray(g.bus_type), device=DEV)[None].repeat(B, 1)
    P = pg - pl
    Qg = torch.tensor(g.q_gen, device=DEV)[None].repeat(B, 1)
    lo, hi = (torch.tensor(a, device=DEV)[None] for a in (g.q_min, g.q_max))
    Y = _ybus(g)
    vm = torch.where(bt == 2, 1.0, torch.tensor(g.v_set, device=DEV)[None])
    va = torch.zeros_like(vm)
    for _ in range(64):
        for _ in range(20):
            V = torch.polar(vm, va)
            I = V @ Y.T
            S = V * I.conj()
            on = torch.cat([bt != 0, bt == 2], 1)
            f = torch.where(on, torch.cat([P - S.real, Qg - ql - S.imag], 1), 0.0)
            if f.abs().max() < 1e-12:
                break
            U = V / V.abs()
            dd = -1j * V[:, :, None] * (Y[None] * V[:, None, :]).conj()
            dd.diagonal(dim1=1, dim2=2).add_(1j * S)
            dm = V[:, :, None] * (Y[None] * U[:, None, :]).conj()
            dm.diagonal(dim1=1, dim2=2).add_(U * I.conj())
            J = torch.cat([torch.cat([dd.real, dm.real], 2), torch.cat([dd.imag, dm.imag], 2)], 1)
            J = J * (on[:, :, None] & on[:, None, :])
            J.diagonal(dim1=1, dim2=2).add_((~on).double())
            dx = torch.linalg.solve(J, f)
            va, vm = va + dx[:, :n], vm + dx[:, n:]
        q = S.imag + ql
        over, under = (bt == 1) & (q > hi), (bt == 1) & (q < lo)
        if not bool((over | under).any()):
            break
        Qg = torch.where(over, hi, torch.where(under, lo, Qg))
        bt = torch.where(over | under, 2, bt)
    return vm, va


def _exact_feeder(g, pl, ql):
    """Backward / forward sweeps over the tree: load currents summed towards the source, voltage
    drops taken from it."""
    n, B = g.n_node, pl.shape[0]
    parent = np.full(n, -1)
    parent[g.br_to] = g.br_from
    Z = np.zeros((n, 3, 3), dtype=np.complex128)
    Z[g.br_to] = g.br_z
    has = ((g.phases[:, None] >> np.arange(3)[None]) & 1).astype(bool)
    Z *= has[:, :, None] & has[:, None, :]
    depth = np.zeros(n, dtype=int)
    for k in range(1, n):
        depth[k] = depth[parent[k]] + 1
    levels = [torch.tensor(np.flatnonzero(depth == d), device=DEV) for d in range(1, depth.max() + 1)]
    par, Z = torch.tensor(parent, device=DEV), torch.tensor(Z, device=DEV)
    mask = torch.tensor(has, device=DEV)[:, :, None]
    S = torch.complex(pl, ql).reshape(B, n, 3).permute(1, 2, 0).contiguous()
    zp, zi, zz = (torch.tensor(g.zip[:, k].copy(), device=DEV)[:, None, None] for k in range(3))
    src = g.v_source * np.exp(-2j * np.pi / 3 * np.arange(3))
    V = torch.tensor(src, device=DEV)[None, :, None].expand(n, 3, B) * mask
    S[0] = 0
    for _ in range(60):
        m = V.abs()
        I = torch.where(mask, (S * (zp + zi * m + zz * m * m) / torch.where(mask, V, 1.0)).conj(), 0)
        for lv in reversed(levels):
            I.index_add_(0, par[lv], I[lv])
        W = V.clone()
        for lv in levels:
            W[lv] = (W[par[lv]] - torch.einsum("nij,njb->nib", Z[lv], I[lv])) * mask[lv]
        d = float((W - V).abs().max())
        V = W
        if d < 1e-15:
            break
    V = V.permute(2, 0, 1).reshape(B, -1)
    return V.abs(), torch.where(V.abs() > 0, V.angle(), 0.0)


def _exact_one(g, loads, qlim):
    if isinstance(g, grids.ThreePhaseCase):
        return _exact_feeder(g, loads[0], loads[1])
    return (_exact_qlim if qlim else _exact_mesh)(g, *loads)


def exact(case, seed):
    if case["call"] != "serve":
        g = _grids(case)[0]
        vm, va = _exact_one(g, _loads(g, case["B"], seed), case["qlim"])
        return {"vm": vm, "va": va, "status": None}
    vm, va = [], []
    for k, g in enumerate(_grids(case)):
        m, a = _exact_one(g, _loads(g, 2, seed * 64 + k), False)
        vm += [m[0], m[1]]
        va += [a[0], a[1]]
    return {"vm": vm, "va": va, "status": None}
