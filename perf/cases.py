"""Performance cases of the traveltime-parameter search.

Each case is one call (or one short chain of calls) that a program makes
through the package's entry points, on seeded synthetic gathers built on the
GPU: Ricker events on CRS surfaces plus Gaussian noise, with the shapes of the
repository's workloads (CMP gather, CRS line, FO-CRS common-offset section,
batched uneven problems, large BF16-stored line). A line case solves the CMPs
of an interior slab of a longer line, so its apertures are whole; the ENS and
stack cases take a complete line, whose end apertures are clipped.

    listed()            the named cases
    draw(rng)           one more case of the same ranges
    prepare(case, seed) context, parameter vectors and whatever a program keeps
    run(state)          one pass
    work(case)          bytes and operations no implementation can avoid
    exact(case, seed)   the outputs of evaluations in 64 bits (plain torch)
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2304_11399_gb300 as tt

CMP, CRS, FO = 0, 1, 2
DIM = {"cmp": 1, "crs": 3, "fo": 5}
OP = {"cmp": CMP, "crs": CRS, "fo": FO}
LO = {"cmp": (1.0 / 4500.0 ** 2,), "crs": (-6e-4, -1.5e-7, 1.0 / 4800.0 ** 2),
      "fo": (-6e-4, -1e-4, -3e-7, -1e-6, -2e-8)}
HI = {"cmp": (1.0 / 1400.0 ** 2,), "crs": (6e-4, 1.5e-7, 1.0 / 1400.0 ** 2),
      "fo": (6e-4, 8e-4, 3e-7, 1e-6, 1.0 / 1400.0 ** 2 + 2e-8)}
DCMP, DOFF, H0 = 12.5, 50.0, 1000.0
DEV = "cuda"


def _line(name, kind, *, op="crs", n_cmp, ns=1500, dt=0.004, n_off=48, ap_half=10, whole=False,
          storage="f32", w=5, P=1, spread=1.0, events=20, snr=3.0, np_=64, ng=0, exch=0,
          polish=0, adapt=0, n_skip=2, n_bucket=64, n_cycle=1, n_points=0):
    c = dict(name=name, kind=kind, op=op, n_cmp=n_cmp, ns=ns, dt=dt, n_off=n_off,
             ap_half=ap_half, whole=whole, storage=storage, w=w, P=P, spread=spread,
             events=events, snr=snr, np=np_, ng=ng, exch=exch, polish=polish, adapt=adapt,
             n_skip=n_skip, n_bucket=n_bucket, n_cycle=n_cycle, n_points=n_points)
    if name is None:
        del c["name"]
    return c


def _batch(name, *, n_prob, ng, ntr_lo=16, ntr_hi=240, ns_lo=750, ns_hi=3000, np_=64, w=5,
           adapt=0):
    c = dict(name=name, kind="batched", op="crs", n_prob=n_prob, ntr_lo=ntr_lo, ntr_hi=ntr_hi,
             ns_lo=ns_lo, ns_hi=ns_hi, np=np_, ng=ng, w=w, storage="f32", adapt=adapt)
    if name is None:
        del c["name"]
    return c


def listed():
    return [
        # a velocity search on one CMP gather (48 traces, 500 samples, DE 32 x 50): the
        # smallest whole search, an interactive velocity analysis
        _line("cmp_search", "search", op="cmp", n_cmp=1, ns=500, ap_half=0, events=8, snr=5.0,
              np_=32, ng=50),
        # the main workload's search (DE 64 x 100, exchange every 10 generations, 5 polish
        # steps, apertures of +-10 CMPs) on 12 CMPs of the line
        _line("crs_search", "search", n_cmp=12, np_=64, ng=100, exch=10, polish=5),
        # independent uneven problems (16-240 traces, 750-3000 samples) searched in one
        # batch, DE 64 x 80
        _batch("batched_search", n_prob=64, ng=80),
        # the ENS 5 x 1 sweep over a whole 200-CMP line: many small dependent launches
        _line("ens_sweep", "ens", n_cmp=200, whole=True, np_=5, ng=1),
        # a first-generation population on 20 CMPs of the line: parameters uniform in the bounds
        _line("line_eval_random", "eval", n_cmp=20, P=64),
        # a late-generation population: each sample's members close to one another
        _line("line_eval_late", "eval", n_cmp=20, P=64, spread=0.02),
        # the large line's apertures (+-25 CMPs x 120 offsets at 2 ms), BF16-stored traces,
        # NP 96, midway through a search
        _line("large_bf16_eval", "eval", n_cmp=2, ns=2000, dt=0.002, n_off=120, ap_half=25,
              storage="bf16", P=96, spread=0.1, events=60, snr=2.0),
        # five-parameter FO-CRS population on a common-offset section
        _line("fo_eval", "eval", op="fo", n_cmp=12, ap_half=8, P=64, spread=0.1),
        # coherence of a handful of trial parameter sets along one CMP (a panel looked at
        # interactively): too few pairs to fill the GPU one warp per 64
        _line("panel_eval", "eval", n_cmp=1, P=5, spread=0.3),
        # S and dS/dtheta of one parameter vector per sample through autograd, 40 CMPs of
        # the line: a refinement step driven by a user's own optimiser
        _line("line_grad", "grad", n_cmp=40, P=1, spread=0.05),
        # the same at 1000 scattered points of one CMP gather: the smallest call
        _line("points_grad", "grad", n_cmp=1, ns=500, ap_half=0, events=8, snr=5.0, P=1,
              n_points=1000),
        # the stacked section of a whole line along the searched operators
        _line("line_stack", "stack", n_cmp=200, whole=True, P=1, spread=0.05),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search", "search", "batched", "ens", "eval", "eval", "eval", "grad", "grad",
                       "points", "stack"])
    w = rng.choice([3, 5, 5, 5, 8])
    if kind == "batched":
        return _batch(None, n_prob=_log(rng, 4, 48), ng=_log(rng, 10, 80),
                      np_=rng.choice([24, 50, 64]), w=rng.choice([4, 5]), adapt=rng.choice([0, 1]))
    if kind == "search":
        if rng.random() < 0.4:
            return _line(None, "search", op="cmp", n_cmp=1, ns=_log(rng, 120, 1000), ap_half=0,
                         n_off=rng.randint(24, 60), events=8, snr=5.0, np_=rng.choice([16, 32, 37]),
                         ng=_log(rng, 10, 60), w=w, polish=rng.choice([0, 3]))
        op = rng.choice(["crs", "crs", "fo"])
        return _line(None, "search", op=op, n_cmp=rng.randint(2, 8), ns=_log(rng, 200, 1500),
                     ap_half=rng.randint(4, 10), np_=rng.choice([30, 48, 64]),
                     ng=_log(rng, 10, 60), exch=rng.choice([0, 5, 10]), polish=rng.choice([0, 5]),
                     storage=rng.choice(["f32", "f32", "bf16"]), adapt=rng.choice([0, 1]))
    if kind == "ens":
        np_ = rng.choice([5, 8, 20])
        return _line(None, "ens", n_cmp=rng.randint(20, 120), ns=_log(rng, 300, 1500), whole=True,
                     np_=np_, ng=rng.choice([1, 2, 5]), n_skip=rng.choice([0, 1, 2]),
                     n_bucket=rng.choice([16, 64]), adapt=rng.choice([0, 1]))
    if kind == "points":
        return _line(None, "grad", op=rng.choice(["cmp", "crs"]), n_cmp=1, ns=_log(rng, 200, 2500),
                     ap_half=0, events=8, snr=5.0, P=rng.choice([1, 3]), w=w,
                     n_points=_log(rng, 100, 4000))
    if kind == "grad":
        return _line(None, "grad", op=rng.choice(["crs", "crs", "fo"]), n_cmp=_log(rng, 1, 30),
                     ns=_log(rng, 300, 2600), ap_half=rng.randint(3, 10), P=1, w=w,
                     spread=rng.choice([0.02, 0.1, 1.0]),
                     storage=rng.choice(["f32", "f32", "bf16"]))
    if kind == "stack":
        return _line(None, "stack", op=rng.choice(["crs", "crs", "fo"]), n_cmp=_log(rng, 1, 150),
                     ns=_log(rng, 300, 2600), ap_half=rng.randint(3, 15), whole=True, P=1,
                     spread=rng.choice([0.02, 0.1]), storage=rng.choice(["f32", "f32", "bf16"]))
    big = rng.random() < 0.25
    return _line(None, "eval", op=rng.choice(["crs", "crs", "fo"]), n_cmp=_log(rng, 1, 3 if big else 16),
                 ns=_log(rng, 300, 2600), dt=0.002 if big else 0.004, n_off=120 if big else 48,
                 ap_half=rng.randint(15, 25) if big else rng.randint(2, 12),
                 storage=rng.choice(["f32", "bf16"]), P=_log(rng, 2, 96), w=w,
                 spread=rng.choice([0.01, 0.05, 0.2, 1.0]))


# ---- inputs -------------------------------------------------------------------------------


def _events(n, x0, x1, tau_max, op, g):
    """[n, 6]: m_e, tau, A, B, C, amplitude."""
    u = torch.rand((n, 7), generator=g, dtype=torch.float64)
    e = torch.empty((n, 6), dtype=torch.float64)
    e[:, 0] = x0 + (x1 - x0) * u[:, 0]
    e[:, 1] = 0.2 + (tau_max - 0.2) * u[:, 1]
    e[:, 2] = 0.0 if op == "cmp" else 8e-4 * (u[:, 2] - 0.5)
    e[:, 3] = 0.0 if op == "cmp" else 2e-7 * (u[:, 3] - 0.5)
    e[:, 4] = 1.0 / (1500.0 + 2500.0 * u[:, 4]) ** 2
    e[:, 5] = (0.5 + 0.5 * u[:, 5]) * torch.where(u[:, 6] < 0.5, -1.0, 1.0)
    return e


def _record(mid, off, ns, dt, ev, snr, seed):
    """Ricker events on their traveltime surfaces plus noise: [n_tr, ns] float32. ev [n, 6], or
    [n, 6, n_tr] for events of their own on every trace; dt a number or [n_tr]."""
    n = torch.arange(ns, device=DEV, dtype=torch.float32)
    dt = dt if isinstance(dt, float) else dt[:, None]
    x = torch.zeros((mid.numel(), ns), device=DEV)
    for e in ev.to(device=DEV, dtype=torch.float32):
        dm = mid - e[0]
        T = (e[1] + e[2] * dm) ** 2 + e[3] * dm * dm + e[4] * off * off
        t = torch.where(T >= 0, T, torch.full_like(T, 1e6)).sqrt()
        a = (math.pi * 25.0 * (n * dt - t[:, None])) ** 2
        amp = e[5] if e[5].dim() == 0 else e[5][:, None]
        x += amp * (1.0 - 2.0 * a) * torch.exp(-a)
    g = torch.Generator(device=DEV).manual_seed(seed)
    x += torch.randn(x.shape, generator=g, device=DEV) / snr
    return x


def _inputs(case, seed):
    """(traces, mid, off, problem, cfg) of one case: what a program has read from its files."""
    g = torch.Generator().manual_seed(seed)
    if case["kind"] == "batched":
        return _batched_inputs(case, seed, g)
    op, ap, n_off, ns = case["op"], case["ap_half"], case["n_off"], case["ns"]
    n = case["n_cmp"] + (0 if case["whole"] else 2 * ap)
    first = 0 if case["whole"] else ap
    x = DCMP * torch.arange(n, dtype=torch.float32)
    mid = x.repeat_interleave(n_off).to(DEV)
    off = (DOFF * torch.arange(n_off, dtype=torch.float32)).repeat(n).to(DEV)
    ev = _events(case["events"], 0.0, float(x[-1]), 0.93 * (ns - 1) * case["dt"], op, g)
    traces = _record(mid, off, ns, case["dt"], ev, case["snr"], seed)
    offs = np.arange(n_off)
    if op == "fo":  # offsets within 1000 m of the section's
        offs = offs[np.abs(DOFF * offs - H0) <= 1000.0]
    per = []
    for c in range(first, first + case["n_cmp"]):
        rows = np.arange(max(0, c - ap), min(n - 1, c + ap) + 1)
        per.append((rows[:, None] * n_off + offs[None, :]).ravel())
    if case["n_points"]:  # points of their own midpoint near the CMP, one group each
        k = case["n_points"]
        it0 = torch.randint(0, ns, (k,), generator=g).numpy()
        m0 = (float(x[first]) + 250.0 * (torch.rand((k,), generator=g) - 0.5)).numpy()
        per, dom_group, grid = per * k, np.arange(k), (0, 0)
    else:
        it0 = np.tile(np.arange(ns), case["n_cmp"])
        m0 = x[first:first + case["n_cmp"]].numpy()
        dom_group, grid = np.repeat(np.arange(case["n_cmp"]), ns), (case["n_cmp"], ns)
    prob = _problem(op, case["w"], m0, np.full(len(per), case["dt"]), per, it0, dom_group, grid)
    return traces, mid, off, prob, _cfg(case, seed)


def _batched_inputs(case, seed, g):
    P = case["n_prob"]
    s = torch.Generator().manual_seed(P)  # the problems' sizes belong to the case
    ntr = torch.randint(case["ntr_lo"], case["ntr_hi"] + 1, (P,), generator=s)
    nsp = torch.randint(case["ns_lo"], case["ns_hi"] + 1, (P,), generator=s)
    dtp = torch.where(torch.rand(P, generator=s) < 0.5, 0.002, 0.004)
    ns, n = int(nsp.max()), int(ntr.sum())
    p = torch.arange(P).repeat_interleave(ntr)
    mid = DCMP * torch.randint(-10, 11, (n,), generator=g).float()
    off = DOFF * torch.randint(0, 48, (n,), generator=g).float()
    ev = torch.stack([_events(8, 0.0, 0.0, 1.9, "crs", g) for _ in range(P)])  # [P, 8, 6]
    traces = _record(mid.to(DEV), off.to(DEV), ns, dtp[p].to(DEV), ev[p].permute(1, 2, 0), 5.0,
                     seed)
    traces *= torch.arange(ns, device=DEV) < nsp[p].to(DEV)[:, None]
    at = np.concatenate([[0], np.cumsum(ntr.numpy())])
    per = [np.arange(at[k], at[k + 1]) for k in range(P)]
    it0 = np.concatenate([np.arange(int(k)) for k in nsp])
    prob = _problem("crs", case["w"], np.zeros(P), dtp.numpy(), per, it0,
                    np.repeat(np.arange(P), nsp.numpy()), (0, 0))
    return traces, mid.to(DEV), off.to(DEV), prob, _cfg(case, seed)


def _problem(op, w, m0, dt, per, it0, dom_group, grid):
    f, i = np.float32, np.int32
    return SimpleNamespace(
        op=OP[op], half_window=w, group_m0=np.asarray(m0, f), group_dt=np.asarray(dt, f),
        ap_ptr=np.concatenate([[0], np.cumsum([len(r) for r in per])]).astype(i),
        ap_idx=np.concatenate(per).astype(i), dom_it0=np.asarray(it0, i),
        dom_group=np.asarray(dom_group, i), n_m0=grid[0], n_t0=grid[1],
        group_h0=np.full(len(per), H0, f) if op == "fo" else None)


def _cfg(case, seed):
    return SimpleNamespace(np=case["np"], ng=case["ng"], F=0.5, CR=0.9, seed=seed,
                           lo=LO[case["op"]], hi=HI[case["op"]],
                           exch_every=case.get("exch", 0), polish_steps=case.get("polish", 0),
                           polish_lr=2e-4, adapt=case["adapt"])


def _theta(case, prob, seed):
    """[n_dom, P, D]: spread 1 is uniform in the bounds; less is a population around a centre
    that varies smoothly along the section, with its members within that share of the bounds."""
    op, P, s = case["op"], case["P"], case["spread"]
    lo = torch.tensor(LO[op], device=DEV, dtype=torch.float64)
    hi = torch.tensor(HI[op], device=DEV, dtype=torch.float64)
    g = torch.Generator(device=DEV).manual_seed(seed + 1)
    n_dom = prob.dom_it0.size
    u = torch.rand((n_dom, P, lo.numel()), generator=g, device=DEV, dtype=torch.float64)
    if s < 1:
        t = torch.as_tensor(prob.dom_it0, device=DEV).double() / max(1, case["ns"])
        m = torch.as_tensor(prob.dom_group, device=DEV).double()
        ph = 6.283 * torch.rand((2, lo.numel()), generator=g, device=DEV, dtype=torch.float64)
        c = 0.5 + 0.2 * torch.sin(5.0 * t[:, None] + ph[0]) + 0.2 * torch.sin(0.05 * m[:, None] + ph[1])
        u = (c[:, None, :] + s * (u - 0.5)).clamp(0.0, 1.0)
    return (lo + u * (hi - lo)).float().contiguous()


def prepare(case, seed):
    traces, mid, off, prob, cfg = _inputs(case, seed)
    search = case["kind"] in ("search", "batched", "ens")
    st = {"case": case, "ctx": tt.tt_ctx_create(traces, mid, off, prob, cfg if search else None,
                                                storage=case["storage"], device=DEV)}
    if not search:
        th = _theta(case, prob, seed)
        st["theta"] = (th[:, 0].contiguous() if case["kind"] == "stack" else
                       th.requires_grad_() if case["kind"] == "grad" else th)
    return st


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind in ("search", "batched"):
        return tt.tt_search(ctx)
    if kind == "ens":
        return tt.tt_ens_search(ctx, case["np"], case["ng"], case["np"], case["ng"],
                                case["n_skip"], case["n_cycle"], case["n_bucket"])
    if kind == "stack":
        return tt.tt_stack(ctx, state["theta"])
    if kind == "eval":
        return tt.tt_semblance_eval(ctx, state["theta"])
    theta = state["theta"]
    theta.grad = None
    S = tt.semblance(ctx, theta)
    S.sum().backward()
    return S.detach(), theta.grad


# ---- work ---------------------------------------------------------------------------------


def _sizes(case):
    """(trace samples, aperture entries, domains, sum of aperture sizes over domains)."""
    if case["kind"] == "batched":
        n = case["n_prob"]
        tr = n * 0.5 * (case["ntr_lo"] + case["ntr_hi"])
        nt = 0.5 * (case["ns_lo"] + case["ns_hi"])
        return tr * case["ns_hi"], tr, n * nt, tr * nt
    op, ap, ns = case["op"], case["ap_half"], case["ns"]
    offs = case["n_off"] if op != "fo" else sum(
        1 for k in range(case["n_off"]) if abs(DOFF * k - H0) <= 1000.0)
    n = case["n_cmp"] + (0 if case["whole"] else 2 * ap)
    if case["n_points"]:
        k = case["n_points"]
        return n * case["n_off"] * ns, k * offs, k, k * offs
    first = 0 if case["whole"] else ap
    ent = sum((min(n - 1, c + ap) - max(0, c - ap) + 1) * offs
              for c in range(first, first + case["n_cmp"]))
    return n * case["n_off"] * ns, ent, case["n_cmp"] * ns, ent * ns


def work(case):
    samples, entries, n_dom, sum_n = _sizes(case)
    D, K, kind = DIM[case["op"]], 2 * case["w"] + 1, case["kind"]
    pos = {"cmp": 5, "crs": 9, "fo": 15}[case["op"]]
    pair = pos + 7 * K  # traveltime, interpolation (3), stack (1), energy (2) and 1 weight a sample
    data = samples * (2 if case["storage"] == "bf16" else 4) + 12 * entries + 8 * n_dom
    if kind == "eval":
        return {"bytes": data + 4.0 * n_dom * case["P"] * (D + 1), "flops": sum_n * case["P"] * pair}
    if kind == "grad":  # the value, and the adjoint over the same windows
        return {"bytes": data + 4.0 * n_dom * case["P"] * (2 * D + 1),
                "flops": sum_n * case["P"] * (pair + 6 * K + 4 * D)}
    if kind == "stack":
        return {"bytes": data + 4.0 * n_dom * (D + 1), "flops": sum_n * (pos + 4)}
    out = 4.0 * n_dom * (D + 1)
    if kind == "ens":
        est = 1.0 / (case["n_skip"] + 1)
        per = case["np"] * (1 + case["ng"])
        stages = 1 + 2 * case["n_cycle"]
        calls = est * (per + (stages - 1) * (per - 1)) + stages * (1 - est)
    else:
        calls = case["np"] * (1 + case["ng"]) + (case.get("polish", 0) and case["polish"] + 1)
        if case.get("exch", 0):
            calls += 4 * (case["ng"] // case["exch"])
    return {"bytes": data + out, "flops": sum_n * calls * pair}


# ---- outputs in 64 bits ---------------------------------------------------------------------


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("eval", "grad", "stack"):
        return None
    traces, mid, off, prob, _ = _inputs(case, seed)
    if case["storage"] == "bf16":
        traces = traces.bfloat16().float()
    theta = _theta(case, prob, seed).double()
    n_dom, P, D = theta.shape
    w, ns = case["w"], case["ns"]
    pad = torch.nn.functional.pad(traces, (w + 2, 2 * w + 4))  # zero outside the record
    flat, pitch = pad.reshape(-1), pad.shape[1]
    S = torch.zeros((n_dom, P), device=DEV, dtype=torch.float64)
    G = torch.zeros((n_dom, P, D), device=DEV, dtype=torch.float64)
    out = torch.zeros((n_dom,), device=DEV, dtype=torch.float64)
    it0 = torch.as_tensor(prob.dom_it0, device=DEV).double()
    for grp in range(len(prob.group_m0)):
        rows = torch.as_tensor(prob.ap_idx[prob.ap_ptr[grp]:prob.ap_ptr[grp + 1]], device=DEV).long()
        dom = torch.as_tensor(np.nonzero(prob.dom_group == grp)[0], device=DEV)
        N, dt = rows.numel(), float(prob.group_dt[grp])
        dm = mid[rows].double() - float(prob.group_m0[grp])
        h = off[rows].double()
        dh = h - H0
        for q in torch.arange(dom.numel() * P, device=DEV).split(max(1, 40_000_000 // max(1, N))):
            d = dom[q // P]
            th = theta[d, q % P]
            t0 = (it0[d] * dt)[:, None]
            a = [th[:, k:k + 1] for k in range(D)]
            if case["op"] == "cmp":
                lin, T = t0, t0 * t0 + a[0] * h * h
                dT = (h * h,)
            elif case["op"] == "crs":
                lin = t0 + a[0] * dm
                T = lin * lin + a[1] * dm * dm + a[2] * h * h
                dT = (2 * lin * dm, dm * dm, h * h)
            else:
                lin = t0 + a[0] * dm + a[1] * dh
                T = lin * lin + a[2] * dm * dm + a[3] * dm * dh + a[4] * dh * dh
                dT = (2 * lin * dm, 2 * lin * dh, dm * dm, dm * dh, dh * dh)
            u = T.clamp(min=0).sqrt() / dt
            inside = (T >= 0) & (u < ns + w)
            u = torch.where(inside, u, torch.full_like(u, float(ns + w)))
            j = u.floor()
            f = u - j
            base = rows * pitch + (w + 2) + j.long()
            if kind == "stack":
                v = (1 - f) * flat[base].double() + f * flat[base + 1].double()
                out[d] = v.sum(1) / N
                continue
            E = torch.zeros(q.numel(), device=DEV, dtype=torch.float64)
            sk, lo = [], flat[base - w].double()
            ag = []
            for k in range(-w, w + 1):
                hi = flat[base + k + 1].double()
                v = torch.lerp(lo, hi, f)
                sk.append(v.sum(1))
                E += (v * v).sum(1)
                if kind == "grad":
                    ag.append((v, hi - lo))
                lo = hi
            Q = sum(s * s for s in sk)
            ok = E > 0
            s_ = torch.where(ok, Q / (N * E), torch.zeros_like(E))
            S[d, q % P] = s_
            if kind == "grad":
                al = torch.where(ok, 2 / (N * E), torch.zeros_like(E))
                be = torch.where(ok, 2 * s_ / E, torch.zeros_like(E))
                dS = sum((al * s)[:, None] * gk - be[:, None] * v * gk for s, (v, gk) in zip(sk, ag))
                c = torch.where(inside & (u > 0), dS / (2 * u * dt * dt), torch.zeros_like(u))
                for k in range(D):
                    G[d, q % P, k] = (c * dT[k]).sum(1)
    return out if kind == "stack" else S if kind == "eval" else (S, G)
