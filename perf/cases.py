"""Performance cases of the aggregate risk analysis library, through its public Python binding.

A case is a dict of plain values; `prepare` makes what a caller has in hand before the call (the
portfolio, the Year Event Table on the device, a plan, a server), `run` makes one pass, and `exact`
gives the same outputs in 64 bits with plain torch.  Losses are lognormal, event IDs uniform over
the catalogue, and every cover attaches at the 20th percentile of what it covers with a limit
amount of its 95th percentile, the rule of the synthetic workloads in `synth/`.

Kinds of cases:
  ylt       Portfolio.run_ylt and risk_metrics, the call a pricing or capital run makes
  oep       the occurrence basis: run_ylt with ARA_RUN_OEP and risk_metrics
  host      Portfolio.run_ylt_host on pinned host arrays
  metrics   risk_metrics of a book's YLT rows (PML, TVaR, mean)
  adjoint   Portfolio.adjoint: sensitivities of mean and TVaR, from the trial-major YET or from an
            event-major index that the caller keeps
  plan      BatchedPlan.launch: every layer of a book in one graph-captured pass
  serve     a burst of queries to a Server over a resident pool and YET
"""
import math

import numpy as np
import torch

import paper_1606_04473_gb300 as ara


def _case(name, kind, **kw):
    c = dict(name=name, kind=kind, catalogue=2_000_000, layers=1, pool=15, elts_lo=15, elts_hi=15, own_elts=False,
             nnz=20_000, f32=True, trials=100_000, events=1000, spread="poisson", regimes=False, index=False,
             n_rp=2, n_tvar=1, mean=False, queries=0)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest analysis: one layer over a small catalogue, a few trials (quick quotes)
        _case("ylt_tiny", "ylt", catalogue=10_000, pool=4, elts_lo=4, elts_hi=4, nnz=1000, f32=False, trials=1000,
              events=100),
        # an ordinary regional layer: FP64 losses, a catalogue whose hit bitmap fits on chip, ragged trials
        _case("ylt_regional", "ylt", catalogue=200_000, pool=30, elts_lo=30, elts_hi=30, nnz=10_000, f32=False,
              trials=30_011, events=800),
        # the headline: one layer of 15 ELTs, a million trials of 1,000 events
        _case("ylt_million", "ylt", trials=1_000_000, spread="fixed"),
        # a program of 16 layers with its aggregate regimes recorded (the forward of a sensitivity run)
        _case("ylt_program", "ylt", layers=16, pool=240, own_elts=True, trials=200_000, spread="fixed", regimes=True),
        # occurrence exceedance curve of one layer: six return periods, uneven trial lengths
        _case("oep_curve", "oep", catalogue=1_000_003, f32=False, trials=150_001, spread="uneven", n_rp=6, n_tvar=0),
        # the whole analysis from pinned host memory
        _case("host_staged", "host", trials=100_000),
        # reporting on a book: PML, TVaR and mean of 64 YLT rows
        _case("metrics_book", "metrics", layers=64, trials=200_000, n_rp=4, n_tvar=2, mean=True),
        # sensitivities of one layer
        _case("adjoint_layer", "adjoint", trials=300_007),
        # sensitivities of a program of 16 layers
        _case("adjoint_program", "adjoint", layers=16, pool=240, own_elts=True, trials=200_000, spread="fixed"),
        # sensitivities of a few layers that share ELTs, over an index of the YET kept by the caller
        _case("adjoint_indexed", "adjoint", layers=5, pool=60, elts_lo=5, elts_hi=20, trials=150_007, index=True),
        # a book of 64 layers in one pass, uneven trial lengths
        _case("plan_book", "plan", layers=64, pool=200, elts_lo=3, elts_hi=30, trials=200_000, spread="uneven"),
        # a burst of queries from several tenants on slices of a resident YET
        _case("serve_burst", "serve", layers=8, pool=120, elts_lo=5, elts_hi=20, trials=200_000, queries=12),
    ]


def draw(rng):
    log = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    kind = rng.choice(["ylt", "ylt", "ylt", "oep", "host", "metrics", "adjoint", "adjoint", "plan", "serve"])
    c = _case("", kind)
    del c["name"]
    c["catalogue"] = log(10_000, 2_500_000)
    c["nnz"] = min(log(500, 30_000), c["catalogue"] // 2)
    c["f32"] = rng.random() < 0.6
    c["spread"] = rng.choice(["fixed", "poisson", "uneven"])
    c["events"] = log(50, 1500)
    c["layers"] = {"oep": log(1, 3), "host": log(1, 3), "metrics": log(1, 100), "plan": log(2, 100),
                   "serve": log(1, 12)}.get(kind, log(1, 24))
    c["elts_lo"] = rng.randint(1, 8)
    c["elts_hi"] = rng.randint(c["elts_lo"], 30)
    c["pool"] = max(c["elts_hi"], log(4, 200))
    c["regimes"] = kind == "ylt" and rng.random() < 0.5
    c["index"] = kind == "adjoint" and rng.random() < 0.4
    c["mean"] = rng.random() < 0.4
    c["n_rp"], c["n_tvar"] = rng.randint(1, 6), rng.randint(0, 2)
    if kind == "oep":
        c["n_tvar"] = 0
    c["queries"] = rng.randint(2, 12) if kind == "serve" else 0
    # occurrences at most those of the listed cases, fewer the more layers read them
    most = 4e8 if kind in ("ylt", "oep") and c["layers"] == 1 else 1.5e8
    if kind == "ylt" and c["layers"] > 1:
        most = min(most, 2e9 / c["layers"])
    if kind == "metrics":
        c["trials"] = log(1000, 10_000_000 // c["layers"])
    else:
        c["trials"] = log(500, max(1000, min(1_000_000, most / c["events"])))
    return c


# ------------------------------------------------------------------------------------------------
# Inputs
# ------------------------------------------------------------------------------------------------
RETURN_PERIODS = [100.0, 250.0, 50.0, 10.0, 200.0, 20.0]
LEVELS = [0.99, 0.95]
ADJOINT_LEVEL = 0.99


def _metrics_args(c):
    return RETURN_PERIODS[:c["n_rp"]], LEVELS[:c["n_tvar"]]


def _counts(c, gen):
    n, ev = c["trials"], float(c["events"])
    if c["spread"] == "fixed":
        return torch.full((n,), int(ev), dtype=torch.int64, device="cuda")
    lam = torch.full((n,), ev, dtype=torch.float64, device="cuda")
    if c["spread"] == "uneven":   # per-trial mean uniform on [0.2, 2] x events
        lam *= 0.2 + 1.8 * torch.rand(n, dtype=torch.float64, device="cuda", generator=gen)
    return torch.poisson(lam, generator=gen).to(torch.int64)


def _yet(c, seed):
    """Trial offsets (int64) and event IDs (int32) on the device."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed * 1009 + 7)
    off = torch.zeros(c["trials"] + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(_counts(c, gen), 0, out=off[1:])
    ids = torch.randint(0, c["catalogue"], (int(off[-1]),), dtype=torch.int32, device="cuda", generator=gen)
    return off, ids


def _structure(c):
    """Generator of what does not change with the seed: which ELTs the layers hold."""
    return np.random.default_rng([c["layers"], c["pool"], c["elts_lo"], c["elts_hi"], c["trials"]])


def _pick_elts(c, rng):
    k = int(rng.integers(c["elts_lo"], c["elts_hi"] + 1))
    return sorted(int(j) for j in rng.choice(c["pool"], size=k, replace=False))


class _Tables:
    """The tables of a portfolio: ELTs and layers with their terms."""


def _percentiles(x, ps):
    s = torch.sort(x).values
    n = s.numel()
    if n == 0:
        return [0.0] * len(ps)
    return [float(s[min(n - 1, int(p * n))]) for p in ps]


def _tables(c, seed):
    rng = np.random.default_rng(seed * 7919 + 13)
    C, t = c["catalogue"], _Tables()
    t.catalogue, t.losses_f32 = C, bool(c["f32"])
    t.elt_ids, t.elt_losses = [], []
    for _ in range(c["pool"]):
        t.elt_ids.append(rng.choice(C, size=c["nnz"], replace=False, shuffle=False).astype(np.int32))
        x = np.exp(11.0 + 2.0 * rng.standard_normal(c["nnz"]))
        t.elt_losses.append(x.astype(np.float32).astype(np.float64) if c["f32"] else x)
    p = np.percentile(np.stack(t.elt_losses), [20.0, 50.0, 95.0], axis=1)
    t.elt_ret, t.elt_p50, t.elt_lim = p[0], p[1], p[2]
    t.elt_p95 = p[2]
    t.layer_elts, pick = [], _structure(c)
    for i in range(c["layers"] if c["kind"] != "serve" else 0):
        if c["own_elts"]:
            t.layer_elts.append(list(range(15 * i, 15 * i + 15)))
        else:
            t.layer_elts.append(_pick_elts(c, pick))
    # occurrence and aggregate covers by the percentile rule; the trial sum's percentiles from its
    # mean and variance
    dev = _device_elts(t)
    occ_r, occ_l, agg_r, agg_l = [], [], [], []
    ev = float(c["events"]) * (1.1 if c["spread"] == "uneven" else 1.0)
    var_n = {"fixed": 0.0, "poisson": ev, "uneven": ev + (1.8 * c["events"]) ** 2 / 12.0}[c["spread"]]
    for l in t.layer_elts:
        s = _event_sums(t, dev, l)
        r, lim = _percentiles(s[s > 0], [0.2, 0.95])
        o = (s - r).clamp(min=0.0, max=lim)
        m, v = float(o.mean()), float(o.var())
        mean, sd = ev * m, math.sqrt(ev * v + var_n * m * m)
        occ_r.append(r)
        occ_l.append(lim)
        if c["kind"] == "plan":   # a book's covers differ around the rule
            f = rng.uniform(0.5, 1.5, 2)
        else:
            f = (1.0, 1.0)
        agg_r.append(max(0.0, mean - 0.84 * sd) * f[0])
        agg_l.append((mean + 1.64 * sd) * f[1])
    t.occ_ret, t.occ_lim, t.agg_ret, t.agg_lim = map(np.asarray, (occ_r, occ_l, agg_r, agg_l))
    return t


def _queries(c, t, seed):
    """Queries of several tenants: layers of pool ELTs on contiguous slices of the trials."""
    rng, pick = np.random.default_rng(seed * 31 + 5), _structure(c)
    out, n = [], c["trials"]
    for k in range(c["queries"]):
        layers = [_pick_elts(c, pick) for _ in range(int(pick.integers(1, c["layers"] + 1)))]
        w = int(rng.integers(max(1, n // 4), n + 1))
        b = int(rng.integers(0, n - w + 1))
        out.append(dict(layer_elts=layers,
                        occ_ret=[float(t.elt_p50[l].max()) for l in layers],
                        occ_lim=[float(t.elt_p95[l].sum()) for l in layers],
                        agg_ret=[float(10.0 * t.elt_p50[l].sum()) for l in layers],
                        agg_lim=[float(200.0 * t.elt_p95[l].sum()) for l in layers],
                        trials=(b, b + w), return_periods=RETURN_PERIODS[:2], tvar_levels=LEVELS[:1],
                        want_mean=bool(c["mean"]), want_adjoint=k % 5 == 4, adjoint_level=ADJOINT_LEVEL, tenant=k))
    return out


def _book_ylt(c, seed):
    """YLT rows as aggregate covers leave them: a fifth of the years zero, a few at the limit."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed * 1013 + 3)
    z = torch.randn((c["layers"], c["trials"]), dtype=torch.float64, device="cuda", generator=gen)
    scale = torch.exp(2.0 * torch.randn((c["layers"], 1), dtype=torch.float64, device="cuda", generator=gen) + 15.0)
    return ((z + 0.84).clamp(min=0.0, max=4.0) * scale).contiguous()


def prepare(case, seed):
    c = case
    if c["kind"] == "metrics":
        return dict(case=c, ylt=_book_ylt(c, seed))
    t = _tables(c, seed)
    off, ids = _yet(c, seed)
    st = dict(case=c, off=off, ids=ids, pf=ara.Portfolio.from_tables(t))
    n = c["trials"]
    if c["kind"] == "ylt" and c["regimes"]:
        st["reg"] = torch.empty((c["layers"], n), dtype=torch.uint8, device="cuda")
    if c["kind"] == "host":
        st["h_off"] = torch.empty(off.numel(), dtype=torch.int64, pin_memory=True).copy_(off).numpy()
        st["h_ids"] = torch.empty(ids.numel(), dtype=torch.int32, pin_memory=True).copy_(ids).numpy()
        st["h_out"] = torch.empty((c["layers"], n), dtype=torch.float64, pin_memory=True).numpy()
        del st["off"], st["ids"]
    if c["kind"] == "adjoint":
        st["reg"] = torch.empty((c["layers"], n), dtype=torch.uint8, device="cuda")
        st["ylt"] = st["pf"].run_ylt(off, ids, regimes=st["reg"])
        st["pf"].check()
        if c["index"]:
            st["index"] = st["pf"].yet_index(off, ids)
    if c["kind"] == "plan":
        st["reg"] = torch.empty((c["layers"], n), dtype=torch.uint8, device="cuda")
        st["plan"] = ara.BatchedPlan(st["pf"], off, ids, regimes=st["reg"])
    if c["kind"] == "serve":
        st["queries"] = _queries(c, t, seed)
        st["server"] = ara.Server(st["pf"], off, ids)
        st["server"].set_adjoint_index(True)
    torch.cuda.synchronize()
    return st


def run(state):
    c = state["case"]
    kind = c["kind"]
    rps, levels = _metrics_args(c)
    if kind == "metrics":
        r = ara.risk_metrics(state["ylt"], rps, levels, want_mean=c["mean"])
        return dict(zip(("pml", "tvar", "mean"), r))
    if kind in ("ylt", "oep"):
        y = state["pf"].run_ylt(state["off"], state["ids"], regimes=state.get("reg"),
                                flags=ara.ARA_RUN_OEP if kind == "oep" else 0)
        r = ara.risk_metrics(y, rps, levels, want_mean=c["mean"])
        out = dict(zip(("pml", "tvar", "mean"), r))
        out["ylt"] = y
        if "reg" in state:
            out["regimes"] = state["reg"]
        return out
    if kind == "host":
        r = state["pf"].run_ylt_host(state["h_off"], state["h_ids"], out=state["h_out"], return_periods=rps,
                                     tvar_levels=levels, want_mean=c["mean"])
        return dict(zip(("ylt", "pml", "tvar", "mean"), r))
    if kind == "adjoint":
        if c["index"]:
            return state["pf"].adjoint(None, None, state["ylt"], state["reg"], ADJOINT_LEVEL, index=state["index"])
        return state["pf"].adjoint(state["off"], state["ids"], state["ylt"], state["reg"], ADJOINT_LEVEL)
    if kind == "plan":
        return dict(ylt=state["plan"].launch(), regimes=state["reg"])
    srv = state["server"]
    tickets = [srv.submit(**q) for q in state["queries"]]
    out = []
    for k in tickets:
        r = srv.wait(k)
        out.append({x: r[x] for x in ("pml", "tvar", "mean", "grad_layer") if r[x] is not None})
    return out


def work(case):
    """Bytes: the YET (or its index), the ELT records and the outputs, once each.  Operations: one
    addition per occurrence and layer with a loss for it, and the terms of every record and year."""
    c = case
    n, L = c["trials"], max(1, c["layers"])
    ev = n * c["events"] * (1.1 if c["spread"] == "uneven" else 1.0)
    rec = 8 if c["f32"] else 12
    if c["kind"] == "metrics":
        return {"bytes": 8.0 * n * L, "flops": float(n * L)}
    elts = 15.0 if c["own_elts"] else (c["elts_lo"] + c["elts_hi"]) / 2.0
    hits = 1.0 - math.exp(-elts * c["nnz"] / c["catalogue"])   # share of events with a loss in a layer
    if c["kind"] == "serve":
        L = c["queries"] * (1 + c["layers"]) / 2.0
        used = float(c["pool"])
        return {"bytes": 4.0 * ev + 8.0 * n + rec * used * c["nnz"], "flops": 0.62 * ev * L * hits}
    used = min(float(c["pool"]), elts * L)
    b = 8.0 * (n + 1) + rec * used * c["nnz"]
    if c["kind"] == "adjoint":
        b += (2.0 if c["index"] else 4.0) * ev + 9.0 * n * L + 16.0 * elts * L * c["nnz"]
    else:
        b += 4.0 * ev + (9.0 if c["regimes"] or c["kind"] == "plan" else 8.0) * n * L
    return {"bytes": b, "flops": ev * L * hits + 3.0 * elts * L * c["nnz"] + 3.0 * n * L}


# ------------------------------------------------------------------------------------------------
# The same outputs in 64 bits, with plain torch
# ------------------------------------------------------------------------------------------------
def _device_elts(t):
    return [(torch.from_numpy(i).cuda().long(), torch.from_numpy(x).cuda()) for i, x in zip(t.elt_ids, t.elt_losses)]


def _event_sums(t, dev, layer):
    s = torch.zeros(t.catalogue, dtype=torch.float64, device="cuda")
    for j in layer:
        i, x = dev[j]
        s[i] += (x - float(t.elt_ret[j])).clamp(min=0.0, max=float(t.elt_lim[j]))
    return s


def _chunks(off, most=1 << 27):
    h = off.cpu().numpy()
    a, n = 0, h.size - 1
    while a < n:
        b = max(a + 1, int(np.searchsorted(h, h[a] + most, side="right")) - 1)
        b = min(b, n)
        yield a, b, int(h[a]), int(h[b])
        a = b


def _trial_reduce(off, ids, o, how):
    out = torch.zeros(off.numel() - 1, dtype=torch.float64, device="cuda")
    for a, b, e0, e1 in _chunks(off):
        if e1 > e0:
            out[a:b] = torch.segment_reduce(o[ids[e0:e1].long()], how, lengths=off[a + 1:b + 1] - off[a:b],
                                            unsafe=True, initial=0.0)
    return out


def _count(x):
    """The whole number that x is up to rounding, else the next one above."""
    r = round(x)
    return r if abs(x - r) <= 1e-9 * max(1.0, abs(x)) else math.ceil(x)


def _metrics(y, rps, levels, mean):
    n = y.shape[1]
    s = torch.sort(y, dim=1, descending=True).values
    pml = torch.stack([s[:, _count(n / r) - 1] for r in rps], 1) if rps else y.new_zeros((y.shape[0], 0))
    tv = [s[:, :_count(n * (1.0 - p))].mean(1) for p in levels]
    tvar = torch.stack(tv, 1) if tv else y.new_zeros((y.shape[0], 0))
    out = dict(pml=pml.cpu().numpy(), tvar=tvar.cpu().numpy())
    if mean:
        out["mean"] = y.mean(1).cpu().numpy()
    return out


def _layer_grads(t, dev, layer, terms, off, ids, level):
    """Gradients of one layer's mean and TVaR: (elt [2, k, 2], layer [2, 4], loss per ELT, tie)."""
    occ_r, occ_l, agg_r, agg_l = terms
    s = _event_sums(t, dev, layer)
    ex = s - occ_r
    r1, r2 = (ex > 0) & (ex < occ_l), ex > occ_l
    S = _trial_reduce(off, ids, ex.clamp(min=0.0, max=occ_l), "sum")
    d = S - agg_r
    inner, above = (d > 0) & (d < agg_l), d > agg_l
    y = d.clamp(min=0.0, max=agg_l)
    n = y.numel()
    m = _count(n * (1.0 - level))
    v = torch.sort(y, descending=True).values[m - 1]
    gt, eq = int((y > v).sum()), int((y == v).sum())
    w = torch.stack([torch.full_like(y, 1.0 / n), ((y > v).double() + (m - gt) / eq * (y == v).double()) / m])
    c = torch.zeros((2, t.catalogue), dtype=torch.float64, device="cuda")
    cnt = off[1:] - off[:-1]
    for a, b, e0, e1 in _chunks(off, 1 << 25):
        if e1 > e0:
            e = ids[e0:e1].long()
            for k in range(2):
                c[k].index_add_(0, e, (w[k, a:b] * inner[a:b]).repeat_interleave(cnt[a:b]))
    g_layer = torch.stack([-(c * r1).sum(1), (c * r2).sum(1), -(w * inner).sum(1), (w * above).sum(1)], 1)
    g_elt, g_loss = [], []
    for j in layer:
        i, x = dev[j]
        dx, lim = x - float(t.elt_ret[j]), float(t.elt_lim[j])
        g = c[:, i] * r1[i]
        j1, j2 = (dx > 0) & (dx < lim), dx > lim
        g_loss.append(g * j1)
        g_elt.append(torch.stack([-(g * j1).sum(1), (g * j2).sum(1)], 1))
    return torch.stack(g_elt, 1), g_layer, torch.cat(g_loss, 1), int(gt + eq > m)


def exact(case, seed):
    c = case
    rps, levels = _metrics_args(c)
    if c["kind"] == "metrics":
        return _metrics(_book_ylt(c, seed), rps, levels, c["mean"])
    t = _tables(c, seed)
    off, ids = _yet(c, seed)
    dev = _device_elts(t)
    if c["kind"] == "serve":
        out = []
        for q in _queries(c, t, seed):
            b, e = q["trials"]
            so = off[b:e + 1]
            si = ids[int(so[0]):int(so[-1])]
            so = so - so[0]
            terms = list(zip(q["occ_ret"], q["occ_lim"], q["agg_ret"], q["agg_lim"]))
            y = torch.stack([(_trial_reduce(so, si, (_event_sums(t, dev, l) - r).clamp(min=0.0, max=x), "sum") - p)
                             .clamp(min=0.0, max=z) for l, (r, x, p, z) in zip(q["layer_elts"], terms)])
            one = _metrics(y, q["return_periods"], q["tvar_levels"], q["want_mean"])
            if q["want_adjoint"]:
                g = [_layer_grads(t, dev, l, k, so, si, ADJOINT_LEVEL)[1] for l, k in zip(q["layer_elts"], terms)]
                one["grad_layer"] = torch.stack(g, 1).cpu().numpy()
            out.append(one)
        return out
    terms = list(zip(t.occ_ret, t.occ_lim, t.agg_ret, t.agg_lim))
    if c["kind"] == "adjoint":
        g = [_layer_grads(t, dev, l, k, off, ids, ADJOINT_LEVEL) for l, k in zip(t.layer_elts, terms)]
        return dict(elt=torch.cat([x[0] for x in g], 1), layer=torch.stack([x[1] for x in g], 1),
                    loss=torch.cat([x[2] for x in g], 1), ties=np.array([x[3] for x in g], dtype=np.int32))
    y = torch.empty((c["layers"], c["trials"]), dtype=torch.float64, device="cuda")
    for i, (l, (r, x, p, z)) in enumerate(zip(t.layer_elts, terms)):
        o = (_event_sums(t, dev, l) - r).clamp(min=0.0, max=x)
        if c["kind"] == "oep":
            y[i] = _trial_reduce(off, ids, o, "max")
        else:
            y[i] = (_trial_reduce(off, ids, o, "sum") - p).clamp(min=0.0, max=z)
    if c["kind"] == "plan":
        return dict(ylt=y, regimes=None)
    out = _metrics(y, rps, levels, c["mean"])
    out["ylt"] = y.cpu().numpy() if c["kind"] == "host" else y
    if c["kind"] == "ylt" and c["regimes"]:
        out["regimes"] = None
    return out
