"""Timed cases: what a user of this framework has it do, each through its
public entry points (api.py, serve.py, calib.py).

The fit.  A trigger node hands over batches of events and wants one record per
road back.  Batches run from a single event, where latency is all that counts,
to a few thousand; roads run from two hits a layer to sixteen.  The workloads
are the ones of synth.SPECS; `via` says how the batch gets to the GPU:
  fused   one svt_run call on a batch in device memory (FusedPath)
  graph   the same sequence replayed from a CUDA graph with the batch's sizes
          read on the device (GraphPath)
  noalloc svt_run_noalloc, for callers that own no device memory
  host    batches in pinned host memory, records back in host memory, two
          batches in turn on two streams (StreamingRunner)
  serve   single events submitted to the continuous-batching server (Server)
  plain   the per-stage calls, every intermediate kept (PlainPath)

The calibration.  Tracks with known parameters improve the fit constants:
  prepare the tracks put in sector order (CalibData), once per track set
  loss    the loss and its gradient with respect to the constants
  eval    the loss alone, as for a validation set
  monitor the loss, its gradient and every track's fitted parameters
  fit     the fitted parameters, and the gradient of a loss the user has of
          their own on them
"""
import functools
import math

import numpy as np
import torch

from paper_1311_0380_gb300 import api, calib, serve, synth

N_SECTORS = 512


def _fit(name, spec, events, via="fused", sched=(0, 0, 0, 0, 0, 0), max_comb=262144,
         min_layers=5, cut=99):
    return {"name": name, "kind": "fit", "spec": spec, "events": events, "via": via,
            "warps": sched[0], "bps": sched[1], "rows": sched[2], "chunk": sched[3],
            "small": sched[4], "pair": sched[5], "max_comb": max_comb,
            "min_layers": min_layers, "cut": cut}


def _calib(name, what, tracks, sectors=N_SECTORS):
    return {"name": name, "kind": "calib", "what": what, "tracks": tracks, "sectors": sectors}


# the schedules svt_autotune picks on this GPU for these shapes
TUNED_SCALED = (16, 0, 256, 4, 4096, 0)
TUNED_PAPER_SMALL = (8, 0, 16, 8, 4096, 3)
TUNED_PAPER_LARGE = (8, 0, 16, 16, 4096, 3)
TUNED_SERVE = (0, 0, 0, 1, 0, 0)


def listed():
    return [
        # one trigger event of the paper's shape (32 roads of 64 combinations): pure latency
        _fit("paper_1", "paper", 1, sched=TUNED_PAPER_SMALL),
        # the paper's largest batch, 3000 such events
        _fit("paper_3000", "paper", 3000, sched=TUNED_PAPER_LARGE),
        # a small batch of mixed roads as a first-time user runs it (default schedule)
        _fit("scaled_100", "scaled", 100),
        # the benchmark's headline batch in its tuned schedule
        _fit("scaled_3000", "scaled", 3000, sched=TUNED_SCALED),
        # crowded, uneven events (1..2048 roads, up to 16 hits a layer) replayed from a graph
        _fit("uneven_graph_512", "uneven", 512, via="graph", sched=TUNED_SERVE, max_comb=4096),
        # roads whose last two layers come in track-trigger pairs
        _fit("xft_1000", "xft", 1000),
        # the trigger node's loop: batches in host memory, copies included
        _fit("host_scaled_1000", "scaled", 1000, via="host", sched=TUNED_SCALED),
        # a burst of single events through the server
        _fit("serve_uneven_64", "uneven", 64, via="serve", sched=TUNED_SERVE, max_comb=4096),
        # the per-stage calls, every combination's fit kept
        _fit("plain_scaled_200", "scaled", 200, via="plain"),
        # a calibration set put in order
        _calib("calib_prepare_4m", "prepare", 4_000_000),
        # one optimiser step's loss and gradient on an ordinary calibration set
        _calib("calib_loss_1m", "loss", 1_000_000),
        # fitted parameters and a user's own loss on them, a large set
        _calib("calib_fit_16m", "fit", 16_000_003),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    if rng.random() < 0.3:
        what = rng.choice(["prepare", "loss", "eval", "monitor", "fit"])
        return {k: v for k, v in _calib("", what, _log_int(rng, 20_000, 16_000_003),
                                        rng.choice([64, 512, 337])).items() if k != "name"}
    spec = rng.choice(["small", "scaled", "uneven", "paper", "xft"])
    via = rng.choice(["fused", "fused", "graph", "noalloc", "host", "serve", "plain"])
    most = {"small": 3000, "scaled": 3000, "uneven": 512, "paper": 3000, "xft": 3000}[spec]
    most = min(most, {"noalloc": 64 if spec == "uneven" else 1000,
                      "host": 256 if spec == "uneven" else 1000, "serve": 64,
                      "plain": 3 if spec == "uneven" else 200}.get(via, most))
    if spec in ("paper", "small") and via != "plain":
        sched = rng.choice([(0,) * 6, TUNED_PAPER_SMALL, TUNED_PAPER_LARGE, (8, 0, 16, 32, 4096, 3),
                            (0, 0, 0, 8, 0, 1), (0, 0, 0, 8, 0, 2)])
    else:
        sched = rng.choice([(0,) * 6, TUNED_SCALED, TUNED_SERVE])
    max_comb = 4096 if spec == "uneven" else rng.choice([262144, 262144, 1000])
    case = _fit("", spec, _log_int(rng, 1, most), via, sched, max_comb,
                rng.choice([5, 5, 6]), rng.choice([99, 99, 90]))
    del case["name"]
    return case


# ------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=4)
def _constants(n_sectors):
    return synth.make_constants(n_sectors)


def _batch(case, seed):
    spec = synth.SPECS[case["spec"]]
    consts = _constants(spec.n_sectors)
    b = synth.make_batch(spec, case["events"], consts, seed=1 + seed)
    # the 99 % (or a tighter 90 %) point of a true track's chi-square
    cut = consts.chi2_cut_99 if case["cut"] == 99 else int(consts.chi2_cut_99 * 6.251 / 11.345)
    return spec, consts, b, cut


def _road_cap(case):
    """Roads a program sizes its buffers for: six standard deviations above
    what the workload's events hold on average."""
    spec = synth.SPECS[case["spec"]]
    sd = {"const": 0.0, "poisson": spec.roads[1] ** 0.5, "loguniform": 0.22 * spec.roads[1]}
    e = case["events"]
    return int(e * _mean_shape(case)[0] + 6 * sd[spec.roads[0]] * e ** 0.5) + 64


def _comb_cap(case):
    """The same for combinations (the scatter of the uncapped product of the
    layers' hits; no road has more than 16 ** 6)."""
    roads = _road_cap(case)
    worst = min(case["max_comb"], 16 ** 6)
    return min(roads * worst, int(roads * _mean_shape(case)[2] + 20000 * roads ** 0.5))


def _prepare_fit(case, seed):
    spec, consts, b, cut = _batch(case, seed)
    cfg = api.config(consts.oshift, consts.qshift, cut, case["max_comb"], case["min_layers"],
                     spec.n_sectors, 1 if spec.xft else 0)
    dc = api.DeviceConstants.from_numpy(consts.F, consts.q, cfg)
    s = [case[k] for k in ("warps", "bps", "rows", "chunk", "small", "pair")]
    sched = api.schedule(*s) if any(s) else None
    nw, ne, cap = len(b.words), b.n_events, _road_cap(case)
    st = {"via": case["via"], "nw": nw, "ne": ne}
    if case["via"] == "host":
        _, _, b2, _ = _batch(case, seed + 7919)
        r = api.StreamingRunner(max(nw, len(b2.words)), ne, cap, dc, sched)
        for h in r.h_out:
            h.zero_()
        st.update(runner=r, batches=[api.HostRunner.pin_batch(x.words, x.event_off)
                                     for x in (b, b2)])
        return st
    if case["via"] == "serve":
        srv = serve.Server(dc, n_slots=4, max_words=1 << 22, max_events=256, max_roads=1 << 17,
                           sched=sched, small_batch_events=4, small_blocks_per_sm=1)
        pool = serve.pinned_pool(b.words)
        off = b.event_off.astype(np.int64)
        roads = np.zeros(ne + 1, np.int64)
        np.cumsum(b.n_roads, out=roads[1:])
        rec = np.zeros((cap, 6), np.uint32)
        st.update(srv=srv, pool=pool, rec=rec,
                  events=[(pool[off[e]: off[e + 1]], e, rec[roads[e]: roads[e + 1]])
                          for e in range(ne)])
        return st
    st.update(words=api.to_device_u32(b.words), off=api.to_device_u64(b.event_off))
    if case["via"] == "plain":
        p = st["path"] = api.PlainPath(nw, ne, cap, _comb_cap(case), dc)
        for t in (p.out, p.comb_off, p.comb_road, p.comb_hits, p.fit_chi2, p.fit_par):
            t.zero_()
        return st
    st["path"] = api.FusedPath(nw, ne, cap, dc, sched)
    st["path"].out.zero_()
    if case["via"] == "graph":
        st["graph"] = api.GraphPath(st["path"], st["words"], st["off"])
        st["graph"].set_sizes(nw, ne)
    return st


def _tracks(case, seed):
    """Calibration tracks made on the GPU by the recipe of synth.make_calib."""
    S, n = case["sectors"], case["tracks"]
    c = _constants(S)
    g = torch.Generator(device="cuda").manual_seed(1 + seed)
    rnd = lambda *s: torch.rand(*s, generator=g, device="cuda")
    dev = lambda a: torch.as_tensor(a, device="cuda", dtype=torch.float32)
    sector = torch.randint(0, S, (n,), generator=g, device="cuda", dtype=torch.int32)
    d0 = (2 * rnd(n) - 1) * synth.D0_MAX_CM
    dphi = (rnd(n) - 0.5) * c.geometry.sector_width
    pt = synth.PT_MIN + (synth.PT_MAX - synth.PT_MIN) * rnd(n)
    curv = torch.where(rnd(n) < 0.5, -1.0, 1.0) * 0.003 * synth.B_TESLA / pt / 2.0
    A, x0 = synth.design(c.geometry, np.arange(S))
    A, x0, sl = dev(A), dev(x0), sector.long()
    x = x0[sl] + torch.randn(n, 6, generator=g, device="cuda") * dev(synth.SIGMA_LSB)
    for k, p in enumerate((d0, dphi, curv)):
        x += A[:, :, k][sl] * p[:, None]
    x = x.clamp_(0.0, float(synth.COORD_MAX))
    theta = torch.stack([d0, dphi, curv], 1) / dev(c.unit)
    rng = np.random.default_rng([seed, 0xCA])
    F = c.F[:, 63] / 2.0 ** c.oshift
    q = c.q[:, 63] * 2.0 ** (c.qshift - c.oshift)
    F = dev(F * (1.0 + 0.02 * rng.normal(size=F.shape)))
    q = dev(q + 0.02 * np.abs(q).mean() * rng.normal(size=q.shape))
    gy = torch.randn(n, 6, generator=g, device="cuda") if case["what"] == "fit" else None
    return x, sector, theta, 1.0 / theta.var(0), F, q, gy


def _prepare_calib(case, seed):
    x, sector, theta, w, F, q, gy = _tracks(case, seed)
    st = {"what": case["what"], "sectors": case["sectors"]}
    if case["what"] == "prepare":
        st.update(x=x, sector=sector, theta=theta, w=w)
        return st
    st.update(data=calib.CalibData(x, sector, theta, case["sectors"], w), gy=gy,
              F=F.requires_grad_(), q=q.requires_grad_())
    return st


def prepare(case, seed):
    return (_prepare_fit if case["kind"] == "fit" else _prepare_calib)(case, seed)


# ------------------------------------------------------------------ one pass
def _run_fit(st):
    via = st["via"]
    if via == "host":
        r = st["runner"]
        for words, off in st["batches"]:
            r.submit(words, off)
        r.wait()
        return {"records": r.h_out, "status": r.h_status}
    if via == "serve":
        srv, left = st["srv"], len(st["events"])
        for words, tag, rec in st["events"]:
            srv.submit(words, tag, rec)
        status = np.zeros(left, np.uint64)
        while left:
            for r in srv.poll(wait_us=10000):
                status[r.tag] = r.status
                left -= 1
        return {"records": st["rec"], "status": status}
    p = st["path"]
    if via == "plain":
        p.run(st["words"], st["nw"], st["off"], st["ne"])
        return {"records": p.out, "event_road": p.event_road, "n_roads": p.n_roads,
                "n_combs": p.n_combs, "comb_off": p.comb_off, "comb_road": p.comb_road,
                "comb_hits": p.comb_hits, "chi2": p.fit_chi2, "par": p.fit_par,
                "status": p.status}
    if via == "graph":
        st["graph"].launch()
    elif via == "noalloc":
        c = p.consts
        api.svt_run_noalloc(st["words"], st["nw"], st["off"], st["ne"], c.F, c.q, c.cfg,
                            p.road_cap, p.out, p.event_road, p.counts, p.status, p.sched)
    else:
        p.run(st["words"], st["nw"], st["off"], st["ne"])
    return {"records": p.out, "event_road": p.event_road, "counts": p.counts, "status": p.status}


def _run_calib(st):
    what = st["what"]
    if what == "prepare":
        d = calib.CalibData(st["x"], st["sector"], st["theta"], st["sectors"], st["w"])
        return {"perm": d.perm, "x": d.x, "theta": d.theta}
    F, q, data = st["F"], st["q"], st["data"]
    F.grad = q.grad = None
    if what == "eval":
        with torch.no_grad():
            return {"loss": calib.calib_loss(F, q, data)}
    if what == "fit":
        y = calib.fit_fp32(F, q, data)
        y.backward(st["gy"])
        return {"y": y.detach(), "dF": F.grad, "dq": q.grad}
    if what == "monitor":
        loss, y = calib.calib_loss_and_fit(F, q, data)
        loss.backward()
        return {"loss": loss.detach(), "y": y, "dF": F.grad, "dq": q.grad}
    loss = calib.calib_loss(F, q, data)
    loss.backward()
    return {"loss": loss.detach(), "dF": F.grad, "dq": q.grad}


def run(state):
    return _run_fit(state) if "via" in state else _run_calib(state)


# ------------------------------------------------------------------ necessary work
def _mean_shape(case):
    """Expected roads per event, hits per road and evaluated combinations per road."""
    spec = synth.SPECS[case["spec"]]
    kind = spec.roads[0]
    roads = (spec.roads[1] if kind in ("const", "poisson")
             else spec.roads[1] / math.log(spec.roads[1] + 1.0))
    if spec.hits[0] == "const":
        p = {spec.hits[1]: 1.0}
    elif spec.hits[0] == "uniform":
        lo, hi = spec.hits[1:]
        p = {n: 1.0 / (hi - lo + 1) for n in range(lo, hi + 1)}
    else:
        g, cap = spec.hits[1:]
        p = {n: g * (1 - g) ** (n - 1) for n in range(1, cap)}
        p[cap] = (1 - g) ** (cap - 1)
    hits = 6 * sum(n * w for n, w in p.items())
    prod = {1: 1.0}   # distribution of the product over the layers
    for _ in range(5 if spec.xft else 6):
        nxt = {}
        for c, w in prod.items():
            for n, v in p.items():
                nxt[c * n] = nxt.get(c * n, 0.0) + w * v
        prod = nxt
    return roads, hits, sum(min(c, case["max_comb"]) * w for c, w in prod.items())


def work(case):
    if case["kind"] == "calib":
        n, S = case["tracks"], case["sectors"]
        consts = 4 * 42 * S
        return {
            # sector, x, theta in; permutation, x, theta out
            "prepare": {"bytes": n * (4 + 36 + 4 + 36), "flops": 0},
            "eval": {"bytes": n * 36 + consts, "flops": n * (72 + 15)},
            # y = F x + q, the residuals, then the outer product with x
            "loss": {"bytes": n * 36 + 2 * consts, "flops": n * (72 + 15 + 78)},
            "monitor": {"bytes": n * 60 + 2 * consts, "flops": n * (72 + 15 + 78)},
            # x in, y out; x again and the gradient of y in
            "fit": {"bytes": n * (48 + 48) + 2 * consts, "flops": n * (72 + 78)},
        }[case["what"]]
    roads, hits, combs = _mean_shape(case)
    e = case["events"] * (2 if case["via"] == "host" else 1)
    # words and offsets in, one record per road and the event table out
    nbytes = e * (8 + 4 + 4 * (1 + roads * (1 + hits)) + 24 * roads)
    if case["via"] == "plain":
        # combinations written, read by the fit, its results written, chi2 read
        nbytes += e * roads * combs * (8 + 8 + 16 + 4)
    # three sums of a prefix and a suffix term, three squares summed, one compare
    return {"bytes": int(nbytes), "flops": int(e * roads * combs * 9)}


# ------------------------------------------------------------------ 64-bit results
EXACT_MAX_COMBS = 2_500_000


def _exact_records(words, off, consts, cfg):
    """Records of a batch by plain int64 numpy, one road at a time."""
    cut, max_comb, min_layers, xft = cfg
    F, q = consts.F.astype(np.int64), consts.q.astype(np.int64)
    out, first = [], [0]
    for e in range(len(off) - 1):
        ev = words[int(off[e]): int(off[e + 1])].astype(np.int64)
        heads = np.flatnonzero(ev >> 30 == 2)
        ends = np.append(heads[1:], len(ev))
        for h, z in zip(heads, ends):
            sector, rid = int(ev[h] >> 21) & 511, int(ev[h]) & 0x1FFFFF
            hit = ev[h + 1: z]
            lay = [hit[hit >> 27 == l] & 0x7FFF for l in range(6)]
            mask = sum(1 << l for l in range(6) if len(lay[l]))
            n_lay = bin(mask).count("1")
            x = [v if len(v) else np.zeros(1, np.int64) for v in lay]
            radix = [len(v) for v in x[:5 if xft else 6]]
            flags = 8 if len(hit) == 0 else 0
            rec = [rid, 0xFFFFFFFF, 0, 0, 0, 0]
            if n_lay < min_layers:
                flags |= 4
            else:
                total = math.prod(radix)
                flags |= 2 if total > max_comb else 0
                c = np.arange(min(total, max_comb))
                d = list(np.unravel_index(c, radix))
                if xft:
                    d.append(d[4])
                xs = np.stack([x[l][d[l]] for l in range(6)])
                y = (F[sector, mask] @ xs + (q[sector, mask] << consts.qshift)[:, None]) \
                    >> consts.oshift
                chi2 = (np.clip(y[3:], -32767, 32767) ** 2).sum(0)
                b = int(np.argmin(chi2))
                if chi2[b] <= cut:
                    flags |= 1
                    rec = [rid, b, int(chi2[b])] + [int(v) & 0xFFFFFFFF for v in y[:3, b]]
            rec[0] |= flags << 24
            out.append(rec)
        first.append(len(out))
    return np.array(out, np.uint32).reshape(-1, 6), np.array(first, np.int32)


def _exact_fit(case, seed):
    spec, consts, b, cut = _batch(case, seed)
    cfg = (cut, case["max_comb"], case["min_layers"], spec.xft)
    both = [b] + ([_batch(case, seed + 7919)[2]] if case["via"] == "host" else [])
    if case["via"] == "plain" or \
            sum(int(v.combinations(case["max_comb"]).sum()) + 50 * v.total_roads
                for v in both) > EXACT_MAX_COMBS:
        return None
    res = [_exact_records(v.words, v.event_off, consts, cfg) for v in both]
    ok = np.array([-1], np.int64)
    recs = []
    for rec, _ in res:
        full = np.zeros((_road_cap(case), 6), np.uint32)
        full[: len(rec)] = rec
        recs.append(full.view(np.int32).reshape(-1))
    if case["via"] == "host":
        return {"records": recs, "status": [ok, ok]}
    if case["via"] == "serve":
        return {"records": full, "status": np.repeat(ok, b.n_events).view(np.uint64)}
    return {"records": recs[0], "event_road": res[0][1], "counts": None, "status": ok}


def _exact_calib(case, seed):
    x, sector, theta, w, F, q, gy = _tracks(case, seed)
    S, n = case["sectors"], case["tracks"]
    perm = torch.sort(sector, stable=True)[1]
    x, theta = x[perm], theta[perm]
    if case["what"] == "prepare":
        return {"perm": perm.to(torch.int32), "x": x.double(), "theta": theta.double()}
    count = torch.bincount(sector, minlength=S).tolist()
    F, q, w = F.double(), q.double(), w.double()
    dF, dq = torch.zeros_like(F), torch.zeros_like(q)
    loss = torch.zeros((), dtype=torch.float64, device=F.device)
    y = torch.empty(n, 6, dtype=torch.float64, device=F.device)
    a = 0
    for s in range(S):
        z = a + count[s]
        xs = x[a:z].double()
        ys = xs @ F[s].T + q[s]
        y[a:z] = ys
        if gy is not None:
            g = gy[a:z].double()
        else:
            r = torch.cat([ys[:, :3] - theta[a:z].double(), ys[:, 3:]], 1)
            wt = torch.cat([w, torch.ones_like(w)])
            loss += (wt * r * r).sum() / n
            g = 2.0 / n * wt * r
        dF[s], dq[s] = g.T @ xs, g.sum(0)
        a = z
    return {"loss": {"loss": loss, "dF": dF, "dq": dq}, "eval": {"loss": loss},
            "monitor": {"loss": loss, "y": y, "dF": dF, "dq": dq},
            "fit": {"y": y, "dF": dF, "dq": dq}}[case["what"]]


def exact(case, seed):
    return (_exact_fit if case["kind"] == "fit" else _exact_calib)(case, seed)
