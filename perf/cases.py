"""The calls a single-pulse search makes of this library, as measurable cases.

Every case is a stream of filterbank data that repeats after `period` blocks
(one, or two for the host stream): the carried tail of a beam is then the same
before every pass, and a pass can be repeated with the same results.

Kinds of pass:
  block    one device-resident block of one beam through `execute`
  stream   two host blocks of one beam through `Pipeline` (push, push, pop, pop)
  batch    one block of every beam of a `Batch`
  plan     one block through a `DownsampledPlan` (six or fewer DM segments)
  cluster  the candidates of a searched block through `Clusterer`
"""
import math

import numpy as np
import torch

import paper_2401_13834_gb300 as tx
from paper_2401_13834_gb300.plans import DownsampledPlan

K_DM = 4.148808e3      # s MHz^2 pc^-1 cm^3
GAMMA = 7.0            # S/N threshold of candidate searches
MAX_CANDS = 1 << 16    # records a search has room for (what it finds fits)
MAX_POINTS = 1 << 18   # points a clustering has room for
MEERKAT = dict(f_lo=856.0, f_hi=1712.0, tsamp_us=153.12, descending=False, wmax=256, ratio=2.0)
SMALL = dict(f_lo=1200.0, f_hi=1456.0, tsamp_us=64.0, descending=False, wmax=64, ratio=2.0)


def _case(name, kind, nchan, nsub, ndm, dm_max, nseg, nsamp, layout, interm, norm, output, band=MEERKAT, **more):
    c = dict(name=name, kind=kind, nchan=nchan, nsub=nsub, ndm=ndm, dm_max=dm_max, nseg=nseg, nsamp=nsamp,
             layout=layout, interm=interm, norm=norm, output=output, stats="block", compact=False, beams=1, pulses=2,
             **band)
    c.update(more)
    return c


def listed():
    return [
        # a quick look at a narrow band in one short odd-length block: the smallest call, de-dispersed series only
        _case("tiny-series", "block", 64, 8, 24, 120.0, 1, 2003, "ft", "u16", "none", "series", band=SMALL),
        # one block of one beam that does not fill the GPU (the small workload): latency of the chain of kernels
        _case("small-plane", "block", 256, 16, 128, 200.0, 1, 16384, "tf", "u16", "none", "plane", band=SMALL),
        # many such beams served together in one step, replayed as a CUDA graph
        _case("small-batch", "batch", 256, 16, 128, 200.0, 1, 16384, "tf", "u16", "none", "plane", band=SMALL,
              beams=64),
        # the headline: MeerKAT-L blocks from pinned host memory, candidates back on the host
        _case("meerkat-stream", "stream", 4096, 64, 4096, 2000.0, 4, 65536, "tf", "u16", "none", "cands"),
        # the same block in device memory, as the DM-time plane of the best width
        _case("meerkat-plane", "block", 4096, 64, 4096, 2000.0, 4, 65536, "tf", "u16", "none", "plane"),
        # the whole S/N cube (every width kept) of a beam of moderate shape
        _case("cube", "block", 1024, 16, 1024, 1000.0, 4, 32768, "tf", "u16", "none", "cube"),
        # odd everything: channel-major, descending band, 125 channels a sub-band, prime block length, widths that
        # are no powers of two, running statistics
        _case("ragged-plane", "block", 1000, 8, 301, 220.0, 1, 20011, "ft", "u16", "none", "plane",
              band=dict(f_lo=1100.0, f_hi=1500.0, tsamp_us=100.0, descending=True, wmax=150, ratio=1.5),
              stats="running"),
        # uneven beams of a server: compact beams, FP16 intermediates, running statistics
        _case("served-f16", "batch", 2048, 32, 1024, 1500.0, 4, 32768, "tf", "f16", "none", "plane", beams=5,
              compact=True, stats="running"),
        # the MeerKAT-L block with every channel normalised to unit variance (the float path)
        _case("meerkat-float", "block", 4096, 64, 4096, 2000.0, 4, 65536, "tf", "f32", "unit", "plane"),
        # the float path on an odd shape: inverse-variance weights, channel-major, every width kept
        _case("ragged-float", "block", 768, 24, 333, 300.0, 1, 15013, "ft", "f32", "invvar", "cube",
              band=dict(f_lo=1200.0, f_hi=1600.0, tsamp_us=128.0, descending=True, wmax=81, ratio=3.0)),
        # the MeerKAT-L DM range as a plan that downsamples where a channel smears
        _case("downsampled-plan", "plan", 4096, 64, 4096, 2000.0, 4, 65536, "tf", "u16", "none", "cands"),
        # DBSCAN of a block's candidates: a few bright pulses, wide blobs on the DM-time plane
        _case("cluster", "cluster", 2048, 32, 2048, 1000.0, 4, 32768, "tf", "u16", "none", "cands", pulses=6,
              radius_ms=4.0, k=2),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """Another case of the same ranges; never more work than the largest listed one."""
    kind = rng.choice(["block"] * 6 + ["stream", "batch", "batch", "plan", "cluster"])
    wide = rng.random() < 0.5
    f_lo = rng.uniform(800.0, 900.0) if wide else rng.uniform(1100.0, 1300.0)
    f_hi = f_lo * (rng.uniform(1.7, 2.0) if wide else rng.uniform(1.15, 1.4))
    tsamp_us = rng.uniform(60.0, 160.0)
    m = rng.choice([16, 32, 50, 64, 64, 96, 125])
    nsub = max(2, int(_log(rng, 64, 4096) / m))
    nsub = min(nsub, 64)
    nchan = m * nsub
    ndm = int(_log(rng, 16, 4096))
    nsamp = int(_log(rng, 1500, 65536))
    if rng.random() < 0.5:
        nsamp = max(1024, nsamp // 1024 * 1024)
    # steps of the DM grid of 3 to 24 samples of delay across the band, as the listed grids have
    unit = K_DM * (f_lo ** -2 - f_hi ** -2) / (tsamp_us * 1e-6)
    dm_max = ndm * rng.uniform(3.0, 12.0) / unit
    interm, norm = rng.choice([("u16", "none")] * 5 + [("f16", "none"), ("i32", "none"), ("f32", "unit"),
                                                       ("f32", "invvar")])
    output = rng.choice(["plane", "plane", "cube", "series", "cands"])
    more = {}
    if kind in ("batch", "plan") and interm in ("f32", "i32"):
        interm, norm = "u16", "none"
    if kind == "stream":
        output = "cands"
    if kind == "plan":
        output, nsamp = "cands", max(8192, nsamp // 8192 * 8192)
    if kind == "cluster":
        output, interm, norm = "cands", "u16", "none"
        ndm, nsamp = max(ndm, 256), max(nsamp, 8192)
        more = dict(radius_ms=rng.choice([1.0, 2.0, 4.0, 8.0]), k=rng.choice([2, 4]), pulses=rng.randint(2, 6))
    if kind == "batch":
        more["beams"] = rng.choice([2, 4, 8, 16]) if nchan * ndm < 300000 else 2
        output = "plane" if output == "cands" else output
    stats = rng.choice(["block", "running"])
    compact = norm == "none" and rng.random() < 0.3
    if output == "cube":
        ndm, nsamp = min(ndm, 1024), min(nsamp, 32768)
    return _case("", kind, nchan, nsub, ndm, round(dm_max, 3), rng.choice([1, 4]) if ndm % 4 == 0 else 1, nsamp,
                 rng.choice(["tf", "tf", "ft"]), interm, norm, output,
                 band=dict(f_lo=round(f_lo, 3), f_hi=round(f_hi, 3), tsamp_us=round(tsamp_us, 3),
                           descending=rng.random() < 0.4, wmax=rng.choice([32, 64, 100, 256]),
                           ratio=rng.choice([2.0, 2.0, 1.5, 3.0])),
                 stats=stats, compact=compact, **more)


# ---- shapes ---------------------------------------------------------------------------
def _freqs(c):
    bw = (c["f_hi"] - c["f_lo"]) / c["nchan"]
    f = c["f_lo"] + (np.arange(c["nchan"], dtype=np.float64) + 0.5) * bw
    return f[::-1].copy() if c["descending"] else f


def _dms(c):
    """`nseg` segments of equally many trials whose step doubles from one to the next."""
    n, nseg = c["ndm"], c["nseg"]
    if nseg == 1:
        return c["dm_max"] * np.arange(n, dtype=np.float64) / max(n - 1, 1)
    per, total = n // nseg, float(2 ** nseg - 1)
    return np.concatenate([c["dm_max"] * (2 ** j - 1) / total + c["dm_max"] * 2 ** j / total / per
                           * np.arange(per, dtype=np.float64) for j in range(nseg)])


def _widths(c):
    out, w = [], 1.0
    while int(w + 0.5) <= c["wmax"]:
        if not out or int(w + 0.5) != out[-1]:
            out.append(int(w + 0.5))
        w *= c["ratio"]
    return np.asarray(out, dtype=np.int32)


def _members(c):
    """The shapes of a batch's beams: alike, or (compact beams) of uneven channel counts, DM counts and lengths."""
    n = c["beams"]
    if not c["compact"]:
        return [c] * n
    out = []
    for i in range(n):
        d = dict(c)
        d["nsub"] = max(1, c["nsub"] >> (i % 3))
        d["nchan"] = d["nsub"] * (c["nchan"] // c["nsub"])
        if c["nseg"] == 1 or c["ndm"] % 8 == 0:
            d["ndm"] = max(c["nseg"], c["ndm"] >> (i % 2))
        d["nsamp"] = c["nsamp"] * (1 + i % 2)
        out.append(d)
    return out


def _plan_args(c):
    return dict(freqs_mhz=_freqs(c), tsamp_s=c["tsamp_us"] * 1e-6, dms=_dms(c), nsub=c["nsub"], widths=_widths(c),
                nsamp=c["nsamp"], layout=c["layout"], interm=c["interm"], output=c["output"], stats=c["stats"],
                snr_threshold=GAMMA, max_cands=1 << 21 if c["kind"] == "cluster" else MAX_CANDS)


def _make_plan(c):
    return tx.Plan(norm=c["norm"], **_plan_args(c))


# ---- inputs ----------------------------------------------------------------------------
def _data(c, seed, period=1, device="cuda"):
    """uint8 [nchan, period * nsamp]: noise of mean 128 and a standard deviation of 8 to 16 counts per channel,
    `pulses` dispersed pulses of S/N 9 to 25 (20 to 50 for the clustering), wrapped at the period's end."""
    n, P = c["nchan"], period * c["nsamp"]
    rng = np.random.default_rng([seed, n, P])
    g = torch.Generator(device=device)
    g.manual_seed(seed)
    x = torch.randn((n, P), generator=g, device=device, dtype=torch.float32)
    sig = rng.uniform(8.0, 16.0, n).astype(np.float32)
    x.mul_(torch.from_numpy(sig).to(device)[:, None]).add_(128.0)
    f = torch.from_numpy(_freqs(c)).to(device)
    for _ in range(c["pulses"]):
        dm = rng.uniform(0.0, c["dm_max"])
        fwhm = math.exp(rng.uniform(math.log(4.0), math.log(60.0)))      # samples
        snr = rng.uniform(20.0, 50.0) if c["kind"] == "cluster" else rng.uniform(9.0, 25.0)
        t0 = rng.uniform(0.0, P)
        sd = fwhm / 2.3548
        amp = snr * 12.0 / math.sqrt(n * sd * math.sqrt(math.pi))
        at = t0 + K_DM * dm * (f ** -2 - float(f.max()) ** -2) / (c["tsamp_us"] * 1e-6)
        h = min(int(4 * sd) + 1, (P - 1) // 2)
        tt = torch.floor(at).to(torch.int64)[:, None] + torch.arange(-h, h + 1, device=device)[None, :]
        v = amp * torch.exp(-0.5 * ((tt.double() - at[:, None]) / sd) ** 2)
        x.scatter_add_(1, tt % P, v.float())
    return x.round_().clamp_(0.0, 255.0).to(torch.uint8)


def _window(X, end, n):
    """The n samples of the repeating stream before sample `end`."""
    P = X.shape[1]
    return X[:, torch.arange(end - n, end, device=X.device) % P]


def _lay(x, layout):
    return (x.t() if layout == "tf" else x).contiguous()


# ---- prepare / run ----------------------------------------------------------------------
def _batch(make):
    """A batch; a device holds two at a time, a third has no room."""
    try:
        return make()
    except tx.TxError as e:
        if e.code == -7:
            raise MemoryError("no room for another batch on this device") from e
        raise


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"case": c}
    if kind == "block":
        X = _data(c, seed)
        p = s["plan"] = _make_plan(c)
        b = s["beam"] = tx.Beam(p, compact=c["compact"])
        if p.overlap:
            b.prime(_lay(_window(X, 0, p.overlap), c["layout"]).reshape(-1))
        s["block"] = _lay(X, c["layout"]).reshape(-1)
        s["out"], s["ncand"] = p.alloc_out()
        s["ws"] = p.alloc_workspace(compact=c["compact"])
    elif kind == "stream":
        X = _data(c, seed, period=2)
        p = s["plan"] = _make_plan(c)
        b = s["beam"] = tx.Beam(p, compact=c["compact"])
        if p.overlap:
            b.prime(_lay(_window(X, 0, p.overlap), c["layout"]).reshape(-1))
        s["blocks"] = []
        for i in range(2):
            blk = _lay(X[:, i * c["nsamp"]:(i + 1) * c["nsamp"]], c["layout"]).reshape(-1)
            h = torch.empty(blk.numel(), dtype=torch.uint8, pin_memory=True)
            h.copy_(blk)
            s["blocks"].append(h)
        s["pipe"] = tx.Pipeline(p, b, depth=2)
        s["got"] = [_record_arrays() for _ in range(2)]
    elif kind == "batch":
        s["plans"], s["beams"], s["blocks"], s["outs"] = [], [], [], []
        same = {}
        for i, d in enumerate(_members(c)):
            key = (d["nchan"], d["ndm"], d["nsamp"])
            p = same[key] = same.get(key) or _make_plan(d)
            X = _data(d, seed * 1000 + i)
            b = tx.Beam(p, compact=c["compact"])
            if p.overlap:
                b.prime(_lay(_window(X, 0, p.overlap), c["layout"]).reshape(-1))
            s["plans"].append(p)
            s["beams"].append(b)
            s["blocks"].append(_lay(X, c["layout"]).reshape(-1))
        if len(same) == 1:      # beams of one shape: their outputs are rows of one buffer
            p = s["plans"][0]
            s["rows"] = torch.empty((len(s["plans"]), -(-p.out_bytes // 16) * 16), dtype=torch.uint8, device="cuda")
            s["outs"] = [(r[:p.out_bytes], None) for r in s["rows"]]
        else:
            s["outs"] = [p.alloc_out() for p in s["plans"]]
        s["batch"] = _batch(lambda: tx.Batch(s["plans"], s["beams"], graph=True))
        s["ws"] = s["batch"].alloc_workspace()
    elif kind == "plan":
        X = _data(c, seed)
        p = s["plan"] = DownsampledPlan(f_max=64, **_plan_args(c))
        s["beams"] = p.beams(compact=c["compact"])
        p.prime(s["beams"], _lay(_window(X, 0, p.overlap), c["layout"]).reshape(-1))
        s["batch"] = _batch(lambda: p.batch(s["beams"]))
        s["block"] = _lay(X, c["layout"]).reshape(-1)
        s["outs"] = s["batch"].alloc_outs()
        s["ws"], s["staging"] = s["batch"].alloc_workspace(), p.alloc_staging()
        s["got"] = _record_arrays()
    else:
        X = _data(c, seed)
        p = s["plan"] = _make_plan(c)
        b = tx.Beam(p)
        if p.overlap:
            b.prime(_lay(_window(X, 0, p.overlap), c["layout"]).reshape(-1))
        out, nc = tx.execute(p, b, _lay(X, c["layout"]).reshape(-1))
        n = min(int(nc.item()), p.max_cands)
        # the records come in no fixed order: the same shuffle of the sorted ones for everybody
        r = out[:n]
        n = min(n, MAX_POINTS)
        r = r[torch.argsort(r[:, 0].long() * c["nsamp"] + r[:, 1].long())[:n]]
        g = torch.Generator(device="cuda")
        g.manual_seed(seed + 1)
        s["cands"], s["n"] = r[torch.randperm(n, generator=g, device="cuda")].contiguous(), n
        s["clusterer"] = tx.Clusterer(p, c["radius_ms"], c["k"], MAX_POINTS)
        s["out"] = torch.zeros((MAX_POINTS, 10), dtype=torch.int32, device="cuda")
        s["count"] = torch.zeros(1, dtype=torch.int64, device="cuda")
        s["labels"] = torch.full((MAX_POINTS,), -2, dtype=torch.int32, device="cuda")
        s["order"] = torch.full((MAX_POINTS,), -2, dtype=torch.int32, device="cuda")
    return s


def _records(dm, t, w, snr):
    return {"dm": dm, "t": t, "w": w, "snr": snr}


def _record_arrays():
    return _records(np.zeros(MAX_CANDS, np.int32), np.zeros(MAX_CANDS, np.int64), np.zeros(MAX_CANDS, np.int32),
                    np.zeros(MAX_CANDS, np.float32))


def _sorted_host(r, t, into):
    """The records in order of DM and time in the caller's arrays, zeros behind them."""
    o, n = np.argsort(r["dm_index"].astype(np.int64) * (1 << 32) + t, kind="stable"), r.size
    for k, v in (("dm", r["dm_index"]), ("t", t), ("w", r["w_index"]), ("snr", r["snr"])):
        into[k][:n] = v[o]
        into[k][n:] = 0
    return into


def _view(plan, out):
    if plan.output == "plane":
        snr, w = tx.plane_view(plan, out)
        return {"snr": snr, "w": w}
    return {plan.output: tx.cube_view(plan, out) if plan.output == "cube" else tx.series_view(plan, out)}


def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "block":
        p = s["plan"]
        tx.execute(p, s["beam"], s["block"], out=s["out"], ncand=s["ncand"], workspace=s["ws"])
        if p.output != "cands":
            return _view(p, s["out"])
        # the records in order of DM and time, zeros behind them, without waiting for their number
        r = s["out"]
        have = torch.arange(MAX_CANDS, device="cuda") < s["ncand"]
        key = torch.where(have, r[:, 0].long() * c["nsamp"] + r[:, 1].long(), 1 << 62)
        r = torch.where(have[:, None], r[torch.argsort(key)], 0)
        return _records(r[:, 0], r[:, 1], r[:, 2], r[:, 3].contiguous().view(torch.float32))
    if kind == "stream":
        s["pipe"].push(s["blocks"][0])
        s["pipe"].push(s["blocks"][1])
        got = [s["pipe"].pop()[0], s["pipe"].pop()[0]]
        return [_sorted_host(r, r["t"].astype(np.int64), into) for r, into in zip(got, s["got"])]
    if kind == "batch":
        s["batch"].execute(s["blocks"], s["outs"], s["ws"])
        if "rows" in s:
            p, rows = s["plans"][0], s["rows"]
            n = p.ndm * p.nsamp
            if p.output == "plane":
                return {"snr": rows[:, :4 * n].view(torch.float32), "w": rows[:, 4 * n:5 * n]}
            dt = torch.float32 if p.output == "cube" else torch.int32
            return {p.output: rows[:, :p.out_bytes].view(dt)}
        return [_view(p, o) for p, (o, _) in zip(s["plans"], s["outs"])]
    if kind == "plan":
        s["plan"].execute(s["batch"], s["block"], s["outs"], s["ws"], s["staging"])
        r = s["plan"].merge_cands(s["outs"])
        return _sorted_host(r, r["t_native"], s["got"])
    s["clusterer"].run(s["cands"], s["n"], out=s["out"], nclusters=s["count"], labels=s["labels"], order=s["order"])
    return {"clusters": s["out"], "count": s["count"], "labels": s["labels"], "order": s["order"]}


# ---- the same in 64 bits ------------------------------------------------------------------
def _round(v):
    return np.floor(v + 0.5).astype(np.int64)


def _group(f, nsub, ndm):
    m = f.size // nsub
    full = f.min() ** -2 - f.max() ** -2
    sub = max(b.min() ** -2 - b.max() ** -2 for b in f.reshape(nsub, m))
    cap = 1 << (ndm.bit_length() - 1)
    if sub <= 0:
        return cap
    g = 1
    while 2 * g <= min(1.0 + full / sub, cap):
        g *= 2
    return g


def _tables(f, tsamp, dms, nsub):
    m, G = f.size // nsub, _group(f, nsub, dms.size)
    k_of = np.arange(dms.size) // G
    coarse = np.asarray([(dms[k * G] + dms[min((k + 1) * G, dms.size) - 1]) / 2 for k in range(k_of[-1] + 1)])
    fs = f.reshape(nsub, m).max(axis=1)
    d1 = _round(K_DM * coarse[:, None] * (1 / (f * f) - 1 / np.repeat(fs, m) ** 2)[None, :] / tsamp)
    d2 = _round(K_DM * dms[:, None] * (1 / (fs * fs) - 1 / f.max() ** 2)[None, :] / tsamp)
    span = max(int((d1[k_of][:, s * m:(s + 1) * m].max(axis=1) + d2[:, s]).max()) for s in range(nsub))
    return d1, d2, k_of, span


def _exact_series(X, f, tsamp, dms, nsub, n):
    """D[d][t] for t < n in float64 from X [nchan, span + n or more] (any real type)."""
    d1, d2, k_of, span = _tables(f, tsamp, dms, nsub)
    m, nk = f.size // nsub, d1.shape[0]
    D = torch.zeros((dms.size, n), dtype=torch.float64, device=X.device)
    for s in range(nsub):
        n1 = n + int(d2[:, s].max())
        Ps = torch.zeros((nk, n1), dtype=torch.float64, device=X.device)
        for ch in range(s * m, (s + 1) * m):
            row = torch.zeros(n1 + int(d1[:, ch].max()), dtype=torch.float64, device=X.device)
            have = min(row.numel(), X.shape[1])
            row[:have] = X[ch, :have]
            Ps += row.as_strided((row.numel() - n1 + 1, n1), (1, 1))[torch.from_numpy(d1[:, ch]).to(X.device)]
        rows = Ps.view(-1).as_strided((nk * n1 - n + 1, n), (1, 1))
        start = torch.from_numpy(k_of * n1 + d2[:, s]).to(X.device)
        for i in range(0, dms.size, 512):
            D[i:i + 512] += rows[start[i:i + 512]]
    return D


def _exact_snr(D, T, widths, output):
    """The cube [d][w][t], or the plane's best S/N [d][t]."""
    nd = D.shape[0]
    out = torch.empty((nd, len(widths), T) if output == "cube" else (nd, T), dtype=torch.float64, device=D.device)
    for i in range(0, nd, 128):
        d = D[i:i + 128]
        mu = d[:, :T].mean(dim=1, keepdim=True)
        sg = (d[:, :T] - mu).square().mean(dim=1, keepdim=True).sqrt()
        inv = torch.where(sg > 0, 1 / sg, torch.zeros_like(sg))
        C = torch.nn.functional.pad(torch.cumsum(d, dim=1), (1, 0))
        best = None
        for j, w in enumerate(int(v) for v in widths):
            v = (C[:, w:w + T] - C[:, :T] - w * mu) * (inv / math.sqrt(w))
            if output == "cube":
                out[i:i + 128, j] = v
            else:
                best = v if best is None else torch.maximum(best, v)
        if output != "cube":
            out[i:i + 128] = best
    return out


def _exact_window(X, end, f, tsamp, dms, nsub, w, T, norm, output):
    """What a fresh beam gives for the block of T samples of the stream X that ends at sample `end`."""
    L = _tables(f, tsamp, dms, nsub)[3] + int(w[-1]) - 1
    win = _window(X, end, L + T)
    if norm != "none":      # the tail was normalised as a block of its own
        parts = []
        for x in (win[:, :L], win[:, L:]):
            if x.shape[1]:
                x = x.double()
                mu = x.mean(dim=1, keepdim=True)
                var = (x - mu).square().mean(dim=1, keepdim=True)
                wt = 1 / (var.sqrt() if norm == "unit" else var)
                parts.append((x - mu) * torch.where(var > 0, wt, torch.zeros_like(wt)))
        win = torch.cat(parts, dim=1)
    D = _exact_series(win, f, tsamp, dms, nsub, T + int(w[-1]) - 1)
    return D if output == "series" else _exact_snr(D, T, w, output)


def _exact_beam(c, X, end, output):
    return _exact_window(X, end, _freqs(c), c["tsamp_us"] * 1e-6, _dms(c), c["nsub"], _widths(c), c["nsamp"],
                         c["norm"], output)


def _cands(*planes):
    v = torch.cat([v[v >= GAMMA] for v in planes])
    return _records(None, None, None, torch.nn.functional.pad(v, (0, MAX_CANDS - v.numel())))


def _factors(c):
    """The downsampling factor of every DM trial: the largest power of two, at most 64 and dividing the block, not
    above the smear (samples) of the lowest channel."""
    f, dms, most = _freqs(c), _dms(c), 64
    while c["nsamp"] % most:
        most //= 2
    half = (c["f_hi"] - c["f_lo"]) / c["nchan"] / 2
    smear = K_DM * dms * ((f.min() - half) ** -2 - (f.min() + half) ** -2) / (c["tsamp_us"] * 1e-6)
    return np.minimum(2 ** np.floor(np.log2(np.maximum(smear, 1.0))).astype(np.int64), most)


def _exact_plan(c, X):
    """The candidates of the DM segments, each on the block averaged (rounded half up) over its factor."""
    fac, dms, planes = _factors(c), _dms(c), []
    for k in sorted(set(fac.tolist())):
        Xk = torch.cat([((r.to(torch.int32).view(r.shape[0], -1, k).sum(dim=2) + k // 2) // k).to(torch.uint8)
                        for r in X.split(64)])
        w = np.unique(np.maximum(_widths(c) // k, 1))
        planes.append(_exact_window(Xk, Xk.shape[1], _freqs(c), c["tsamp_us"] * 1e-6 * k, dms[fac == k], c["nsub"], w,
                                    c["nsamp"] // k, "none", "plane"))
    return _cands(*planes)


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "block":
        X = _data(c, seed)
        if c["output"] == "cands":
            return _cands(_exact_beam(c, X, c["nsamp"], "plane"))
        v = _exact_beam(c, X, c["nsamp"], c["output"])
        return {"snr": v, "w": None} if c["output"] == "plane" else {c["output"]: v}
    if kind == "stream":
        X = _data(c, seed, period=2)
        return [_cands(_exact_beam(c, X, (i + 1) * c["nsamp"], "plane")) for i in range(2)]
    if kind == "batch":
        vs = []
        for i, d in enumerate(_members(c)):
            vs.append(_exact_beam(d, _data(d, seed * 1000 + i), d["nsamp"], c["output"]))
        key = "snr" if c["output"] == "plane" else c["output"]
        if len({v.shape for v in vs}) > 1:
            return [{key: v, "w": None} for v in vs]
        return {key: torch.stack([v.reshape(-1) for v in vs]), "w": None}
    return _exact_plan(c, _data(c, seed)) if kind == "plan" else None      # the clustering gives whole numbers


def work(case):
    c, kind = case, case["kind"]
    if kind == "cluster":
        n = 30000 * c["pulses"] // 2
        return {"bytes": n * (16 + 8), "flops": n * 9 * 8}
    nbytes = flops = 0
    for d in (_members(c) if kind == "batch" else [c] * (2 if kind == "stream" else 1)):
        f, w, T, dms = _freqs(d), _widths(d), d["nsamp"], _dms(d)
        tsamp = d["tsamp_us"] * 1e-6
        L = K_DM * d["dm_max"] * (f.min() ** -2 - f.max() ** -2) / tsamp + int(w[-1])
        out = {"plane": 5 * d["ndm"] * T, "cube": 4 * len(w) * d["ndm"] * T, "series": 4 * d["ndm"] * T,
               "cands": 16000}[d["output"]]
        Td = T + int(w[-1]) - 1
        adds = math.ceil(d["ndm"] / _group(f, d["nsub"], d["ndm"])) * d["nchan"] * Td + d["ndm"] * d["nsub"] * Td
        filt = 0 if d["output"] == "series" else 3 * len(w) * d["ndm"] * T
        # a plan's trials are de-dispersed at 1 / factor of the samples
        share = float(np.mean(1.0 / _factors(d))) if kind == "plan" else 1.0
        nbytes += d["nchan"] * (T + L) + out
        flops += (adds + filt) * share
    return {"bytes": float(nbytes), "flops": float(flops)}
