"""The work that users of the library have it do, as timed cases: searches of a peakmap (single maps,
sub-bands, many braking indices, uneven peakmaps, proposed coarse tiles), peakmaps of a series, the
follow-up of a candidate, and the tile proposer's network.  Sizes are those of the package's
workloads (paper_1810_09784_gb300/workloads.py, proposer.py); `draw` spreads over the same ranges.

Hough maps, candidates and peak lists are whole numbers (candidate records and map statistics come
back as bytes and int64): they have no 64-bit counterpart and `exact` gives values for the network
only.
"""
from __future__ import annotations

import math
import pathlib

import numpy as np
import torch
import torch.nn.functional as F

from paper_1810_09784_gb300 import gfh, synth

THETA = 2.5
TILES = 64                       # coarse tiles per axis of the proposer
CLASSES = 4097
WEIGHTS = pathlib.Path(__file__).resolve().parent.parent / "paper_1810_09784_gb300" / "weights" / \
    "proposer_series.npz"
COUT, CIN, STRIDE = (32, 32, 64, 64, 64), (2, 32, 32, 64, 64), (1, 2, 1, 2, 1)


# ---- the cases ------------------------------------------------------------------------------------

def listed():
    return [
        # the original FrequencyHough of one followed-up candidate: the smallest map, all launches
        dict(name="followup_map", kind="hough", n_lo=0.0, n_hi=0.0, maps=1, t_obs=10080.0, t_fft=8.0,
             f_lo=995.0, f_hi=1005.0, rows_lo=32, rows_hi=32, tune=False),
        # one braking index on the half-hour series, 500 k rows
        dict(name="small_map", kind="hough", n_lo=5.0, n_hi=5.0, maps=1, t_obs=1800.0, t_fft=2.0,
             f_lo=100.0, f_hi=400.0, rows_lo=500, rows_hi=500, tune=False),
        # the half-hour peakmap at many braking indices, fewer k rows at higher n, one launch
        dict(name="braking_indices", kind="hough", n_lo=2.0, n_hi=7.0, maps=11, t_obs=1800.0,
             t_fft=2.0, f_lo=100.0, f_hi=400.0, rows_lo=4000, rows_hi=1000, tune=False),
        # the paper-shaped search, series to candidates: 20 sub-bands of 100 Hz (+ 50 Hz), 2000 k
        # rows, tile shape tuned once as a long search does
        dict(name="paper_search", kind="search", n=5.0, fs=4096.0, t_obs=10080.0, t_fft=4.0,
             f_lo=50.0, f_hi=2000.0, rows=2000, tune=True),
        # peakmaps of different lengths, bands and FFT lengths in one launch
        dict(name="uneven_maps", kind="uneven", lists=12, hours_lo=0.5, hours_hi=4.0, rows=500,
             layout=3),
        # the exact Hough on the proposer's tiles: one map per braking index, one of them in full
        dict(name="coarse_tiles", kind="tiles", maps=51, t_obs=1800.0, t_fft=2.0, f_lo=100.0,
             f_hi=400.0, rows=500, picks=50, full=1),
        # peakmap of the half-hour series, and of the 2.8 hour series
        dict(name="peakmap_small", kind="peakmap", fs=1024.0, t_obs=1800.0, t_fft=2.0, f_lo=100.0,
             f_hi=400.0),
        dict(name="peakmap_paper", kind="peakmap", fs=4096.0, t_obs=10080.0, t_fft=4.0, f_lo=50.0,
             f_hi=2000.0),
        # follow-up of one candidate: the peaks of the corrected series in f0 +- 5 Hz, its map
        dict(name="followup_band", kind="followup", fs=4096.0, t_obs=10080.0, t_fft=8.0, f0=1000.0,
             half_band=5.0, rows=32),
        # the network on one batch of maps, its gradients on one training batch, and the costliest
        # of its layers alone (the input gradient of the first strided layer)
        dict(name="network_forward", kind="forward", batch=51),
        dict(name="network_gradients", kind="gradients", batch=256),
        dict(name="layer_input_gradient", kind="layer", mode=1, layer=1, batch=64, h=256),
    ]


def draw(rng):
    logu = lambda a, b: math.exp(rng.uniform(math.log(a), math.log(b)))      # noqa: E731
    kind = rng.choice(("hough", "hough", "search", "uneven", "tiles", "peakmap", "followup",
                       "forward", "gradients", "layer"))
    if kind == "hough":
        while True:
            t_fft = float(rng.choice((1, 2, 4, 8)))
            f_lo = round(logu(70.0, 1500.0), 2) + (130.0 if t_fft == 1.0 else 0.0)
            maps = rng.choice((1, 1, 2, 5))
            n_lo = rng.choice((0.0, round(rng.uniform(2.0, 5.0), 2), round(rng.uniform(5.0, 7.0), 2)))
            c = dict(kind=kind, n_lo=n_lo, n_hi=n_lo if n_lo == 0.0 or maps == 1 else 7.0,
                     maps=1 if n_lo == 0.0 else maps, t_obs=round(logu(600.0, 10080.0), 1),
                     t_fft=t_fft, f_lo=f_lo, f_hi=f_lo + round(logu(10.0, 300.0), 2),
                     rows_lo=int(logu(32, 4000)), rows_hi=int(logu(32, 2000)), tune=False)
            grids = [gfh.grid_make(gfh.Grid(**f)) for f in _hough_fields(c)]
            cells = sum(g.n_k * g.ld_x0 for g in grids)
            if 3.0e4 < cells < 8.0e8 and _updates(grids) < 6.0e9:
                return c
    if kind == "search":
        f_lo = round(rng.uniform(50.0, 800.0))
        return dict(kind=kind, n=round(rng.uniform(2.5, 7.0), 2), fs=4096.0,
                    t_obs=round(logu(900.0, 6000.0)), t_fft=float(rng.choice((2, 4))), f_lo=float(f_lo),
                    f_hi=float(f_lo + rng.randint(60, 1000)), rows=int(logu(100, 1500)), tune=False)
    if kind == "uneven":
        return dict(kind=kind, lists=rng.randint(3, 12), hours_lo=0.5, hours_hi=round(logu(1.0, 4.0), 2),
                    rows=int(logu(60, 500)), layout=rng.randint(4, 1 << 20))
    if kind == "tiles":
        return dict(kind=kind, maps=rng.randint(3, 51), t_obs=round(logu(700.0, 3600.0), 1), t_fft=2.0,
                    f_lo=float(rng.randint(80, 120)), f_hi=float(rng.randint(300, 400)),
                    rows=rng.randint(130, 500), picks=rng.randint(3, 200), full=rng.randint(0, 2))
    if kind == "peakmap":
        fs = float(rng.choice((1024, 2048, 4096)))
        f_lo = round(rng.uniform(140.0, 200.0))
        return dict(kind=kind, fs=fs, t_obs=round(logu(300.0, 10080.0), 1),
                    t_fft=float(rng.choice((1, 2, 4, 8))), f_lo=float(f_lo),
                    f_hi=round(f_lo + logu(20.0, 0.45 * fs - f_lo), 2))
    if kind == "followup":
        t_fft = float(rng.choice((4, 8, 16)))
        return dict(kind=kind, fs=4096.0, t_obs=round(logu(600.0, 10080.0), 1), t_fft=t_fft,
                    f0=round(rng.uniform(300.0, 1800.0), 2),
                    half_band=round(rng.uniform(3.0, 7.0 if t_fft < 16 else 5.0), 2),
                    rows=rng.randint(8, 64))
    if kind == "layer":
        layer = rng.randint(0, 4)
        mode = rng.choice((0, 2)) if layer == 0 else rng.choice((0, 1, 2))
        return dict(kind=kind, mode=mode, layer=layer, batch=int(logu(1, 64)),
                    h=256 >> sum(1 for s in STRIDE[:layer] if s == 2))
    return dict(kind=kind, batch=int(logu(1, 256)))


# ---- inputs ---------------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _n_fft(t_obs, t_fft):
    return int((t_obs - t_fft) // (t_fft / 2)) + 1


def _bins(c):
    """First and last bin of the peakmap band (the equaliser warms up on the 129 bins below it)."""
    return max(130, int(math.ceil(c["f_lo"] * c["t_fft"]))), int(math.floor(c["f_hi"] * c["t_fft"])) - 1


def _peaks(seed, n_fft, bin_lo, bin_hi, tracks=()):
    """Peak list of a noise peakmap with a few power-law tracks, as the peakmap builder emits it: the
    strict local maxima along frequency above the threshold of exponential spectra, sorted by
    (bin, FFT)."""
    g = _gen(seed)
    p = torch.rand((bin_hi - bin_lo + 3, n_fft), generator=g, device="cuda").log_().neg_()
    pk = (p[1:-1] > THETA) & (p[1:-1] > p[:-2]) & (p[1:-1] > p[2:])
    del p
    for tr in tracks:
        i = torch.arange(n_fft, device="cuda")
        j = torch.from_numpy(np.asarray(tr, np.int64)).cuda() - bin_lo
        on = (j >= 0) & (j < pk.shape[0]) & (torch.rand(n_fft, generator=g, device="cuda") < 0.6)
        pk[j[on], i[on]] = True
    at = pk.nonzero()
    return at[:, 1].to(torch.int32).contiguous(), (at[:, 0] + bin_lo).to(torch.int32).contiguous()


def _track(seed, t_fft, n_fft, f_lo, f_hi):
    r = np.random.RandomState(seed % (1 << 31))
    f0, n = r.uniform(f_lo + 0.4 * (f_hi - f_lo), f_hi), r.uniform(2.0, 7.0)
    fdot = math.exp(r.uniform(math.log(1e-4), math.log(1.0 / t_fft ** 2)))
    return synth.powerlaw_track(f0, fdot / f0 ** n, n, 1.0 / t_fft, n_fft, t_fft / 2, t_fft / 2)


def _grid_fields(n, c, bin_lo, bin_hi, rows, ana_lo, ana_hi, lst=0):
    n_fft = _n_fft(c["t_obs"], c["t_fft"])
    f = dict(n=n, df=1.0 / c["t_fft"], bin_lo=bin_lo, bin_hi=bin_hi, n_fft=n_fft, t_first=c["t_fft"] / 2,
             t_hop=c["t_fft"] / 2, t_obs=c["t_obs"], n_k=rows, ana_lo=ana_lo, ana_hi=ana_hi, list=lst)
    if n == 0.0:                                 # the original FrequencyHough: fdot rows around 0
        dk = f["df"] / c["t_obs"]
        f.update(k_min=-(rows // 2) * dk, dk=dk, band_hz=max(1.0, ana_hi - ana_lo))
    return f


def _hough_fields(c):
    lo, hi = _bins(c)
    out = []
    for m in range(c["maps"]):
        u = m / (c["maps"] - 1) if c["maps"] > 1 else 0.0
        n = round(c["n_lo"] + u * (c["n_hi"] - c["n_lo"]), 10)
        rows = int(round(c["rows_lo"] + u * (c["rows_hi"] - c["rows_lo"])))
        out.append(_grid_fields(n, c, lo, hi, rows, lo / c["t_fft"], (hi + 1) / c["t_fft"]))
    return out


def _search_fields(c):
    """100 Hz analysis bands, each with its peakmap band 50 Hz wider upwards."""
    out, a = [], c["f_lo"]
    T, (b_lo, b_hi) = c["t_fft"], _bins(c)
    while a < c["f_hi"] - 1.0:
        b = min(a + 100.0, c["f_hi"])
        top = min(b + 50.0, c["f_hi"])
        lo, hi = max(b_lo, int(round(a * T))), min(b_hi, int(round(top * T)) - 1)
        if hi > lo:
            out.append(_grid_fields(c["n"], c, lo, hi, c["rows"], a, b))
        a = b
    return out


def _uneven_specs(c):
    r = np.random.RandomState(c["layout"])       # the layout of the peakmaps is the case's own
    out = []
    for _ in range(c["lists"]):
        t_fft = float(r.choice([1.0, 2.0, 4.0, 8.0]))
        w = math.exp(r.uniform(math.log(20.0), math.log(400.0)))
        f_lo = r.uniform(140.0, 2000.0 - w)
        out.append(dict(t_obs=3600.0 * math.exp(r.uniform(math.log(c["hours_lo"]), math.log(c["hours_hi"]))),
                        t_fft=t_fft, f_lo=f_lo, f_hi=f_lo + w, n=r.uniform(2.0, 7.0), rows=c["rows"]))
    return out


def _updates(grids):
    """Peaks x k rows, at the noise peaks' density."""
    return sum(0.0755 * g.n_fft * (g.bin_hi - g.bin_lo + 1) * g.n_k for g in grids)


def _plan_state(ctx, grids, tile=None):
    cells = [g.n_k * g.ld_x0 for g in grids]
    flat = torch.zeros(sum(cells), dtype=torch.int32, device="cuda")
    maps = [m.view(g.n_k, g.ld_x0) for m, g in zip(flat.split(cells), grids)]
    nb = [g.n_bands * gfh.CANDIDATE_BYTES for g in grids]
    cand = torch.zeros(sum(nb), dtype=torch.uint8, device="cuda")
    stats = torch.zeros(3 * len(grids), dtype=torch.int64, device="cuda")
    plan = gfh.Plan(ctx, grids, maps, list(cand.split(nb)), stats, tile=tile)
    return dict(plan=plan, out=[flat, cand, stats])


def _layer_inputs(c, seed):
    g, l, B, h = _gen(seed), c["layer"], c["batch"], c["h"]
    ho = h // STRIDE[l]
    rn = lambda *s: torch.randn(s, generator=g, device="cuda")             # noqa: E731
    w = (rn(COUT[l], 3, 3, CIN[l]) * math.sqrt(2.0 / (9 * CIN[l]))).to(torch.bfloat16)
    x = rn(B, h, h, CIN[l]).relu_().to(torch.bfloat16)
    bias = 0.1 * rn(COUT[l])
    y = rn(B, ho, ho, COUT[l]).relu_().to(torch.bfloat16)                   # the layer's activation
    dy = (rn(B, ho, ho, COUT[l]) * 1e-3).to(torch.bfloat16)
    return w, x, bias, y, dy


def _network_inputs(c, seed):
    """Log-count images of noise peakmaps, half of them with a drifting track, and their classes."""
    g, B = _gen(seed), c["batch"]
    cnt = torch.poisson(torch.full((B, 256, 256), 1.24, device="cuda"), generator=g)
    xt = torch.randint(8, TILES, (B,), generator=g, device="cuda")
    d = torch.randint(0, TILES, (B,), generator=g, device="cuda")
    sig = torch.rand(B, generator=g, device="cuda") < 0.5
    tb = torch.arange(256, device="cuda")
    fb = 4 * xt[:, None] + 2 - ((d[:, None] + 0.5) * 3.3 * tb[None] / 256).long()
    on = (fb >= 0) & sig[:, None]
    b_i, t_i = on.nonzero(as_tuple=True)
    cnt[b_i, t_i, fb[b_i, t_i]] += 4.0
    img = torch.empty((B, 256, 256, 2), dtype=torch.bfloat16, device="cuda")
    img[..., 0] = torch.log1p(cnt).to(torch.bfloat16)
    n = torch.rand(B, generator=g, device="cuda")
    img[..., 1] = n[:, None, None].to(torch.bfloat16)
    labels = torch.where(sig, d * TILES + xt, torch.full_like(d, CLASSES - 1)).to(torch.int32)
    return img, labels


def _weights():
    with np.load(WEIGHTS) as z:
        return z["params"].copy()


def prepare(case, seed):
    c, kind = case, case["kind"]
    ctx = gfh.Context(0, torch.cuda.current_stream())
    s = dict(case=c, ctx=ctx)
    if kind in ("hough", "uneven", "tiles"):
        specs = {"hough": [c], "uneven": None, "tiles": [c] * c.get("maps", 0)}[kind] or _uneven_specs(c)
        if kind == "hough":
            fields = _hough_fields(c)
        elif kind == "tiles":
            lo, hi = _bins(c)
            fields = [_grid_fields(round(2.0 + 5.0 * m / 50, 10), c, lo, hi, c["rows"], lo / c["t_fft"],
                                   (hi + 1) / c["t_fft"], m) for m in range(c["maps"])]
        else:
            fields = [dict(f, list=l) for l, u in enumerate(specs) for f in _search_fields(u)]
        lists = []
        for l, u in enumerate(specs):
            n_fft, (lo, hi) = _n_fft(u["t_obs"], u["t_fft"]), _bins(u)
            q = 1009 * seed + l
            lists.append(_peaks(q, n_fft, lo, hi, [_track(q, u["t_fft"], n_fft, u["f_lo"], u["f_hi"])]))
        s["fft"], s["bin"] = (torch.cat([x[k] for x in lists]) for k in (0, 1))
        s["off"] = torch.tensor([0] + [len(x[0]) for x in lists], device="cuda").cumsum(0)
        s["n_lists"] = len(lists)
        s.update(_plan_state(ctx, [gfh.grid_make(gfh.Grid(**f)) for f in fields]))
        if kind == "tiles":
            s["plan"].set_coarse(TILES, TILES, 256)
            g = _gen(seed + 7)
            pick = torch.rand((c["maps"], TILES * TILES), generator=g, device="cuda").argsort(1)
            s["coarse"] = pick[:, :c["picks"]].to(torch.int32).contiguous()
            s["full"] = torch.zeros(c["maps"], dtype=torch.int32, device="cuda")
            s["full"][c["maps"] // 2:c["maps"] // 2 + c["full"]] = 1
    elif kind in ("search", "peakmap", "followup"):
        r = np.random.RandomState(seed)
        f0 = c.get("f0", 0.5 * (c.get("f_lo", 0.0) + c.get("f_hi", 0.0)))
        n = c.get("n", 5.0)
        k = math.exp(r.uniform(math.log(1e-4), math.log(1e-2))) / f0 ** n
        amp = synth.amplitude_for_snr(4.0, 1.0, int(c["fs"] * c["t_fft"]))
        s["x"] = torch.empty(int(c["fs"] * c["t_obs"]), dtype=torch.float32, device="cuda")
        synth.strain_series_device(s["x"], c["fs"], seed, (synth.Injection(f0, k, n, amp),))
        s.update(f0=f0, k=k, n=n)
        n_fft = _n_fft(c["t_obs"], c["t_fft"])
        if kind == "followup":
            s["band"] = tuple(int(f((f0 + d * c["half_band"]) * c["t_fft"]))
                              for f, d in ((math.floor, -1), (math.ceil, 1)))
            fields = [_grid_fields(0.0, c, *s["band"], c["rows"], f0 - c["half_band"] + 1.0,
                                   f0 + c["half_band"] - 1.0)]
        else:
            s["band"] = _bins(c)
            fields = _search_fields(c) if kind == "search" else []
        cap = int(n_fft * (s["band"][1] - s["band"][0] + 1) * 0.12) + 4096
        s["fft"], s["bin"] = (torch.zeros(cap, dtype=torch.int32, device="cuda") for _ in range(2))
        s["off"] = torch.zeros(2, dtype=torch.int64, device="cuda")
        s["n_lists"] = 1
        if fields:
            s.update(_plan_state(ctx, [gfh.grid_make(gfh.Grid(**f)) for f in fields]))
        if kind == "search":
            ctx.peakmap_async(s["x"], c["fs"], c["t_fft"], *s["band"], THETA, s["fft"], s["bin"],
                              s["off"][1:2])
    elif kind == "layer":
        w, x, bias, y, dy = _layer_inputs(c, seed)
        l = c["layer"]
        s.update(w=w, x=x, bias=bias, y=y, dy=dy,
                 res=(torch.empty_like(y) if c["mode"] == 0 else torch.empty_like(x) if c["mode"] == 1
                      else torch.empty(w.shape, dtype=torch.float32, device="cuda")),
                 db=torch.empty(COUT[l], dtype=torch.float32, device="cuda"))
    else:
        s["img"], s["labels"] = _network_inputs(c, seed)
        s["net"] = gfh.Cnn(ctx, c["batch"], seed=1)
        s["net"].set_params(_weights())
        s["logits"] = torch.empty((c["batch"], CLASSES), dtype=torch.float32, device="cuda")
    if c.get("tune"):
        s["plan"].autotune(s["fft"], s["bin"], s["off"], s["n_lists"], reps=2)
    return s


# ---- one pass -------------------------------------------------------------------------------------

def run(s):
    c, ctx, kind = s["case"], s["ctx"], s["case"]["kind"]
    if kind in ("hough", "uneven"):
        s["plan"].execute(s["fft"], s["bin"], s["off"], s["n_lists"])
        return s["out"]
    if kind == "tiles":
        s["plan"].execute_tiles(s["fft"], s["bin"], s["off"], s["n_lists"], s["coarse"], c["picks"],
                                s["full"])
        return s["out"]
    if kind == "search":
        ctx.peakmap_async(s["x"], c["fs"], c["t_fft"], *s["band"], THETA, s["fft"], s["bin"],
                          s["off"][1:2])
        s["plan"].execute(s["fft"], s["bin"], s["off"], 1)
        return [s["off"], s["fft"], s["bin"], *s["out"]]
    if kind == "peakmap":
        n = ctx.peakmap(s["x"], c["fs"], c["t_fft"], *s["band"], THETA, s["fft"], s["bin"])
        return [n, s["fft"], s["bin"]]                       # zeros behind the n peaks
    if kind == "followup":
        n = ctx.heterodyne_band_peaks(s["x"], c["fs"], 0.0, s["f0"], s["k"], s["n"], c["t_fft"],
                                      *s["band"], THETA, s["fft"], s["bin"])
        s["off"][1] = n
        s["plan"].execute(s["fft"], s["bin"], s["off"], 1)
        return [n, s["fft"], s["bin"], *s["out"]]
    if kind == "layer":
        l, h = c["layer"], c["h"]
        args = (ctx, c["mode"], CIN[l], COUT[l], STRIDE[l], c["batch"], h)
        if c["mode"] == 0:
            gfh.conv3x3(*args, inp=s["x"], w=s["w"], bias=s["bias"], res=s["res"])
            return s["res"]
        if c["mode"] == 1:
            gfh.conv3x3(*args, w=s["w"], out=s["y"], dout=s["dy"], res=s["res"])
            return s["res"]
        s["res"].zero_()                                     # the gradients are added to these
        s["db"].zero_()
        gfh.conv3x3(*args, inp=s["x"], out=s["y"], dout=s["dy"], res=s["res"], db=s["db"])
        return [s["res"], s["db"]]
    if kind == "forward":
        s["net"].forward(s["img"], s["logits"])
        return s["logits"]
    loss = s["net"].gradients(s["img"], s["labels"])
    return [loss, s["net"].grads()]


# ---- what a pass cannot do without ----------------------------------------------------------------

def _layer_macs(l, h):
    return (h // STRIDE[l]) ** 2 * 9 * CIN[l] * COUT[l]


def work(case):
    c, kind = case, case["kind"]
    if kind in ("hough", "uneven", "search", "tiles"):
        if kind == "uneven":
            specs = _uneven_specs(c)
            fields = [f for u in specs for f in _search_fields(u)]
        else:
            specs = [c] * (c["maps"] if kind == "tiles" else 1)
            fields = _hough_fields(c) if kind == "hough" else _search_fields(c) if kind == "search" else []
            if kind == "tiles":
                lo, hi = _bins(c)
                fields = [_grid_fields(round(2.0 + 5.0 * m / 50, 10), c, lo, hi, c["rows"],
                                       lo / c["t_fft"], (hi + 1) / c["t_fft"]) for m in range(c["maps"])]
        grids = [gfh.grid_make(gfh.Grid(**f)) for f in fields]
        peaks = sum(0.0755 * _n_fft(u["t_obs"], u["t_fft"]) * (_bins(u)[1] - _bins(u)[0] + 1) for u in specs)
        cells, upd = [float(g.n_k * g.ld_x0) for g in grids], [_updates([g]) for g in grids]
        if kind == "tiles":                       # the picked share of each map, the flagged in full
            share = [1.0 if len(grids) // 2 <= m < len(grids) // 2 + c["full"]
                     else c["picks"] / float(TILES * TILES) for m in range(len(grids))]
            cells, upd = ([v * w for v, w in zip(x, share)] for x in (cells, upd))
        # the peak list read, every cell written, one addition per peak and k row; from a series
        # also the series read and its FFTs
        b, f = 8.0 * peaks + 4.0 * sum(cells), sum(upd)
        if kind == "search":
            N = c["fs"] * c["t_fft"]
            b += 4.0 * c["fs"] * c["t_obs"] + 8.0 * peaks
            f += _n_fft(c["t_obs"], c["t_fft"]) * 2.5 * N * math.log2(N)
        return dict(bytes=b, flops=f)
    if kind in ("peakmap", "followup"):
        n_fft, N = _n_fft(c["t_obs"], c["t_fft"]), c["fs"] * c["t_fft"]
        nb = 2 * c["half_band"] * c["t_fft"] if kind == "followup" else _bins(c)[1] - _bins(c)[0] + 1
        peaks = 0.0755 * n_fft * nb
        fl = n_fft * (5.0 * N * math.log2(nb + 130) + 8 * N if kind == "followup" else 2.5 * N * math.log2(N))
        return dict(bytes=4.0 * c["fs"] * c["t_obs"] + 8.0 * peaks, flops=fl)
    if kind == "layer":
        l, B, h = c["layer"], c["batch"], c["h"]
        ins, outs = B * h * h * CIN[l], B * (h // STRIDE[l]) ** 2 * COUT[l]
        # forward: input and output; input gradient: two outputs (activation, its gradient) and one
        # input; weight gradient: the same read
        return dict(bytes=2.0 * (ins + (outs if c["mode"] == 0 else 2 * outs)),
                    flops=2.0 * B * _layer_macs(l, h))
    B, hs = c["batch"], (256, 256, 128, 128, 64)
    fwd = sum(2.0 * _layer_macs(l, hs[l]) for l in range(5))
    img, prm = B * 256 * 256 * 4.0, 114561 * 4.0
    if kind == "forward":
        return dict(bytes=img + prm + B * CLASSES * 4.0, flops=B * fwd)
    return dict(bytes=img + 2 * prm, flops=B * (3.0 * fwd - 2.0 * _layer_macs(0, 256)))


# ---- 64-bit values of the network -----------------------------------------------------------------

def _net64(p, img):
    """Logits of images [b, 256, 256, 2]; p: the parameters as one float64 vector (with gradient)."""
    x, o = img.permute(0, 3, 1, 2), 0
    for l in range(5):
        nw = COUT[l] * 9 * CIN[l]
        w = p[o:o + nw].view(COUT[l], 3, 3, CIN[l]).permute(0, 3, 1, 2)
        x = F.conv2d(x, w, p[o + nw:o + nw + COUT[l]], stride=STRIDE[l], padding=1).relu()
        o += nw + COUT[l]
    pooled = x.mean(2)                                                     # over time: [b, c, f]
    wh = p[o:o + 64 * 3 * 64].view(64, 3, 64).permute(0, 2, 1)
    o += 64 * 3 * 64
    y = F.conv1d(pooled, wh, p[o:o + 64], padding=1)                       # [b, d, xt]
    return torch.cat([y.reshape(len(img), -1), p[o + 64].expand(len(img), 1)], 1)


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "layer":
        l = c["layer"]
        w, x, bias, y, dy = (t.double() for t in _layer_inputs(c, seed))
        w, x = w.permute(0, 3, 1, 2), x.permute(0, 3, 1, 2)
        g = (dy * (y > 0)).permute(0, 3, 1, 2)
        if c["mode"] == 0:
            return F.conv2d(x, w, bias, stride=STRIDE[l], padding=1).relu().permute(0, 2, 3, 1)
        if c["mode"] == 1:
            return torch.nn.grad.conv2d_input(x.shape, w, g, stride=STRIDE[l], padding=1).permute(0, 2, 3, 1)
        dw = torch.nn.grad.conv2d_weight(x, w.shape, g, stride=STRIDE[l], padding=1)
        return [dw.permute(0, 2, 3, 1), g.sum((0, 2, 3))]
    if kind not in ("forward", "gradients"):
        return None
    img, labels = _network_inputs(c, seed)
    p = torch.from_numpy(_weights()).double().cuda()
    B, step = c["batch"], 8
    if kind == "forward":
        with torch.no_grad():
            return torch.cat([_net64(p, img[i:i + step].double()) for i in range(0, B, step)])
    p.requires_grad_(True)
    loss = 0.0
    for i in range(0, B, step):
        part = F.cross_entropy(_net64(p, img[i:i + step].double()), labels[i:i + step].long(),
                               reduction="sum") / B
        part.backward()
        loss += float(part)
    return [torch.tensor(loss, dtype=torch.float64), p.grad]
