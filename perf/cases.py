"""The calls this framework is used for, as timed cases: total viewsheds of
one DEM through each single-DEM entry point, batches of tiles, the request
server, and the point viewsheds and visibility maps of a POV list.

The terrain is seeded spectral fractal noise (Hurst exponent 0.6 to 0.9,
rescaled to the stated relief), as everywhere else in this repository; it is
drawn on the GPU here, so that inputs are quick to make.  Handles, servers and
prepared batches are made in prepare(), as a program keeps them between calls.
Every case runs with the library's default tuning unless it says "fp32".
"""
import math
import random

import numpy as np
import torch

import paper_2003_02200_gb300 as tvs

# Directions x cells are spread over the range a user meets: 36 directions
# for a coarse map, 90 / 180 / 360 as the served requests ask for.
SECTORS = (36, 90, 180, 360)

# The most evaluations a drawn total viewshed may have (2000 x 2000 cells,
# 180 directions, unlimited range) and the most for which exact() is quick.
MAX_EVALS = 1.25e12
EXACT_EVALS = 1.6e11


def _map(name, rows, cols, n=180, hurst=0.8, relief=1500.0, step=10.0, h0=1.5, rng=0.0, spikes=0.0,
         entry="device", fp32=False):
    return dict(name=name, kind="map", rows=rows, cols=cols, n=n, hurst=hurst, relief=relief, step=step, h0=h0,
                max_range=rng, spikes=spikes, entry=entry, fp32=fp32)


def _points(name, side, povs, mode, n=180, rng=0.0, h0=1.5):
    return dict(name=name, kind="points", rows=side, cols=side, n=n, hurst=0.8, relief=1500.0, step=10.0, h0=h0,
                max_range=rng, povs=povs, mode=mode)


def listed():
    return [
        # the smallest map of the repository's workloads: one 100 x 100 DEM,
        # where launches and host work count
        _map("map_100", 100, 100, relief=500.0),
        # an odd-sized DEM in host memory, copied in and out by the call
        _map("map_host_333x257", 333, 257, n=90, hurst=0.7, relief=700.0, h0=10.0, entry="host"),
        # an ordinary single map, device buffers
        _map("map_1000", 1000, 1000),
        # the paper's size (its DEM10m-2k), the repository's headline workload
        _map("map_2000", 2000, 2000),
        # the paper's 4000 x 4000 size with a range limit, a 5 m grid and
        # spikes (buildings, masts), a quarter of the large workload's directions
        _map("map_4000_ranged", 4000, 4000, n=90, hurst=0.7, relief=2500.0, step=5.0, h0=10.0, rng=10000.0,
             spikes=0.05),
        # the paper's own single-precision decisions, which a user may choose;
        # an elongated DEM with ragged sides
        _map("map_fp32_1201x777", 1201, 777, fp32=True),
        # many small tiles prepared once and replayed as a CUDA graph, the
        # DEM contents changing between launches
        dict(name="batch_small", kind="batch", tiles=60, lo=64, hi=256, n=180, layout=11, prepared=True),
        # uneven tiles of a survey in one call (sides log-uniform 256 to 1500)
        dict(name="batch_mixed", kind="batch", tiles=12, lo=256, hi=1500, n=180, layout=3, prepared=False),
        # a burst of served requests of different sizes, directions and ranges
        dict(name="serve_burst", kind="serve", requests=12, lo=128, hi=1024, layout=5),
        # the paper's first experiment: 10 observers on the 2000 x 2000 DEM
        _points("points_10", 2000, 10, "sdem"),
        # a long observer list (a siting study), lines through the cells themselves
        _points("points_2000_direct", 2000, 2000, "direct", h0=10.0),
        # which cells 10 observers see
        dict(_points("vismap_10", 2000, 10, "direct"), kind="vismap"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _evals(rows, cols, n, step, max_range):
    """About how many targets the walks of a map visit."""
    w = max(rows, cols)
    k = min(w / 2.0, max_range / step) if max_range > 0.0 else w / 2.0
    return 2.0 * rows * cols * n * 0.8 * k


def draw(rng):
    kind = rng.choice(["map", "map", "map", "map", "batch", "serve", "points", "points", "vismap"])
    step = rng.choice([5.0, 10.0, 30.0])
    h0 = round(rng.uniform(1.5, 30.0), 2)
    hurst = round(rng.uniform(0.6, 0.9), 3)
    if kind == "map":
        rows, cols = _log(rng, 40, 2000), _log(rng, 40, 2000)
        # aspect ratios up to 4
        rows, cols = max(rows, cols // 4), max(cols, rows // 4)
        reach = rng.choice([0.0, 0.0, 5000.0])
        n = rng.choice(SECTORS)
        while _evals(rows, cols, n, step, reach) > MAX_EVALS:
            n //= 2
        side = max(rows, cols)
        entry = rng.choice(["device", "device", "host", "noalloc" if side <= 1000 else "device"])
        fp32 = entry != "noalloc" and rng.random() < 0.2
        c = _map("", rows, cols, n, hurst, round(rng.uniform(200.0, 2500.0), 1), step, h0, reach,
                 rng.choice([0.0, 0.0, 0.05]), entry, fp32)
    elif kind == "batch":
        if rng.random() < 0.5:
            c = dict(kind="batch", tiles=rng.randint(12, 60), lo=64, hi=256, n=rng.choice([90, 180]),
                     layout=rng.randint(100, 10**6), prepared=rng.random() < 0.5)
        else:
            c = dict(kind="batch", tiles=rng.randint(3, 12), lo=256, hi=1200, n=rng.choice([90, 180]),
                     layout=rng.randint(100, 10**6), prepared=rng.random() < 0.5)
    elif kind == "serve":
        c = dict(kind="serve", requests=rng.randint(2, 14), lo=128, hi=1024, layout=rng.randint(100, 10**6))
    else:
        rows, cols = _log(rng, 200, 3000), _log(rng, 200, 3000)
        reach = rng.choice([0.0, 0.0, 5000.0])
        c = dict(kind=kind, rows=rows, cols=cols, n=rng.choice(SECTORS), hurst=hurst, relief=1500.0, step=step,
                 h0=h0, max_range=reach, povs=_log(rng, 1, 1000) if kind == "points" else _log(rng, 1, 30),
                 mode=rng.choice(["sdem", "direct"]) if kind == "points" else "direct")
    c.pop("name", None)
    return c


# ------------------------------------------------------------------ inputs --
def _terrain(rows, cols, hurst, relief, seed, spikes=0.0):
    """Seeded spectral fractal DEM on the GPU, float32."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    fy = torch.fft.fftfreq(rows, device="cuda", dtype=torch.float64)[:, None]
    fx = torch.fft.rfftfreq(cols, device="cuda", dtype=torch.float64)[None, :]
    f = torch.sqrt(fx * fx + fy * fy)
    f[0, 0] = 1.0
    amp = f ** (-(hurst + 1.0))
    amp[0, 0] = 0.0
    noise = torch.randn(2, rows, cols // 2 + 1, device="cuda", dtype=torch.float64, generator=g)
    z = torch.fft.irfft2(torch.complex(noise[0], noise[1]) * amp, s=(rows, cols))
    z = (z - z.min()) / (z.max() - z.min()) * relief
    if spikes > 0.0:
        u = torch.rand(2, rows, cols, device="cuda", dtype=torch.float64, generator=g)
        z = z + torch.where(u[0] < spikes, 20.0 + 40.0 * u[1], torch.zeros_like(u[1]))
    return z.to(torch.float32).contiguous()


def _povs(case, seed):
    r = np.random.default_rng(seed)
    return np.stack([r.integers(0, case["rows"], case["povs"]), r.integers(0, case["cols"], case["povs"])],
                    axis=1).astype(np.int32)


def _jobs(case):
    """The tiles of a batch or the requests of a burst: their shapes and
    parameters follow from the case, their terrain from the seed."""
    r = random.Random(case["layout"])
    jobs = []
    for _ in range(case["tiles"] if case["kind"] == "batch" else case["requests"]):
        a = _log(r, case["lo"], case["hi"])
        b = max(case["lo"], int(a * r.uniform(0.7, 1.0)))
        rows, cols = (a, b) if r.random() < 0.5 else (b, a)
        jobs.append(dict(rows=rows, cols=cols, hurst=r.uniform(0.6, 0.9), relief=r.uniform(200.0, 1500.0),
                         step=r.choice([5.0, 10.0, 30.0]), h0=r.uniform(1.5, 30.0),
                         n=case["n"] if case["kind"] == "batch" else r.choice([90, 180]),
                         max_range=0.0 if case["kind"] == "batch" else r.choice([0.0, 5000.0])))
    return jobs


def _pinned(shape):
    return torch.empty(shape, dtype=torch.float32, pin_memory=True).numpy()


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind == "map":
        dem = _terrain(case["rows"], case["cols"], case["hurst"], case["relief"], seed, case["spikes"])
        if case["entry"] == "host":
            st["dem"], st["out"] = _pinned(dem.shape), _pinned(dem.shape)
            st["dem"][:] = dem.cpu().numpy()
        else:
            st["dem"], st["out"] = dem, torch.empty_like(dem)
        if case["entry"] != "noalloc":
            st["ctx"] = tvs.Context(0)
            if case["fp32"]:
                st["ctx"].set_tuning(fp32_decisions=1)
    elif kind == "batch":
        ctx = tvs.Context(0)
        st["jobs"] = []
        for q, j in enumerate(_jobs(case)):
            dem = _terrain(j["rows"], j["cols"], j["hurst"], j["relief"], seed * 1000 + q)
            st["jobs"].append(dict(dem=dem, out=torch.empty_like(dem), step_m=j["step"], obs_height_m=j["h0"],
                                   n_sectors=j["n"], max_range_m=j["max_range"]))
        # the batch comes before its handle, so that it is given back first
        if case["prepared"]:
            st["batch"] = ctx.prepare_batch(st["jobs"])
        st["ctx"] = ctx
    elif kind == "serve":
        st["server"] = tvs.Server(0, hbm_budget_bytes=8 << 30)
        st["jobs"] = _jobs(case)
        for q, j in enumerate(st["jobs"]):
            j["dem"], j["out"] = _pinned((j["rows"], j["cols"])), _pinned((j["rows"], j["cols"]))
            j["dem"][:] = _terrain(j["rows"], j["cols"], j["hurst"], j["relief"], seed * 1000 + q).cpu().numpy()
    else:
        st["dem"] = _terrain(case["rows"], case["cols"], case["hurst"], case["relief"], seed)
        st["povs"] = _povs(case, seed)
        st["ctx"] = tvs.Context(0)
    return st


def run(state):
    c = state["case"]
    if c["kind"] == "map":
        a = (state["dem"], c["step"], c["h0"], c["n"], c["max_range"])
        if c["entry"] == "host":
            return state["ctx"].total_viewshed(*a, out=state["out"])
        if c["entry"] == "noalloc":
            return tvs.total_viewshed_device_noalloc(*a, out=state["out"])
        return state["ctx"].total_viewshed_device(*a, out=state["out"])
    if c["kind"] == "batch":
        if c["prepared"]:
            state["batch"].launch()
        else:
            state["ctx"].total_viewshed_batch(state["jobs"])
        return [j["out"] for j in state["jobs"]]
    if c["kind"] == "serve":
        s = state["server"]
        tickets = [s.submit(j["dem"], j["step"], j["h0"], j["n"], j["max_range"], out=j["out"])
                   for j in state["jobs"]]
        outs = []
        for t in tickets:
            outs.append(s.wait(t))
            s.forget(t)
        return outs
    a = (state["dem"], c["step"], c["h0"], c["n"], c["max_range"], state["povs"])
    if c["kind"] == "points":
        return state["ctx"].viewshed_points(*a, mode=c["mode"])
    return state["ctx"].visibility_map(*a)


def work(case):
    """Bytes: each DEM cell read once, each output written once.  Operations,
    a lower bound that holds on any terrain: per cell and direction one
    relocation blend (3), for each of the two walks the slope of one target,
    its comparison and the running maximum (4), and the blend back with its
    weighted sum (4).  Every target that is visible costs 4 more; how many
    are depends on the terrain, so they are left out."""
    if case["kind"] in ("batch", "serve"):
        b = f = 0.0
        for j in _jobs(case):
            cells = float(j["rows"]) * j["cols"]
            b += 8.0 * cells
            f += 15.0 * cells * j["n"]
        return {"bytes": b, "flops": f}
    cells = float(case["rows"]) * case["cols"]
    if case["kind"] == "map":
        return {"bytes": 8.0 * cells, "flops": 15.0 * cells * case["n"]}
    # a POV list touches at most the cells of its lines (both rows that a
    # sample blends), and walks each line both ways
    lines = float(case["povs"]) * case["n"] * (2 if case["mode"] == "sdem" else 1)
    reach = min(1.0, case["max_range"] / (case["step"] * max(case["rows"], case["cols"]))) \
        if case["max_range"] > 0.0 else 1.0
    touched = min(cells, 2.0 * lines * reach * min(case["rows"], case["cols"]))
    if case["kind"] == "points":
        return {"bytes": 4.0 * touched + 4.0 * case["povs"], "flops": 15.0 * lines}
    return {"bytes": 4.0 * touched + 4.0 * cells, "flops": 15.0 * lines + 4.0 * cells * case["povs"]}


# ------------------------------------------------- 64-bit values, plain torch --
def _directions(rows, cols, n, step, max_range):
    """The n directions k pi / n: the D4 view they are walked in, the tangent
    as a 32.32 fixed-point number and the walk limit in steps."""
    out = []
    for k in range(n):
        frame = 0 if 4 * k < n else 1 if 4 * k < 2 * n else 2 if 4 * k < 3 * n else 3
        m = (2 * k, n - 2 * k, 2 * k - n, 2 * n - 2 * k)[frame]
        t = math.tan(math.pi * m / (2.0 * n)) * 4294967296.0
        fx = int(math.floor(t + 0.5))
        tt = fx / 4294967296.0
        g = 1.0 + tt * tt
        w = cols if frame in (0, 3) else rows
        limit = w if not (max_range > 0.0) else int(min(w, math.floor(max_range / (step * math.sqrt(g)))))
        out.append((frame, fx, g, limit))
    return out


def _view(z, frame):
    if frame == 0:
        return z
    if frame == 1:
        return z.t()
    if frame == 2:
        return z.t().flip(1)
    return z.flip(0)


def _unview(v, frame):
    if frame == 0:
        return v
    if frame == 1:
        return v.t()
    if frame == 2:
        return v.flip(1).t()
    return v.flip(0)


def _walk(z, ok, h, limits):
    """Measures of the walks toward +j of every sample of lines z (k, R, W)
    whose samples ok are usable (a contiguous stretch of each line):
    1 + the sum of 2 d + 1 over the visible targets but the last one."""
    W = z.shape[2]
    nxt = torch.zeros_like(ok)
    nxt[:, :, :-1] = ok[:, :, 1:]
    tgt = torch.where(ok & nxt, z, torch.full_like(z, -math.inf))   # the last target adds no area
    top = torch.full_like(z, -math.inf)
    acc = torch.zeros(z.shape, dtype=torch.int32, device=z.device)
    dist = torch.arange(W + 1, dtype=torch.float64, device=z.device)   # a tensor divisor: one rounding
    for d in range(1, min(W, max(limits))):
        live = [q for q, lim in enumerate(limits) if d < lim]
        lo, hi = min(live), max(live) + 1
        if any(limits[q] <= d for q in range(lo, hi)):      # limits differ inside the slice
            cut = torch.tensor([limits[q] > d for q in range(lo, hi)], device=z.device)[:, None, None]
        else:
            cut = None
        th = (tgt[lo:hi, :, d:] - h[lo:hi, :, :W - d]).div_(dist[d])
        m = top[lo:hi, :, :W - d]
        v = th > m
        if cut is not None:
            v &= cut
        acc[lo:hi, :, :W - d].add_(v, alpha=2 * d + 1)
        torch.maximum(m, th, out=m)
    lim = torch.tensor(limits, device=z.device)[:, None, None]
    any_target = ok & nxt & (lim >= 1)
    return torch.where(any_target, acc + 1, torch.zeros_like(acc)).to(torch.float64)


def _exact_map(dem, n, step, h0, max_range):
    z = dem.to(torch.float64)
    rows, cols = z.shape
    total = torch.zeros_like(z)
    dirs = _directions(rows, cols, n, step, max_range)
    for frame in range(4):
        V = _view(z, frame).contiguous()
        H, W = V.shape
        mine = sorted((d for d in dirs if d[0] == frame), key=lambda d: d[3])
        per = max(1, int(2.5e7 / ((H + W) * W)))
        back = torch.zeros_like(V)
        j = torch.arange(W, device=z.device)
        for q0 in range(0, len(mine), per):
            part = mine[q0:q0 + per]
            fx = torch.tensor([d[1] for d in part], dtype=torch.int64, device=z.device)[:, None]
            y = j[None, :] * fx
            dest, fr = y >> 32, y & 0xFFFFFFFF
            D = int(dest.max())
            b = torch.arange(-D, H, device=z.device)
            a = b[None, :, None] + dest[:, None, :]
            frac = (fr != 0)[:, None, :]
            ok = (a >= 0) & torch.where(frac, a <= H - 2, a <= H - 1)
            ac = a.clamp(0, H - 1)
            r = (fr.to(torch.float64) / 4294967296.0)[:, None, :]
            jj = j[None, None, :].expand_as(ac)
            s = (1.0 - r) * V[ac, jj] + r * V[(ac + 1).clamp(max=H - 1), jj]
            lims = [d[3] for d in part]
            h = s + h0
            cv = _walk(s, ok, h, lims) + _walk(s.flip(2), ok.flip(2), h.flip(2), lims).flip(2)
            cv = torch.where(ok, cv, torch.zeros_like(cv))
            for q, d in enumerate(part):
                i = torch.arange(H, device=z.device)[:, None]
                p = i - dest[q][None, :] + D
                hi = cv[q][p, j[None, :].expand_as(p)]
                lo = cv[q][(p - 1).clamp(min=0), j[None, :].expand_as(p)]
                f = (fr[q] != 0)[None, :]
                rr = r[q]
                hi_ok, lo_ok = ~f | (i <= H - 2), f & (i >= 1)
                val = torch.where(hi_ok & lo_ok, (1.0 - rr) * hi + rr * lo, torch.where(hi_ok, hi, lo))
                back += d[2] * val
        total += _unview(back, frame)
    return (total * (math.pi / (2.0 * n)) * step * step).to(torch.float64)


def _line_measure(z, ok, j0, j, limit, h):
    """Forward plus backward measures of lines z (..., W) from column j0."""
    out = torch.zeros(z.shape[:-1], dtype=torch.float64, device=z.device)
    for side in (1, -1):
        d = (j - j0[..., None]) * side
        live = ok & (d >= 1) & (d <= limit[..., None])
        cnt = live.sum(-1)
        th = torch.where(live, (z - h[..., None]) / d.clamp(min=1), torch.full_like(z, -math.inf))
        if side < 0:
            th, d = th.flip(-1), d.flip(-1)
        before = torch.full_like(th, -math.inf)
        before[..., 1:] = torch.cummax(th, -1).values[..., :-1]
        v = (th > before) & (d < cnt[..., None])
        out += torch.where(cnt >= 1, 1.0 + (v * (2 * d + 1)).sum(-1).to(torch.float64), torch.zeros_like(out))
    return out


def _exact_points(dem, povs, n, step, h0, max_range, mode):
    z = dem.to(torch.float64)
    rows, cols = z.shape
    res = torch.zeros(len(povs), dtype=torch.float64, device=z.device)
    dirs = _directions(rows, cols, n, step, max_range)
    P = torch.as_tensor(povs, device=z.device).to(torch.int64)
    for frame in range(4):
        V = _view(z, frame).contiguous()
        H, W = V.shape
        mine = [d for d in dirs if d[0] == frame]
        if not mine:
            continue
        fx = torch.tensor([d[1] for d in mine], dtype=torch.int64, device=z.device)[None, :, None]
        g = torch.tensor([d[2] for d in mine], dtype=torch.float64, device=z.device)
        lim = torch.tensor([d[3] for d in mine], dtype=torch.int64, device=z.device)
        j = torch.arange(W, device=z.device)
        per = max(1, int(2.0e7 / (W * len(mine))))
        for q0 in range(0, len(povs), per):
            p = P[q0:q0 + per]
            i0 = (p[:, 0], p[:, 1], p[:, 1], H - 1 - p[:, 0])[frame]
            j0 = (p[:, 1], p[:, 0], W - 1 - p[:, 0], p[:, 1])[frame]
            i0, j0 = i0[:, None].expand(-1, len(mine)), j0[:, None].expand(-1, len(mine))
            y0 = j0 * fx[..., 0]
            fr0 = (y0 & 0xFFFFFFFF) if mode == "sdem" else torch.zeros_like(y0)
            cvs = []
            for v in range(2 if mode == "sdem" else 1):
                y = (j * fx) if mode == "sdem" else (j - j0[..., None]) * fx
                base = (i0 - (y0 >> 32) - v) if mode == "sdem" else i0
                a = base[..., None] + (y >> 32)
                fr = (y & 0xFFFFFFFF).expand_as(a)
                ok = (a >= 0) & torch.where(fr != 0, a <= H - 2, a <= H - 1)
                ac, jj = a.clamp(0, H - 1), j.expand_as(a)
                r = fr.to(torch.float64) / 4294967296.0
                s = (1.0 - r) * V[ac, jj] + r * V[(ac + 1).clamp(max=H - 1), jj]
                h = torch.gather(s, 2, j0[..., None])[..., 0] + h0
                cvs.append(_line_measure(s, ok, j0, j, lim[None, :].expand_as(j0), h))
            val = cvs[0]
            if mode == "sdem":
                f, r0 = fr0 != 0, fr0.to(torch.float64) / 4294967296.0
                hi_ok, lo_ok = ~f | (i0 <= H - 2), f & (i0 >= 1)
                val = torch.where(hi_ok & lo_ok, (1.0 - r0) * cvs[0] + r0 * cvs[1],
                                  torch.where(hi_ok, cvs[0], cvs[1]))
            res[q0:q0 + per] += (val * g).sum(1)
    return res * (math.pi / (2.0 * n)) * step * step


def exact(case, seed):
    """What run() returns in 64-bit arithmetic.  None for the visibility map
    (whole numbers), for single-precision decisions (their values are defined
    by the rounding), and where it would take too long."""
    kind = case["kind"]
    if kind == "vismap" or case.get("fp32"):
        return None
    if kind == "map":
        if _evals(case["rows"], case["cols"], case["n"], case["step"], case["max_range"]) > EXACT_EVALS:
            return None
        dem = _terrain(case["rows"], case["cols"], case["hurst"], case["relief"], seed, case["spikes"])
        return _exact_map(dem, case["n"], case["step"], case["h0"], case["max_range"]).cpu()
    if kind in ("batch", "serve"):
        left, outs = EXACT_EVALS, []
        for q, j in enumerate(_jobs(case)):
            e = _evals(j["rows"], j["cols"], j["n"], j["step"], j["max_range"])
            if e > left:
                outs.append(None)
                continue
            left -= e
            dem = _terrain(j["rows"], j["cols"], j["hurst"], j["relief"], seed * 1000 + q)
            outs.append(_exact_map(dem, j["n"], j["step"], j["h0"], j["max_range"]).cpu())
        return outs
    if 4.0 * case["povs"] * case["n"] * max(case["rows"], case["cols"]) > 6e9:
        return None
    dem = _terrain(case["rows"], case["cols"], case["hurst"], case["relief"], seed)
    return _exact_points(dem, _povs(case, seed), case["n"], case["step"], case["h0"], case["max_range"],
                         case["mode"]).cpu()
