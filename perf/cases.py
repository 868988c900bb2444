"""The work that users of the library have it do, as measurable cases.

A case is a telescope layout, an observation and one call (or the few calls of one
imaging or calibration step) through the public entry points of
``paper_1909_07226_gb300.idg``.  ``prepare`` makes what a program has in hand before the
call -- visibilities of a point-source sky, flags, smooth Jones screens, model grids, the
plan -- from a seed; ``run`` is one pass; ``exact`` is the same result in 64 bits from
the definition of the method, in plain numpy and torch (its own partition, direct sums,
FFTs).

Kinds:
  grid, degrid   idg_grid into a zeroed grid, idg_degrid of a model grid
  cycle          one major cycle: degrid the model, subtract, grid the residual
  batch          idg_batch over several jobs of different shapes: grid, then degrid
  gradient       residuals, cost and A-term gradient of one calibration step
  image          grid -> image and image -> grid, the ends of a major cycle
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1909_07226_gb300 import idg
from paper_1909_07226_gb300 import synthetic as syn

SPEED_OF_LIGHT = 299792458.0
BETA = 7.0
N_SOURCES = 8


def _case(name=None, **kw):
    c = dict(kind="grid", array="core", layout=1, stations=48, n_t=256, dt=1.0, n_chan=16, f_lo=130e6, df=1e6, L=32,
             N=4096, cell=1.0e-5, slot_len=128, t_max=128, w_step=0.0, flag_p=0.0, screens=True, adder="atomic",
             phasor="sincos", fft="fp32")
    if name is not None:
        c["name"] = name
    c.update(kw)
    return c


def listed():
    tiny = dict(array="disc", stations=8, n_t=64, dt=10.0, n_chan=8, f_lo=140e6, L=24, N=512, cell=2.0e-4, slot_len=64,
                t_max=16, screens=False)
    return [
        # a handful of stations for a few minutes: quick looks, tests, the smallest calls, where
        # launches and latency count
        _case("tiny_cycle", kind="cycle", **tiny),
        # a LOFAR-like observation with A-terms every 128 s, the workload the library is quoted on
        _case("lofar_grid", kind="grid", n_t=4096),
        _case("lofar_degrid", kind="degrid", n_t=4096),
        # fast ionosphere: A-terms every 16 s cut the visibilities into many short subgrids;
        # 5 % of the data flagged, an odd number of timesteps
        _case("ionosphere_grid", kind="grid", n_t=1021, slot_len=16, flag_p=0.05),
        _case("ionosphere_degrid", kind="degrid", n_t=1021, slot_len=16, flag_p=0.05),
        # snapshots of other arrays: ragged sizes, smaller subgrids, wide fields whose w-term
        # needs its own offset per subgrid, without A-terms or (second) with W-layers
        _case("snapshot_l16_grid", kind="grid", array="gauss", layout=3, stations=37, n_t=611, n_chan=19, f_lo=117e6,
              df=0.2e6, L=16, N=2048, cell=0.0, slot_len=611, flag_p=0.11, screens=False),
        _case("snapshot_l24_degrid", kind="degrid", array="gauss", layout=4, stations=31, n_t=413, n_chan=13,
              f_lo=151e6, df=0.2e6, L=24, N=1024, cell=0.0, slot_len=200, w_step=40.0, flag_p=0.07),
        # many imaging requests of different shapes served together
        _case("snapshot_batch", kind="batch", layout=5, jobs=8, scale_t=0.4),
        # results that must be the same bit for bit on every run
        _case("deterministic_grid", kind="grid", n_t=512, slot_len=16, adder="sorted"),
        # the precision options: phasors by channel recurrence, tensor-core transform,
        # compensated adder
        _case("precision_cycle", kind="cycle", n_t=128, slot_len=16, phasor="recurrence", fft="tc_split",
              adder="compensated"),
        # the full-size image transforms at the ends of a major cycle
        _case("image_steps", kind="image", n_t=16, N=4096, slot_len=16, screens=False),
        # one iteration of a calibration with the A-terms as free parameters
        _case("calibration_step", kind="gradient", n_t=512, flag_p=0.03),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    form = rng.choice(["tiny", "core", "core", "short", "snapshot", "snapshot", "snapshot", "batch", "precise", "image",
                       "calibration"])
    lay = rng.randrange(1 << 20)
    if form == "tiny":
        n_t = rng.randint(24, 100)
        return _case(kind=rng.choice(["cycle", "grid", "degrid"]), array="disc", layout=lay, stations=rng.randint(5, 12),
                     n_t=n_t, dt=10.0, n_chan=rng.randint(3, 16), f_lo=140e6, L=24, N=512, cell=1.5e-4, slot_len=n_t,
                     t_max=rng.choice([8, 16, 32]), screens=False)
    if form == "core":
        return _case(kind=rng.choice(["grid", "degrid"]), layout=lay, stations=rng.randint(24, 48),
                     n_t=_log_int(rng, 100, 3000), n_chan=rng.randint(7, 16), slot_len=rng.choice([64, 128, 200]),
                     flag_p=rng.choice([0.0, 0.1]))
    if form == "short":
        return _case(kind=rng.choice(["grid", "degrid"]), layout=lay, stations=rng.randint(24, 48),
                     n_t=_log_int(rng, 100, 900), n_chan=rng.randint(7, 16), slot_len=rng.choice([8, 16, 25]),
                     flag_p=rng.choice([0.0, 0.1]))
    if form == "snapshot":
        n_t = _log_int(rng, 64, 1024)
        N = rng.choice([1024, 2048, 4096])
        layers = N == 1024 and rng.random() < 0.5
        return _case(kind=rng.choice(["grid", "degrid"]), array="gauss", layout=lay, stations=rng.randint(12, 64), n_t=n_t,
                     n_chan=rng.randint(4, 32), f_lo=1e6 * rng.randint(100, 190), df=0.2e6, L=rng.choice([16, 24, 32]),
                     N=N, cell=0.0, slot_len=n_t, w_step=50.0 if layers else 0.0, flag_p=rng.uniform(0.0, 0.2),
                     screens=rng.random() < 0.5)
    if form == "batch":
        return _case(kind="batch", layout=lay, jobs=rng.randint(2, 6), scale_t=rng.uniform(0.1, 0.4))
    if form == "precise":
        sorted_adder = rng.random() < 0.5
        return _case(kind=rng.choice(["grid", "cycle"]), layout=lay, stations=rng.randint(24, 48),
                     n_t=_log_int(rng, 48, 150), slot_len=rng.choice([16, 64]),
                     adder="sorted" if sorted_adder else rng.choice(["atomic", "compensated"]),
                     phasor=rng.choice(["sincos", "recurrence"]), fft=rng.choice(["fp32", "tc_split"]))
    if form == "image":
        N = rng.choice([512, 1024, 2048])
        return _case(kind="image", layout=lay, n_t=16, slot_len=16, screens=False, N=N, cell=4.0e-2 / N,
                     w_step=rng.choice([0.0, 4000.0]))
    return _case(kind="gradient", layout=lay, stations=rng.randint(16, 40), n_t=_log_int(rng, 64, 400),
                 n_chan=rng.randint(7, 16), slot_len=rng.choice([32, 128]), flag_p=rng.choice([0.0, 0.05]))


# ---------------------------------------------------------------------------------------
# observations


def _workloads(case, seed):
    """The observation (or, for a batch, the observations): uvw, frequencies, baselines.
    The telescope belongs to the case, the hour angle to the seed."""
    if case["kind"] == "batch":
        jobs = syn.make_batched_jobs(case["jobs"], seed=case["layout"], scale_t=case["scale_t"])
        ha = np.random.default_rng(seed).uniform(-0.05, 0.05)
        for wl in jobs:      # the same arrays a little earlier or later
            u, v, w = wl.uvw_m[..., 0], wl.uvw_m[..., 1], wl.uvw_m[..., 2]
            wl.uvw_m = np.ascontiguousarray(np.stack([u * math.cos(ha) - v * math.sin(ha),
                                                      u * math.sin(ha) + v * math.cos(ha), w], axis=2))
        return jobs
    rng = np.random.default_rng(case["layout"])
    n_st = case["stations"]
    if case["array"] == "disc":
        enu = syn.stations_uniform_disc(rng, n_st, 2000.0)
    elif case["array"] == "gauss":
        enu = np.concatenate([rng.normal(0.0, 3000.0, size=(n_st, 2)), np.zeros((n_st, 1))], axis=1)
    else:
        n_remote = n_st // 6
        enu = syn.stations_core_remote(rng, n_st - n_remote, 3000.0, n_remote, 5000.0, 50000.0)
    # with W-layers the number of layers, so the grid's shape, goes with the hour angle
    start = np.random.default_rng(case["layout"] if case["w_step"] else seed).uniform(-0.3, 0.1)
    bl = syn.all_baselines(n_st)
    uvw = syn.earth_rotation_uvw(enu, bl, syn.hour_angles(case["n_t"], case["dt"], start_rad=start),
                                 math.radians(syn.SOURCE_DEC_DEG), math.radians(syn.LOFAR_LATITUDE_DEG))
    freqs = syn.channel_centres(case["f_lo"], case["df"], case["n_chan"])
    L, N, cell = case["L"], case["N"], case["cell"]
    if not cell:             # the longest baseline lands N / 2.2 pixels from the centre
        cell = 1.0 / (2.2 * float(np.max(np.hypot(uvw[..., 0], uvw[..., 1]))) * freqs[-1] / SPEED_OF_LIGHT)
    offs = np.append(np.arange(0, case["n_t"], case["slot_len"]), case["n_t"]).astype(np.int32)
    return [syn.Workload("case", uvw, freqs, bl, offs, n_st, L, N, cell, case["w_step"], BETA, case["t_max"],
                         syn.separable_taper(syn.pswf_1d(L, BETA)))]


def _generator(seed, k):
    return torch.Generator(device="cuda").manual_seed(1000 * int(seed) + k)


def _sky(wl, gen):
    """Point sources in the central 60 % of the field: l, m [S] and 2 x 2 brightness [S][4]."""
    lm = (torch.rand((2, N_SOURCES), generator=gen, device="cuda", dtype=torch.float64) - 0.5) * 0.6 * wl.image_size
    flux = 0.1 + 0.9 * torch.rand(N_SOURCES, generator=gen, device="cuda")
    pol = 0.05 * torch.randn((N_SOURCES, 4), generator=gen, device="cuda", dtype=torch.complex64)
    pol[:, 0] += 1.0
    pol[:, 3] += 1.0
    return lm[0], lm[1], flux[:, None] * pol


def _visibilities(wl, gen):
    """The sky's visibilities with thermal noise of the order of the sources."""
    l, m, B = _sky(wl, gen)
    n1 = torch.sqrt(1.0 - l * l - m * m) - 1.0
    fc = torch.from_numpy(wl.freqs_hz / SPEED_OF_LIGHT).cuda()
    vis = torch.empty((wl.n_bl, wl.n_t, wl.n_chan, 4), dtype=torch.complex64, device="cuda")
    step = max(1, (1 << 25) // (wl.n_t * wl.n_chan * N_SOURCES))
    lmn = torch.stack([l, m, n1])
    for b in range(0, wl.n_bl, step):
        geo = torch.from_numpy(wl.uvw_m[b:b + step]).cuda() @ lmn                       # [b][t][S] metres
        turns = geo[:, :, None, :] * fc[None, None, :, None]
        ph = (-2.0 * math.pi * (turns - torch.round(turns))).float()
        vis[b:b + step] = torch.polar(torch.ones_like(ph), ph) @ B
        vis[b:b + step] += 0.5 * torch.randn(vis[b:b + step].shape, generator=gen, device="cuda", dtype=torch.complex64)
    return vis


def _model_grid(wl, n_w, gen):
    """The uv grid of a point-source model (plane waves) with a diffuse part that fills the
    field, the same sky in every layer."""
    l, m, B = _sky(wl, gen)
    q = (torch.arange(wl.grid_size, device="cuda", dtype=torch.float64) - wl.grid_size / 2) / wl.image_size
    wave = lambda x: torch.polar(torch.ones_like(q[:, None] * x), -2.0 * math.pi * torch.remainder(q[:, None] * x, 1.0))
    wu, wv = wave(l).to(torch.complex64), wave(m).to(torch.complex64)
    one = torch.stack([(wv * B[:, p]) @ wu.T for p in range(4)], dim=-1)
    one += 0.5 * torch.randn(one.shape, generator=gen, device="cuda", dtype=torch.complex64)
    return one.expand(n_w, -1, -1, -1).contiguous()


def _sky_image(N, gen):
    """A model image: 500 point sources away from the edges."""
    sky = torch.zeros((N, N, 4), dtype=torch.complex64, device="cuda")
    at = torch.randint(N // 8, N - N // 8, (2, 500), generator=gen, device="cuda")
    sky[at[0], at[1]] = 1.0 + torch.rand((500, 4), generator=gen, device="cuda").to(sky.dtype)
    return sky


def _screens(wl, gen):
    """Smooth random Jones matrices per slot and station on the subgrid lattice, complex64."""
    shape = (wl.n_slots, wl.n_stations, 2, 6)
    rand = lambda: (lambda r: r / r.abs().sum(-1, keepdim=True))(torch.randn(shape, generator=gen, device="cuda"))
    L = wl.subgrid_size
    x = (torch.arange(L, device="cuda") - L / 2) / (L / 2)
    X, Y = x[None, :].expand(L, L), x[:, None].expand(L, L)
    basis = torch.stack([torch.ones_like(X), X, Y, X * X, X * Y, Y * Y]).reshape(6, L * L)
    g = torch.polar(1.0 + 0.1 * (rand() @ basis), rand() @ basis)                        # [slot][st][2][pixel]
    leak = 0.035 * torch.randn((wl.n_slots, wl.n_stations, 2, 1), generator=gen, device="cuda", dtype=torch.complex64)
    leak = leak.expand(-1, -1, -1, L * L)
    A = torch.stack([g[:, :, 0], leak[:, :, 0], leak[:, :, 1], g[:, :, 1]], dim=-1)
    return A.reshape(wl.n_slots, wl.n_stations, L, L, 4).contiguous()


def _inputs(case, wl, seed, k, n_w):
    """The device buffers of one observation."""
    gen = _generator(seed, k)
    kind = case["kind"]
    d = dict(flags=None, aterms=None)
    flag_p = wl.flag_p if kind == "batch" else case["flag_p"]
    if flag_p > 0:
        d["flags"] = (torch.rand((wl.n_bl, wl.n_t, wl.n_chan), generator=gen, device="cuda") < flag_p).to(torch.uint8)
    if kind != "batch" and case["screens"]:
        d["aterms"] = _screens(wl, gen)
    d["taper"] = torch.from_numpy(wl.taper).cuda()
    if kind in ("degrid", "cycle", "gradient", "batch", "image"):
        d["model"] = _model_grid(wl, n_w, gen)
    if kind in ("grid", "cycle", "gradient", "batch"):
        d["vis"] = _visibilities(wl, gen)
    return d


def _options(case):
    return dict(adder_mode=["atomic", "compensated", "sorted"].index(case["adder"]),
                precision_mode=["sincos", "recurrence"].index(case["phasor"]),
                fft_mode=["fp32", "tc_split"].index(case["fft"]))


def prepare(case, seed):
    kind = case["kind"]
    states = []
    for k, wl in enumerate(_workloads(case, seed)):
        plan = idg.plan_from_workload(wl, **(_options(case) if kind != "batch" else {}))
        n_w, N = plan.n_w_layers, wl.grid_size
        s = dict(kind=kind, plan=plan, **_inputs(case, wl, seed, k, n_w))
        if kind in ("grid", "cycle", "batch"):
            s["grid"] = torch.zeros((n_w, N, N, 4), dtype=torch.complex64, device="cuda")
        if kind in ("degrid", "cycle", "gradient", "batch"):
            s["vis_out"] = torch.empty((wl.n_bl, wl.n_t, wl.n_chan, 4), dtype=torch.complex64, device="cuda")
        if kind == "gradient":
            s["gradient"] = torch.zeros_like(s["aterms"])
            s["cost"] = torch.zeros(1, dtype=torch.float64, device="cuda")
        if kind == "image":
            s["window"] = syn.pswf_1d(wl.subgrid_size, BETA)
            s["image"] = torch.empty((N, N, 4), dtype=torch.complex64, device="cuda")
            s["grid"] = torch.empty((n_w, N, N, 4), dtype=torch.complex64, device="cuda")
            s["sky"] = _sky_image(N, _generator(seed, 99))
        states.append(s)
    if kind != "batch":
        return states[0]
    plans = [s["plan"] for s in states]
    take = lambda s, vis, out, grid: dict(vis=s[vis] if vis else None, vis_out=s[out] if out else None, flags=s["flags"],
                                          aterms=s["aterms"], taper=s["taper"], grid=s[grid])
    return dict(kind=kind, jobs=states,
                gridder=idg.Batch(plans, [take(s, "vis", None, "grid") for s in states], graph=True),
                degridder=idg.Batch(plans, [take(s, None, "vis_out", "model") for s in states], graph=True))


def run(state):
    s, kind = state, state["kind"]
    if kind == "grid":
        s["grid"].zero_()
        idg.grid(s["plan"], s["vis"], s["flags"], s["aterms"], s["taper"], s["grid"])
        return s["grid"]
    if kind == "degrid":
        idg.degrid(s["plan"], s["model"], s["flags"], s["aterms"], s["taper"], s["vis_out"])
        return s["vis_out"]
    if kind == "cycle":
        idg.degrid(s["plan"], s["model"], s["flags"], s["aterms"], s["taper"], s["vis_out"])
        torch.sub(s["vis"], s["vis_out"], out=s["vis_out"])
        s["grid"].zero_()
        idg.grid(s["plan"], s["vis_out"], s["flags"], s["aterms"], s["taper"], s["grid"])
        return {"residual": s["vis_out"], "grid": s["grid"]}
    if kind == "batch":
        for j in s["jobs"]:
            j["grid"].zero_()
        s["gridder"].grid()
        s["degridder"].degrid()
        return {"grid": [j["grid"] for j in s["jobs"]], "vis": [j["vis_out"] for j in s["jobs"]]}
    if kind == "gradient":
        s["gradient"].zero_()
        s["cost"].zero_()
        idg.aterm_gradient(s["plan"], s["model"], s["vis"], s["flags"], s["aterms"], s["taper"], s["vis_out"],
                           s["gradient"], s["cost"])
        return {"residual": s["vis_out"], "gradient": s["gradient"], "cost": s["cost"]}
    idg.image_from_grid(s["plan"], s["model"], s["window"], s["image"])
    idg.grid_from_image(s["plan"], s["sky"], s["window"], s["grid"])
    return {"image": s["image"], "grid": s["grid"]}


def work(case):
    """Bytes: every input read and every output written once.  Flops: the complex
    multiply-adds of the direct sums, 4 polarisations x L^2 pixels per visibility, and
    5 N^2 log2(N^2) per polarisation of the image transforms."""
    total = dict(bytes=0.0, flops=0.0)
    kind = case["kind"]
    for wl in _workloads(case, 0):
        w = wl.uvw_m[..., 2]
        span = (w.max() * wl.freqs_hz[-1] - min(0.0, w.min()) * wl.freqs_hz[-1]) / SPEED_OF_LIGHT
        n_w = 1 if not wl.w_step else 1 + math.ceil(span / wl.w_step)
        grid = 32.0 * n_w * wl.grid_size ** 2
        if kind == "image":
            image = 32.0 * wl.grid_size ** 2
            total["bytes"] += 2 * (grid + image)
            total["flops"] += 2 * n_w * 4 * 5 * wl.grid_size ** 2 * 2 * math.log2(wl.grid_size)
            continue
        flagged = kind == "batch" or case["flag_p"] > 0
        screens = 32.0 * wl.n_slots * wl.n_stations * wl.subgrid_size ** 2 if kind != "batch" and case["screens"] else 0.0
        coords = 24.0 * wl.n_bl * wl.n_t + (wl.n_vis if flagged else 0.0) + screens
        sums = 32.0 * wl.subgrid_size ** 2 * wl.n_vis
        if kind in ("grid", "degrid"):
            total["bytes"] += coords + 32.0 * wl.n_vis + grid
            total["flops"] += sums
        elif kind in ("cycle", "batch"):
            total["bytes"] += coords + 64.0 * wl.n_vis + 2 * grid
            total["flops"] += 2 * sums
        else:
            total["bytes"] += coords + 64.0 * wl.n_vis + grid + screens
            total["flops"] += 2 * sums
    return total


# ---------------------------------------------------------------------------------------
# the definition in 64 bits: partition (numpy), direct sums and transforms (torch)


class _Subgrids:
    """Subgrids of an observation: per baseline, A-term slot and channel group, runs of
    timesteps whose support fits (fields: one array entry per subgrid)."""

    def __init__(self, wl):
        L, N, S = wl.subgrid_size, wl.grid_size, wl.grid_size * wl.cell_size
        smax, nc = (L - wl.kernel_size + 1.0) * 0.5, wl.n_chan
        scale = wl.freqs_hz / SPEED_OF_LIGHT
        centre = lambda lo, hi: np.floor((lo + hi) * 0.5 + 0.5)

        def box(b, t, c0, n):          # extremes over a group's channels lie at its ends
            x = wl.uvw_m[b, t]
            lo, hi = scale[c0], scale[c0 + n - 1]
            out = []
            for a, f in ((0, lambda v: v * S + 0.5 * N), (1, lambda v: v * S + 0.5 * N), (2, lambda v: v)):
                e, g = f(x[..., a] * lo), f(x[..., a] * hi)
                out.append((np.minimum(e, g), np.maximum(e, g)))
            return out

        def by_size(bx):
            ok = np.ones(bx[0][0].shape, dtype=bool)
            for lo, hi in bx[:2]:
                c = centre(lo, hi)
                ok &= (c - lo <= smax) & (hi - c <= smax)
            return ok & (bx[2][1] - bx[2][0] <= wl.w_step) if wl.w_step > 0 else ok

        def fits(bx):
            ok = by_size(bx)
            for lo, hi in bx[:2]:
                c = centre(lo, hi)
                ok &= (c - L / 2 >= 0) & (c + L / 2 <= N)
            return ok

        units = []                     # (baselines, slot, c0, n) with a common channel grouping
        for a in range(wl.n_slots):
            t = np.arange(wl.aterm_offsets[a], wl.aterm_offsets[a + 1])
            left = np.arange(wl.n_bl)
            for G in range(1, nc + 1):
                n = [nc // G + (g < nc % G) for g in range(G)]
                c0 = np.concatenate([[0], np.cumsum(n)[:-1]])
                ok = np.ones(left.size, dtype=bool)
                if G < nc:
                    for g in range(G):
                        ok &= by_size(box(left[:, None], t[None, :], c0[g], n[g])).all(axis=1)
                for g in range(G):
                    units.append((left[ok], a, c0[g], n[g]))
                left = left[~ok]
                if not left.size:
                    break
        b = np.concatenate([u[0] for u in units])
        a, c0, n = (np.concatenate([np.full(u[0].size, u[i]) for u in units]) for i in (1, 2, 3))
        ts, te = wl.aterm_offsets[a].astype(int), wl.aterm_offsets[a + 1].astype(int)
        got, opened = [], np.zeros(b.size, dtype=bool)
        t0 = np.zeros(b.size, dtype=int)
        cur = [(np.zeros(b.size), np.zeros(b.size)) for _ in range(3)]

        def close(at, end):
            i = np.nonzero(at)[0]
            cu, cv = (centre(cur[k][0][i], cur[k][1][i]) for k in (0, 1))
            k = np.floor((cur[2][0][i] + cur[2][1][i]) * 0.5 / wl.w_step + 0.5) if wl.w_step > 0 else np.zeros(i.size)
            got.append(np.stack([b[i], a[i], t0[i], end[i] - t0[i], c0[i], n[i], cu - L // 2, cv - L // 2, k]))

        for step in range(int((te - ts).max())):
            t = ts + step
            live = t < te
            bx = box(b, np.minimum(t, wl.n_t - 1), c0, n)
            both = [(np.minimum(p[0], q[0]), np.maximum(p[1], q[1])) for p, q in zip(cur, bx)]
            grow = live & opened & (t - t0 < wl.max_timesteps) & fits(both)
            end = opened & ~grow & live
            close(end, t)
            start = live & ~grow & fits(bx)
            for k in range(3):
                for h in (0, 1):
                    np.copyto(cur[k][h], both[k][h], where=grow)
                    np.copyto(cur[k][h], bx[k][h], where=start)
            t0[start] = t[start]
            opened = np.where(live, grow | start, opened)
            close(opened & (t == te - 1), t + 1)
            opened &= t != te - 1
        got = np.concatenate(got, axis=1)
        k_min = got[8].min()
        self.n_w = int(got[8].max() - k_min) + 1
        self.w0 = torch.from_numpy(got[8] * wl.w_step).cuda()
        self.w0_layers = [(k_min + j) * wl.w_step for j in range(self.n_w)]
        f = torch.from_numpy(got.astype(np.int64)).cuda()
        self.b, self.a, self.t0, self.nt, self.c0, self.nc, self.q0, self.r0 = f[:8]
        self.layer = f[8] - int(k_min)
        self.kp = self.nt * self.nc


class _Exact:
    """Direct sums of one observation in FP64."""

    def __init__(self, wl, d):
        self.wl, self.d = wl, d
        self.sub = _Subgrids(wl)
        L, S = wl.subgrid_size, wl.image_size
        self.L, self.N = L, wl.grid_size
        x = torch.arange(L, device="cuda", dtype=torch.float64) - L / 2
        self.l = (x * S / L)[None, :].expand(L, L).reshape(-1)
        self.m = (x * S / L)[:, None].expand(L, L).reshape(-1)
        self.n1 = torch.sqrt(1.0 - self.l ** 2 - self.m ** 2) - 1.0
        self.uvw = torch.from_numpy(wl.uvw_m).cuda().reshape(-1, 3)
        self.fc = torch.from_numpy(wl.freqs_hz / SPEED_OF_LIGHT).cuda()
        self.st = torch.from_numpy(wl.baselines.astype(np.int64)).cuda()
        self.taper = d["taper"].double().reshape(1, -1, 1, 1)
        self.use = torch.ones(wl.n_vis, dtype=torch.bool, device="cuda")
        if d["flags"] is not None:
            self.use = d["flags"].reshape(-1) == 0

    def chunks(self):
        """Indices of subgrids of similar size, a bounded number of phasors at a time."""
        order = torch.argsort(self.sub.kp)
        kp = self.sub.kp[order].cpu().numpy()
        i = 0
        while i < kp.size:
            j = i + 1
            while j < kp.size and (j + 1 - i) * int(kp[j]) * self.L ** 2 <= 1 << 26 and kp[j] <= 1.25 * kp[i] + 16:
                j += 1
            yield order[i:j]
            i = j

    def members(self, s):
        """Visibility index [s][K] (flat), validity [s][K] and phase [s][K][pixel] of subgrids s."""
        g, wl = self.sub, self.wl
        k = torch.arange(int(g.kp[s].max()), device="cuda")[None, :]
        ok = k < g.kp[s, None]
        t = g.t0[s, None] + torch.where(ok, k // g.nc[s, None], 0)
        c = g.c0[s, None] + torch.where(ok, k % g.nc[s, None], 0)
        bt = g.b[s, None] * wl.n_t + t
        x = self.uvw[bt] * self.fc[c][..., None]
        centre = torch.stack([(g.q0[s] + self.L // 2 - self.N / 2) / wl.image_size,
                              (g.r0[s] + self.L // 2 - self.N / 2) / wl.image_size, g.w0[s]], dim=-1)
        x = x - centre[:, None, :]
        turns = x @ torch.stack([self.l, self.m, self.n1])
        ph = 2.0 * math.pi * (turns - torch.round(turns))
        vi = bt * wl.n_chan + c
        return vi, ok & self.use[vi], torch.complex(torch.cos(ph), torch.sin(ph))

    def jones(self, s):
        """A_p, A_q of subgrids s as [s][pixel][2][2] (identity without A-terms)."""
        A = self.d["aterms"]
        if A is None:
            one = torch.eye(2, dtype=torch.complex128, device="cuda").expand(s.numel(), self.L ** 2, 2, 2)
            return one, one
        pq = self.st[self.sub.b[s]]
        return tuple(A[self.sub.a[s], pq[:, i]].to(torch.complex128).reshape(s.numel(), -1, 2, 2) for i in (0, 1))

    def pixels(self, s):
        """Flat grid index [s][L][L] of the subgrids' pixels."""
        i = torch.arange(self.L, device="cuda")
        row = self.sub.layer[s, None] * self.N + self.sub.r0[s, None] + i[None, :]
        return row[:, :, None] * self.N + (self.sub.q0[s, None] + i[None, :])[:, None, :]

    def images(self, s, vis):
        """Direct sums [s][pixel][2][2] of visibilities vis [n_vis][4] over subgrids s."""
        vi, ok, ph = self.members(s)
        v = torch.where(ok[..., None], vis[vi].to(torch.complex128), 0.0)
        return (ph.transpose(1, 2) @ v).reshape(s.numel(), -1, 2, 2)

    def grid(self, vis):
        out = torch.zeros((self.sub.n_w * self.N ** 2, 4), dtype=torch.complex128, device="cuda")
        for s in self.chunks():
            Ap, Aq = self.jones(s)
            I = self.taper * (Ap.mH @ self.images(s, vis) @ Aq)
            I = I.reshape(-1, self.L, self.L, 4)
            V = torch.fft.fftshift(torch.fft.fft2(torch.fft.ifftshift(I, dim=(1, 2)), dim=(1, 2)), dim=(1, 2)) / self.L ** 2
            torch.view_as_real(out).index_add_(0, self.pixels(s).reshape(-1), torch.view_as_real(V.reshape(-1, 4)))
        return out.reshape(self.sub.n_w, self.N, self.N, 4)

    def model_images(self, s, grid):
        """Transformed subgrids [s][pixel][2][2] of a model grid, before taper and A-terms."""
        V = grid.reshape(-1, 4)[self.pixels(s)].to(torch.complex128)
        I = torch.fft.fftshift(torch.fft.ifft2(torch.fft.ifftshift(V, dim=(1, 2)), dim=(1, 2)), dim=(1, 2))
        return I.reshape(s.numel(), -1, 2, 2)

    def degrid(self, grid):
        out = torch.zeros((self.wl.n_vis, 4), dtype=torch.complex128, device="cuda")
        for s in self.chunks():
            Ap, Aq = self.jones(s)
            P = (self.taper * (Ap @ self.model_images(s, grid) @ Aq.mH)).reshape(s.numel(), -1, 4)
            vi, ok, ph = self.members(s)
            out[vi[ok]] = (ph.conj() @ P)[ok]
        return out.reshape(self.wl.n_bl, self.wl.n_t, self.wl.n_chan, 4)

    def planned(self):
        on = torch.zeros(self.wl.n_vis, dtype=torch.bool, device="cuda")
        for s in self.chunks():
            vi, ok, _ = self.members(s)
            on[vi[ok]] = True
        return on.reshape(self.wl.n_bl, self.wl.n_t, self.wl.n_chan, 1)

    def gradient(self, grid, vis):
        r = torch.where(self.planned(), vis.to(torch.complex128) - self.degrid(grid), 0.0)
        A = self.d["aterms"]
        G = torch.zeros(A.shape, dtype=torch.complex128, device="cuda").reshape(-1, self.L ** 2 * 4)
        rows = lambda s, i: self.sub.a[s] * self.wl.n_stations + self.st[self.sub.b[s]][:, i]
        for s in self.chunks():
            Ap, Aq = self.jones(s)
            R = self.images(s, r.reshape(-1, 4))
            B = self.taper * self.model_images(s, grid)
            for i, X in ((0, -2.0 * (R @ Aq @ B.mH)), (1, -2.0 * (R.mH @ Ap @ B))):
                torch.view_as_real(G).index_add_(0, rows(s, i), torch.view_as_real(X.reshape(s.numel(), -1)))
        return r, G.reshape(A.shape), (r.abs() ** 2).sum().reshape(1)


def _exact_image(wl, layers, window, model, sky):
    N, L = wl.grid_size, wl.subgrid_size
    x = torch.arange(N, device="cuda", dtype=torch.float64) - N / 2
    lm = x * wl.image_size / N
    n1 = torch.sqrt(1.0 - lm[None, :] ** 2 - lm[:, None] ** 2) - 1.0
    shift = x[:, None] / N - ((torch.arange(L, device="cuda", dtype=torch.float64) - L / 2) / L)[None, :]
    mm = torch.arange(-(L // 2), L // 2, device="cuda", dtype=torch.float64)
    ph = 2.0 * math.pi * mm * shift[..., None]
    cbar = torch.complex(torch.cos(ph), torch.sin(ph)).sum(-1) @ torch.from_numpy(window).cuda().to(torch.complex128) / L
    cc = (cbar[:, None] * cbar[None, :])[..., None]
    turn = lambda w0: torch.polar(torch.ones_like(n1), 2.0 * math.pi * w0 * n1)[..., None]
    f = lambda fn, v: torch.fft.fftshift(fn(torch.fft.ifftshift(v, dim=(0, 1)), dim=(0, 1)), dim=(0, 1))
    image = sum(f(torch.fft.ifft2, g.to(torch.complex128)) * N * N * turn(w0) for g, w0 in zip(model, layers)) / cc
    src = sky.to(torch.complex128) / cc.conj()
    grid = torch.stack([f(torch.fft.fft2, src * turn(-w0)) for w0 in layers])
    return {"image": image, "grid": grid}


def exact(case, seed):
    kind = case["kind"]
    wls = _workloads(case, seed)
    if kind != "image" and sum(wl.n_vis * wl.subgrid_size ** 2 for wl in wls) > 2.5e10:
        return None                   # the FP64 sums would take too long
    got = []
    for k, wl in enumerate(wls):
        sub = _Subgrids(wl)
        d = _inputs(case, wl, seed, k, sub.n_w)
        if kind == "image":
            return _exact_image(wl, sub.w0_layers, syn.pswf_1d(wl.subgrid_size, BETA), d["model"],
                                _sky_image(wl.grid_size, _generator(seed, 99)))
        e = _Exact(wl, d)
        if kind == "grid":
            return e.grid(d["vis"].reshape(-1, 4))
        if kind == "degrid":
            return e.degrid(d["model"])
        if kind == "cycle":
            r = d["vis"].to(torch.complex128) - e.degrid(d["model"])
            return {"residual": r, "grid": e.grid(r.reshape(-1, 4))}
        if kind == "gradient":
            r, G, cost = e.gradient(d["model"], d["vis"])
            return {"residual": r, "gradient": G, "cost": cost}
        got.append((e.grid(d["vis"].reshape(-1, 4)), e.degrid(d["model"])))
    return {"grid": [g for g, _ in got], "vis": [v for _, v in got]}
