"""Performance cases of the image-domain gridder: what a program that images
with this package has it do, each case one pass through the public entry
points (`idg.Plan` and `idg.grid_many` / `idg.degrid_many`).

A case is a dict of plain values; `prepare` makes a program's inputs and plan
from it and a seed, `run` is one pass, `work` what the pass cannot do without
and `exact` the same outputs in 64 bits.  The arrays and geometries are those
of the package's workloads: the compact 32-station array (32 x 32 subgrids),
the MWA-like disk of up to 128 stations (96 x 96), and the log-normal array
with uneven subgrid occupancy (64 x 64).
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2502_17789_gb300 import idg, synth

C = 299792458.0

# array geometry: grid cells per side, kernel padding, field of view, seconds per timestep
GEOMETRY = {
    "compact": dict(grid=512, padding=12, fov=0.35, dt=8.0),
    "disk": dict(grid=4096, padding=18, fov=0.5, dt=2.0),
    "uneven": dict(grid=4096, padding=18, fov=0.5, dt=0.5),
}


def _case(name, work, array, stations, steps, channels, subgrid, interval, aterms="beam", grid=None,
          spacing="uniform", heights=0.0, stokes_i=False, w_layers=False, normalize=False, graph=False, requests=1):
    return dict(name=name, work=work, array=array, stations=stations, steps=steps, channels=channels,
                subgrid=subgrid, interval=interval, aterms=aterms, grid=grid or GEOMETRY[array]["grid"],
                spacing=spacing, heights=heights, stokes_i=stokes_i, w_layers=w_layers, normalize=normalize,
                graph=graph, requests=requests)


def listed():
    return [
        # the smallest call: one short snapshot of the compact array predicted and gridded by replaying
        # captured graphs, as a real-time loop does it
        _case("small_cycle", "cycle", "compact", 32, 16, 8, 32, 16, graph=True),
        # the package's main workload (the MWA-like observation its benchmark runs), one direction each
        _case("mwa_grid", "grid", "disk", 128, 56, 24, 96, 4),
        _case("mwa_degrid", "degrid", "disk", 128, 56, 24, 96, 4),
        # a snapshot with polarisation leakage in every Jones matrix (calibrated full-Jones A-terms)
        _case("snapshot_jones_grid", "grid", "disk", 64, 8, 24, 96, 4, aterms="jones", grid=2048),
        _case("snapshot_jones_degrid", "degrid", "disk", 64, 8, 24, 96, 4, aterms="jones", grid=2048),
        # a core-heavy array at high time resolution: subgrids from a few hundred to thousands of
        # visibilities, 64 x 64 subgrids
        _case("uneven_grid", "grid", "uneven", 64, 96, 30, 64, 8),
        _case("uneven_degrid", "degrid", "uneven", 64, 96, 30, 64, 8),
        # odd sizes throughout: flagged (irregularly spaced) channels, the largest subgrid; one major-cycle
        # step (predict from the model grid, grid the residual)
        _case("ragged_cycle_l128", "cycle", "disk", 37, 29, 13, 128, 5, aterms="jones", grid=2048,
              spacing="irregular"),
        # Stokes-I imaging of an unpolarised sky: a major-cycle step on one plane
        _case("stokes_i_cycle", "cycle", "disk", 80, 14, 16, 96, 4, grid=2048, stokes_i=True),
        # hilly site: station heights spread |w| over several w layers, prediction from an image and the
        # gridding of the residual
        _case("w_layers_predict", "predict", "disk", 60, 17, 24, 96, 4, grid=2048, heights=50.0, w_layers=True),
        # gridding with the A-term power normalisation
        _case("normalized_grid", "grid", "disk", 48, 28, 24, 96, 4, aterms="jones", grid=2048, normalize=True),
        # serving: several small snapshot requests gridded and degridded through the shared work queue
        _case("serving_many", "many", "compact", 40, 12, 16, 32, 4, requests=6),
    ]


def draw(rng):
    """One more case: a listed kind at sizes spread over the ranges it stands for."""

    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    c = dict(rng.choice(listed()))
    del c["name"]
    if c["array"] == "compact":
        c["stations"], c["steps"], c["channels"] = log_int(8, 64), log_int(1, 48), log_int(1, 32)
        c["requests"] = rng.randint(2, 8) if c["work"] == "many" else 1
    else:
        c["stations"], c["steps"], c["channels"] = log_int(8, 120), log_int(1, 56), log_int(1, 48)
        if c["array"] == "uneven":
            c["steps"] = log_int(8, 160)
        c["subgrid"] = rng.choice([64, 96, 96, 128])
        c["aterms"] = rng.choice(["beam", "beam", "jones"])
        c["spacing"] = rng.choice(["uniform", "uniform", "uniform", "irregular"])
    c["interval"] = rng.choice([2, 3, 4, 5, 8, 16])
    # no drawn case costs more than the largest listed one (both directions count)
    while _vis_pixels(c) > 0.9e11:
        c["steps"] = max(1, c["steps"] // 2)
    return c


# ---------------------------------------------------------------- inputs


def _directions(case):
    return 1 if case["work"] in ("grid", "degrid") else 2


def _n_vis(case):
    s = case["stations"]
    return s * (s - 1) // 2 * case["steps"] * case["channels"]


def _vis_pixels(case):
    return float(_n_vis(case)) * case["subgrid"] ** 2 * _directions(case) * case["requests"]


def _flags(case):
    f = idg.IDG_STOKES_I if case["stokes_i"] else 0
    f |= idg.IDG_W_LAYERS if case["w_layers"] else 0
    return f | (idg.IDG_NORMALIZE_ATERM if case["normalize"] else 0)


def _observation(case, seed):
    rng = np.random.default_rng(seed)
    geo = GEOMETRY[case["array"]]
    n = case["stations"]
    if case["array"] == "compact":
        enu = synth.stations_uniform_disk(rng, n, 1000.0)
        freqs = 150e6 + 1e6 * np.arange(case["channels"])
    else:
        if case["array"] == "disk":
            enu = synth.stations_uniform_disk(rng, n, 3000.0)
        else:
            enu = synth.stations_lognormal(rng, n, 300.0, 1.0, 3000.0)
        freqs = np.linspace(140e6, 170e6, case["channels"])
    if case["spacing"] == "irregular":
        # every third of a finer set of channels is flagged away
        fine = np.linspace(freqs[0], freqs[0] + 30e6, 2 * case["channels"])
        freqs = fine[np.sort(rng.permutation(2 * case["channels"])[: case["channels"]])]
    if case["heights"]:
        enu[:, 2] = rng.normal(0.0, case["heights"], n)
    return synth.make_observation(enu, case["steps"], geo["dt"], freqs, case["interval"], case["grid"],
                                  case["subgrid"], geo["padding"], geo["fov"])


def _aterms(case, obs, seed):
    rng = np.random.default_rng(seed + 1)
    A = synth.aterms_beam_screen(obs, synth.beam_screen_model(rng, rms_rad=2.0))
    return synth.aterms_with_leakage(rng, A, 0.05) if case["aterms"] == "jones" else A


def _visibilities(obs, seed, device):
    """Sixteen point sources with a little polarisation, plus noise, complex64 [bl, t, ch, 4]."""
    g = torch.Generator(device=device)
    g.manual_seed(seed + 2)
    rng = np.random.default_rng(seed + 3)
    sky = synth.point_sources(rng, 16, obs.image_size / 3)
    uvw = torch.as_tensor(obs.uvw, device=device)
    fc = torch.as_tensor(obs.freqs / C, device=device)
    shape = (obs.n_baselines, obs.n_timesteps, obs.n_channels, 4)
    out = 0.5 * torch.randn(shape, dtype=torch.complex64, device=device, generator=g)
    for l, m, s in zip(sky.l, sky.m, sky.flux):
        d = uvw[..., 0] * l + uvw[..., 1] * m + uvw[..., 2] * (math.sqrt(1 - l * l - m * m) - 1)
        turns = d[..., None] * fc
        ph = (-2 * math.pi * (turns - turns.round())).float()
        e = torch.polar(torch.full_like(ph, float(s)), ph)
        for k, b in enumerate((1.0, 0.02, 0.02, 0.9)):
            out[..., k] += b * e
    return out


def _image_taper(n, padding):
    x = (2.0 * np.arange(n) - n) / n
    beta = 0.35 * math.pi * padding
    return np.i0(beta * np.sqrt(np.maximum(1.0 - x * x, 0.0))) / np.i0(beta)


def _model_image(case, seed, device, n_pol):
    """A clean model: 200 components in the central half of the padded field, complex128 [n_pol, N, N]."""
    N = case["grid"]
    rng = np.random.default_rng(seed + 4)
    img = torch.zeros((n_pol, N, N), dtype=torch.complex128, device=device)
    x = torch.as_tensor(rng.integers(N // 4, N - N // 4, 200), device=device)
    y = torch.as_tensor(rng.integers(N // 4, N - N // 4, 200), device=device)
    flux = torch.as_tensor(np.exp(rng.standard_normal(200)), device=device)
    for k, b in enumerate((1.0, 0.03 + 0.01j, 0.03 - 0.01j, 0.9)[:n_pol]):
        img[k].index_put_((y, x), b * flux.to(torch.complex128), accumulate=True)
    return img


def _signs(n, device):
    s = 1.0 - 2.0 * (torch.arange(n, device=device) % 2)
    return torch.outer(s, s).to(torch.float64)


def _model_grid(case, image):
    """The model's uv plane as prediction makes it: taper correction, then the centred transform."""
    N, L = case["grid"], case["subgrid"]
    t = torch.as_tensor(1.0 / _image_taper(N, GEOMETRY[case["array"]]["padding"]), device=image.device)
    s = _signs(N, image.device)
    return torch.fft.fft2(image * (torch.outer(t, t) * s / (L * L))) * s


def _inputs(case, seed, device):
    """Per request: observation, A-terms, visibilities, model image, model grid (those the case's work uses)."""
    out = []
    for r in range(case["requests"]):
        sd = 1000 * seed + 17 * r
        obs = _observation(case, sd)
        A = _aterms(case, obs, sd)
        vis = image = model = None
        if case["work"] != "degrid":
            vis = _visibilities(obs, sd, device)
        if case["work"] != "grid":
            image = _model_image(case, sd, device, 1 if case["stokes_i"] else 4)
            if case["work"] != "predict":
                model = _model_grid(case, image)
        out.append(dict(obs=obs, A=torch.as_tensor(A, device=device), vis=vis, image=image, model=model))
    return out


# ---------------------------------------------------------------- passes


class _State:
    pass


def prepare(case, seed):
    device = torch.device("cuda")
    s = _State()
    s.case = case
    s.inputs = _inputs(case, seed, device)
    s.side = torch.cuda.Stream() if case["graph"] else None
    stream = s.side.cuda_stream if case["graph"] else None
    s.plans, s.grids, s.kept, s.out, s.work = [], [], [], [], []
    for x in s.inputs:
        obs = x["obs"]
        p = idg.Plan(obs, flags=_flags(case), stream=stream)
        s.plans.append(p)
        shape = (obs.n_baselines, obs.n_timesteps, obs.n_channels, 4)
        if case["work"] != "degrid":
            s.grids.append(torch.zeros(p.grid_shape(), dtype=torch.complex128, device=device))
            s.kept.append(torch.zeros(p.grid_shape(), dtype=torch.complex64, device=device))
        if case["work"] != "grid":
            s.out.append(torch.zeros(shape, dtype=torch.complex64, device=device))
        if case["work"] in ("cycle", "predict"):
            s.residual = torch.zeros(shape, dtype=torch.complex64, device=device)
        if case["work"] == "predict":
            s.work.append(torch.zeros(p.grid_shape(), dtype=torch.complex128, device=device))
    torch.cuda.synchronize()
    return s


def run(s):
    """One pass.  The double-precision grid is the sum's accumulator; the program keeps (stores, hands on) the
    gridded planes in single precision, the accuracy of the gridder's sums."""
    case, kind = s.case, s.case["work"]
    x, plan = s.inputs[0], s.plans[0]
    if kind == "many":
        vis, A, model = ([i[k] for i in s.inputs] for k in ("vis", "A", "model"))
        idg.degrid_many(s.plans, model, A, s.out)
        for g in s.grids:
            g.zero_()
        idg.grid_many(s.plans, vis, A, s.grids)
        for g, k in zip(s.grids, s.kept):
            k.copy_(g)
        return {"vis": s.out, "grid": s.kept}
    if s.side is not None:
        cur = torch.cuda.current_stream()
        s.side.wait_stream(cur)
        with torch.cuda.stream(s.side):
            plan.degrid_graph(x["model"], x["A"], s.out[0])
            torch.sub(x["vis"], s.out[0], out=s.residual)
            s.grids[0].zero_()
            plan.grid_graph(s.residual, x["A"], s.grids[0])
            s.kept[0].copy_(s.grids[0])
        cur.wait_stream(s.side)
        return {"vis": s.out[0], "grid": s.kept[0]}
    plan.set_stream(torch.cuda.current_stream().cuda_stream)
    if kind == "degrid":
        return {"vis": plan.degrid(x["model"], x["A"], s.out[0])}
    vis = x["vis"]
    if kind != "grid":
        if kind == "predict":
            plan.predict(x["image"], x["A"], s.work[0], s.out[0])
        else:
            plan.degrid(x["model"], x["A"], s.out[0])
        vis = torch.sub(vis, s.out[0], out=s.residual)
    s.grids[0].zero_()
    plan.grid(vis, x["A"], s.grids[0])
    s.kept[0].copy_(s.grids[0])
    return {"grid": s.kept[0]} if kind == "grid" else {"vis": s.out[0], "grid": s.kept[0]}


def work(case):
    """Bytes: visibilities, uvw and A-terms once and the grid once (and its single-precision copy), per direction.  Flops: the
    method's direct sum, 34 per visibility and subgrid pixel (4 complex multiply-adds, one phase)."""
    n = case["stations"]
    n_int = -(-case["steps"] // case["interval"])
    n_pol = 1 if case["stokes_i"] else 4
    per = (_n_vis(case) * 32 + n * (n - 1) // 2 * case["steps"] * 24 + n_int * n * 81 * 32
           + case["grid"] ** 2 * n_pol * (16 if case["work"] == "degrid" else 24))
    return {"bytes": float(per * _directions(case) * case["requests"]), "flops": 34.0 * _vis_pixels(case)}


# ---------------------------------------------------------------- the same outputs in 64 bits


def _partition(case, obs):
    """The partition of Section 3.1 (with w layers of Section 2.4): rows (b, t0, t1, c0, c1, x0, y0, k, mirrored)
    and the layer width (0 without layers)."""
    N, L, P, fov = obs.grid_size, obs.subgrid_size, obs.kernel_padding, obs.image_size
    S = L - P - 4
    Sc = max(0, S - max(2, S // 4))
    r2 = 0.5 * fov * fov
    w_step = 2.0 * ((0.5 * P - 1.0) / (math.sqrt(r2) / math.sqrt(1.0 - r2) * fov)) if case["w_layers"] else 0.0
    rows = []
    for b in range(obs.n_baselines):
        r = obs.uvw[b]
        sgn = np.where((r[:, 2] < 0.0) & (w_step > 0.0), -1.0, 1.0)[:, None]
        x = (sgn * r[:, :1] * obs.freqs) / C * fov + N / 2
        y = (sgn * r[:, 1:2] * obs.freqs) / C * fov + N / 2
        if w_step > 0.0:
            w = (sgn * r[:, 2:] * obs.freqs) / C
            key = 2 * np.floor(w / w_step).astype(np.int64) + (sgn < 0)
        else:
            key = np.zeros(x.shape, np.int64)
        todo, runs = [(0, 0, obs.n_channels)], []
        while todo:
            ts, c_lo, c_hi = todo.pop()
            lo = c_lo
            while lo < c_hi:
                xs, ys, ks = x[ts, lo:c_hi], y[ts, lo:c_hi], key[ts, lo:c_hi]
                bad = (np.abs(xs - xs[0]) > Sc) | (np.abs(ys - ys[0]) > Sc) | (ks != ks[0])
                hi = lo + (int(bad.argmax()) if bad.any() else c_hi - lo)
                cols = [lo, hi - 1]

                def spread(v):
                    top = np.maximum(v[ts:, cols].max(1), v[ts, cols].max())
                    return top - np.minimum(v[ts:, cols].min(1), v[ts, cols].min())

                bad = (spread(x) > S) | (spread(y) > S) | (key[ts:, cols] != ks[0]).any(1)
                bad[0] = False
                te = ts + (int(bad.argmax()) if bad.any() else obs.n_timesteps - ts)
                while te > ts + 1:
                    bx, by = x[ts:te, lo:hi], y[ts:te, lo:hi]
                    if bx.max() - bx.min() <= S and by.max() - by.min() <= S and (key[ts:te, lo:hi] == ks[0]).all():
                        break
                    te -= 1
                bx, by = x[ts:te, lo:hi], y[ts:te, lo:hi]
                x0 = math.floor((bx.min() + bx.max()) / 2.0) - L // 2
                y0 = math.floor((by.min() + by.max()) / 2.0) - L // 2
                runs.append((b, ts, te, lo, hi, x0, y0, int(ks[0]) >> 1, int(ks[0]) & 1))
                if te < obs.n_timesteps:
                    todo.append((te, lo, hi))
                lo = hi
        rows += sorted(runs, key=lambda q: (q[1], q[3]))
    return rows, w_step


class _Exact:
    """Gridding and degridding of one request by the method's sums in complex128."""

    def __init__(self, case, x):
        self.case, self.obs = case, x["obs"]
        obs, dev = self.obs, x["A"].device
        L, fov, nodes = obs.subgrid_size, obs.image_size, obs.aterm_nodes
        self.rows, self.w_step = _partition(case, obs)
        ks = [r[7] for r in self.rows] or [0]
        self.k_min, self.n_layers = min(ks), max(ks) - min(ks) + 1
        self.n_pol = 1 if case["stokes_i"] else 4
        f64 = dict(dtype=torch.float64, device=dev)
        self.dev = dev
        self.l = torch.as_tensor((np.arange(L) - L // 2) * fov / L, **f64)
        self.n1 = (torch.sqrt(1 - self.l[None, :] ** 2 - self.l[:, None] ** 2) - 1).reshape(-1)  # [j, i]
        t = (2.0 * np.arange(L) - L) / L
        beta = 0.35 * math.pi * obs.kernel_padding
        t = torch.as_tensor(np.i0(beta * np.sqrt(1 - t * t)) / np.i0(beta), **f64)
        self.taper = torch.outer(t, t).reshape(-1, 1)
        self.signs = _signs(L, dev)
        # bilinear interpolation from the nodes to the pixels, along one axis
        B = np.zeros((L, nodes))
        for i in range(L):
            q = (nodes - 1) * i / L
            a = min(int(q), nodes - 2)
            B[i, a], B[i, a + 1] = 1.0 - (q - a), q - a
        B = torch.as_tensor(B, **f64).to(torch.complex128)
        A = x["A"].to(torch.complex128)
        self.jones = functools.lru_cache(maxsize=None)(
            lambda a, s: torch.einsum("jy,ix,yxe->jie", B, B, A[a, s]).reshape(-1, 2, 2))
        self.uvw = torch.as_tensor(obs.uvw, **f64)
        self.fc = torch.as_tensor(obs.freqs / C, **f64)
        off = obs.aterm_offsets
        self.intervals = [(a, int(off[a]), int(off[a + 1])) for a in range(len(off) - 1)]

    def subgrids(self):
        """Per subgrid: its row, stations, phasors e^{2 pi i phi} [k, pixels], segments (interval, k0, k1)."""
        obs, L = self.obs, self.obs.subgrid_size
        for r in self.rows:
            b, t0, t1, c0, c1, x0, y0, k, mirror = r
            p, q = (int(v) for v in obs.baselines[b][:: -1 if mirror else 1])
            uvw = (-1.0 if mirror else 1.0) * self.uvw[b, t0:t1, None, :] * self.fc[c0:c1, None]
            u, v, w = uvw.reshape(-1, 3).unbind(1)
            u = u - (x0 + L // 2 - obs.grid_size // 2) / obs.image_size
            v = v - (y0 + L // 2 - obs.grid_size // 2) / obs.image_size
            w = w - (k + 0.5) * self.w_step if self.w_step else w
            ph = (v[:, None, None] * self.l[:, None] + u[:, None, None] * self.l[None, :]).flatten(1)
            ph = (ph + w[:, None] * self.n1) * (2 * math.pi)
            nc = c1 - c0
            seg = [(a, (max(lo, t0) - t0) * nc, (min(hi, t1) - t0) * nc) for a, lo, hi in self.intervals
                   if max(lo, t0) < min(hi, t1)]
            yield r, p, q, torch.polar(torch.ones_like(ph), ph), seg

    def grid(self, vis):
        obs, L, N = self.obs, self.obs.subgrid_size, self.obs.grid_size
        G = torch.zeros((self.n_layers, self.n_pol, N, N), dtype=torch.complex128, device=self.dev)
        for (b, t0, t1, c0, c1, x0, y0, k, mirror), p, q, e, seg in self.subgrids():
            V = vis[b, t0:t1, c0:c1].reshape(-1, 2, 2).to(torch.complex128)
            V = (V.mH if mirror else V).reshape(-1, 4)
            X = 0.0
            for a, k0, k1 in seg:
                Ap, Aq = self.jones(a, p), self.jones(a, q)
                part = Ap.mH @ (e[k0:k1].T @ V[k0:k1]).reshape(-1, 2, 2) @ Aq
                if self.case["normalize"]:
                    f = torch.linalg.matrix_norm(Ap.mH @ Aq)[:, None, None]
                    part = torch.where(f > 0, part / f, torch.zeros_like(part))
                X = X + part
            X = (X.reshape(-1, 4) * self.taper).T.reshape(4, L, L)
            if self.n_pol == 1:
                X = 0.5 * (X[:1] + X[3:])
            X = torch.fft.fft2(X * self.signs) * self.signs
            G[k - self.k_min, :, y0:y0 + L, x0:x0 + L] += X
        return G if self.case["w_layers"] else G[0]

    def degrid(self, G):
        L = self.obs.subgrid_size
        obs = self.obs
        out = torch.zeros((obs.n_baselines, obs.n_timesteps, obs.n_channels, 4), dtype=torch.complex128,
                          device=self.dev)
        G = G if self.case["w_layers"] else G[None]
        for (b, t0, t1, c0, c1, x0, y0, k, mirror), p, q, e, seg in self.subgrids():
            Y = torch.fft.ifft2(G[k - self.k_min, :, y0:y0 + L, x0:x0 + L] * self.signs) * self.signs * (L * L)
            Y = Y.reshape(self.n_pol, -1).T * self.taper
            if self.n_pol == 1:
                Y = Y * torch.tensor([1.0, 0.0, 0.0, 1.0], dtype=torch.complex128, device=self.dev)
            V = torch.empty((e.shape[0], 4), dtype=torch.complex128, device=self.dev)
            for a, k0, k1 in seg:
                Z = self.jones(a, p) @ Y.reshape(-1, 2, 2) @ self.jones(a, q).mH
                V[k0:k1] = e[k0:k1].conj() @ Z.reshape(-1, 4)
            V = V.reshape(-1, 2, 2)
            out[b, t0:t1, c0:c1] = (V.mH if mirror else V).reshape(t1 - t0, c1 - c0, 4)
        return out

    def predict(self, image):
        """Eq. 12: the image shifted to each layer's w0, taper-corrected and transformed, then degridded."""
        if not self.case["w_layers"]:
            return self.degrid(_model_grid(self.case, image))
        N, fov = self.obs.grid_size, self.obs.image_size
        l = torch.as_tensor((np.arange(N) - N // 2) * fov / N, device=self.dev)
        n1 = torch.sqrt(1 - l[None, :] ** 2 - l[:, None] ** 2) - 1
        layers = []
        for k in range(self.k_min, self.k_min + self.n_layers):
            turns = (k + 0.5) * self.w_step * n1
            ph = -2 * math.pi * (turns - turns.round())
            layers.append(_model_grid(self.case, image * torch.polar(torch.ones_like(ph), ph)))
        return self.degrid(torch.stack(layers))


def exact(case, seed):
    if _vis_pixels(case) > 4e10:
        return None  # minutes in 64 bits
    device = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    outs = []
    for x in _inputs(case, seed, device):
        ref, o = _Exact(case, x), {}
        if case["work"] == "predict":
            o["vis"] = ref.predict(x["image"])
        elif case["work"] != "grid":
            o["vis"] = ref.degrid(x["model"])
        if case["work"] in ("cycle", "predict"):
            o["grid"] = ref.grid(x["vis"] - o["vis"])
        elif case["work"] != "degrid":
            o["grid"] = ref.grid(x["vis"])
        outs.append(o)
    if case["work"] == "many":
        return {k: [o[k] for o in outs] for k in ("vis", "grid")}
    return outs[0]
