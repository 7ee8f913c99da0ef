"""The work a user of this library has it do, as cases that can be timed and compared.

Every case goes through the public entry points (scene.Scene, scene.Batch, scene.FluoroRender) the way
a program calls them: the scene handle is made once, a pass renders and reads what it needs. Inputs
are synthetic and made from a seed: random dye blobs and spheres, the sizes of this repository's
benchmark, tests and generators. Path counts, grid edges and films run from a first look (10^4 paths,
where launches and the longest path count) to the full light sheet (6.7 * 10^7 paths).
"""
import math

import numpy as np
import torch

from paper_1706_03024_gb300 import scene as fs

LAMBDA0, DLAMBDA, N_BINS = 380.0, 5.0, 81

# Units of work per path, from the counters of the listed cases: (tracking steps, real events, sensor
# connections, ratio-tracking steps). An event of the batch or the camera walk has no film vertex.
UNITS = {
    "cube": (23.8, 22.9, 22.9, 0.0),
    "cornell": (38.8, 13.9, 14.9, 39.0),
    "frames": (39.6, 13.9, 14.9, 39.7),
    "vial": (30.1, 17.2, 16.7, 19.9),
    "sheet": (64.9, 62.1, 62.1, 68.2),
    "batch": (34.1, 20.0, 0.0, 0.0),
    "adjoint": (45.0, 20.0, 20.0, 40.0),
    "camera": (6.0, 2.7, 1.1, 15.9),
}


def listed():
    return [
        # a first look at a homogeneous solution: the smallest call, latency and launches
        {"name": "cube_first_look", "kind": "cube", "n_paths": 10_000, "film": 64},
        # its spectra in earnest: closed-form transmittance, a beam down the film's axis
        {"name": "cube_spectra", "kind": "cube", "n_paths": 20_000_000, "film": 64},
        # a preview of the Cornell box of dye spheres while a scene is being set up; ragged sizes
        {"name": "cornell_preview", "kind": "cornell", "width": 97, "height": 71, "spp": 4, "grid": 45,
         "form": "wavefront_warp", "cell": 1, "hero": 0},
        # the benchmark image: 512 x 512 x 81 film, 16 paths per pixel, 128^3 x 4 grids
        {"name": "cornell_render", "kind": "cornell", "width": 512, "height": 512, "spp": 16, "grid": 128,
         "form": "wavefront_warp", "cell": 1, "hero": 0},
        # the same scene with four wavelengths per path
        {"name": "cornell_hero", "kind": "cornell", "width": 512, "height": 512, "spp": 8, "grid": 128,
         "form": "wavefront_warp", "cell": 1, "hero": 4},
        # render() with its default options, at the size the tests use
        {"name": "cornell_defaults", "kind": "cornell", "width": 100, "height": 100, "spp": 10, "grid": 48,
         "form": "plain", "cell": 0, "hero": 0},
        # a dye vial in a refracting cuvette, seen from the front
        {"name": "vial", "kind": "vial", "film": 96, "spp": 32, "grid": 50, "conc": 1.0},
        # the light sheet at full size: the largest call, grids beyond the L2
        {"name": "light_sheet", "kind": "sheet", "film": 1024, "spp": 64, "grid": 256},
        # hundreds of uneven media in one launch (face spectra for a data set)
        {"name": "media_batch", "kind": "batch", "media": 256, "max_edge": 128, "scale": 1.0},
        # one step of a fit of concentrations to an image: forward and backward
        {"name": "fit_step", "kind": "adjoint", "grid": 64, "film": 256, "spp": 32},
        # the camera-side estimator of the single-inelastic model
        {"name": "camera_view", "kind": "camera", "grid": 64, "film": 256, "spp": 16},
        # a time series: every frame uploads new grids, renders briefly and reads its result
        {"name": "frames", "kind": "frames", "width": 256, "height": 256, "spp": 4, "grid": 96},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["cube", "cornell", "cornell", "hero", "defaults", "vial", "sheet", "batch", "adjoint",
                       "camera", "frames"])
    if kind == "cube":
        return {"kind": "cube", "n_paths": _log(rng, 2_000, 40_000_000), "film": _log(rng, 16, 256)}
    if kind in ("cornell", "hero", "defaults"):
        plain = kind == "defaults"
        w, h = _log(rng, 40, 300 if plain else 640), _log(rng, 40, 300 if plain else 640)
        return {"kind": "cornell", "width": w, "height": h, "spp": rng.randint(1, 8 if plain else 16),
                "grid": rng.randint(17, 128), "form": "plain" if plain else "wavefront_warp",
                "cell": 0 if plain else rng.choice([1, 1, 2, 4]), "hero": rng.randint(2, 4) if kind == "hero" else 0}
    if kind == "vial":
        return {"kind": "vial", "film": _log(rng, 24, 300), "spp": rng.randint(1, 48),
                "grid": rng.choice([0, rng.randint(16, 96)]), "conc": rng.choice([0.1, 1.0, 10.0])}
    if kind == "sheet":
        return {"kind": "sheet", "film": _log(rng, 64, 1000), "spp": rng.randint(2, 40), "grid": rng.randint(48, 256)}
    if kind == "batch":
        return {"kind": "batch", "media": _log(rng, 4, 200), "max_edge": rng.randint(20, 128),
                "scale": math.exp(rng.uniform(math.log(0.05), 0.0))}
    if kind == "adjoint":
        return {"kind": "adjoint", "grid": rng.randint(16, 80), "film": _log(rng, 32, 300), "spp": rng.randint(2, 32)}
    if kind == "camera":
        return {"kind": "camera", "grid": rng.randint(16, 80), "film": _log(rng, 24, 400), "spp": rng.randint(1, 24)}
    return {"kind": "frames", "width": _log(rng, 48, 400), "height": _log(rng, 48, 400), "spp": rng.randint(1, 6),
            "grid": rng.randint(20, 128)}


# Scenes ----------------------------------------------------------------------------------------


def _bands(peaks, sigmas):
    lam = LAMBDA0 + DLAMBDA * np.arange(N_BINS)
    return np.stack([np.exp(-0.5 * ((lam - p) / s) ** 2) for p, s in zip(peaks, sigmas)]).astype(np.float32)


def _dyes(abs_peaks, abs_sigma, em_peaks, em_sigma, eps, qy):
    n = len(abs_peaks)
    return {"abs_shape": _bands(abs_peaks, np.broadcast_to(abs_sigma, n)),
            "emit_spec": _bands(em_peaks, np.broadcast_to(em_sigma, n)),
            "eps": np.asarray(eps, np.float32), "qy": np.asarray(qy, np.float32)}


def _medium(n_dyes, sigma_s, conc=0.0, walls=0, albedo=0.0, ior=1.0):
    return {"lo": (0.0, 0.0, 0.0), "hi": (1.0, 1.0, 1.0), "dims": None, "conc": None, "solvent": None,
            "conc_uniform": np.full(n_dyes, conc, np.float32), "sigma_s": float(sigma_s), "sigma_a0": 0.0,
            "wall_mask": walls, "wall_albedo": albedo, "ior": ior}


def _source(kind, origin, eu, ev, direction, lines):
    return {"kind": kind, "origin": origin, "eu": eu, "ev": ev, "dir": direction, "lines_nm": list(lines),
            "power": [1.0] * len(lines)}


def _sensor(kind, width, height, origin, u, v, view, fov=0.0):
    return {"kind": kind, "width": width, "height": height, "origin": origin, "U": u, "V": v, "view": view,
            "fov_y_deg": fov}


def _scene(dyes, medium, source, sensor, n_paths, seed):
    return {"spectrum": {"lambda0": LAMBDA0, "dlambda": DLAMBDA, "n_bins": N_BINS}, "dyes": dyes, "medium": medium,
            "sources": [source], "sensor": sensor,
            "params": {"n_paths": int(n_paths), "seed": int(seed) & 0x7FFFFFFF, "n_rr": 5, "max_events": 1_000_000,
                       "max_inelastic": -1, "analog": 0, "max_steps": 10_000_000}}


def _blobs(rng, n, count, smin, smax):
    """Sum of Gaussian blobs on an n^3 grid (widths in voxels), scaled to mean 1."""
    c, s, a = rng.uniform(0, n, (count, 3)), rng.uniform(smin, smax, count), rng.uniform(0.5, 1.5, count)
    x = np.arange(n) + 0.5
    g = np.exp(-0.5 * ((x[None, None] - c.T[:, :, None]) / s[None, :, None]) ** 2)
    g[np.abs(x[None, None] - c.T[:, :, None]) > 3.0 * s[None, :, None]] = 0.0
    gx, gy, gz = (torch.from_numpy(v.astype(np.float32)).cuda() for v in g)
    gz = gz * torch.from_numpy(a.astype(np.float32)).cuda()[:, None]
    f = ((gz[:, :, None] * gy[:, None, :]).reshape(count, n * n).t() @ gx).reshape(n, n, n)
    return f / f.double().mean().clamp_min(1e-3).float()


def _spheres(rng, n):
    """Four disjoint balls of radius 0.15 to 0.25, one dye each, with solvent inside them only."""
    balls = []
    while len(balls) < 4:
        balls = []
        for _ in range(2000):
            r = rng.uniform(0.15, 0.25)
            c = rng.uniform(r, 1.0 - r, 3)
            if all(np.linalg.norm(c - c2) >= r + r2 + 0.01 for c2, r2 in balls):
                balls.append((c, r))
            if len(balls) == 4:
                break
    x = (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) / n
    ins = torch.stack([((x - c[0]) ** 2)[None, None, :] + ((x - c[1]) ** 2)[None, :, None]
                       + ((x - c[2]) ** 2)[:, None, None] <= r * r for c, r in balls])
    return ins.float(), ins.any(0).to(torch.uint8)


def _cornell(case, seed):
    rng = np.random.default_rng(seed)
    em = [450.0, 520.0, 600.0, 680.0]
    ab = [p - 30.0 for p in em]
    conc, solvent = _spheres(rng, case["grid"])
    light = _source("lambertian", (0.35, 0.35, 1.0), (0.3, 0.0, 0.0), (0.0, 0.3, 0.0), (0.0, 0.0, -1.0), ab)
    cam = _sensor("pinhole", case["width"], case["height"], (0.5, -1.4, 0.5), (1.0, 0.0, 0.0), (0.0, 0.0, 1.0),
                  (0.0, 1.0, 0.0), 40.0)
    desc = _scene(_dyes(ab, 15.0, em, 20.0, [2.0] * 4, rng.uniform(0.3, 0.95, 4)),
                  _medium(4, 50.0, walls=0b111011, albedo=0.8), light, cam,
                  case["width"] * case["height"] * case["spp"], seed)
    return desc, {"conc": conc, "solvent": solvent}


def _batch_scenes(case, seed):
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(case["media"]):
        n, d = int(rng.integers(16, case["max_edge"] + 1)), int(rng.integers(1, 4))
        albedo, n_paths = float(rng.uniform(0.5, 0.999)), int(10 ** rng.uniform(4.0, 6.0) * case["scale"])
        ab = rng.uniform(420.0, 620.0) + np.concatenate([[0.0], rng.uniform(-25.0, 25.0, d - 1)])
        blobby = rng.random() < 0.5
        conc = (torch.stack([_blobs(rng, n, 8, n / 16, n / 6) for _ in range(d)]) if blobby
                else torch.ones(d, n, n, n)).cpu().numpy()
        dyes = _dyes(ab, rng.uniform(12.0, 25.0, d), ab + rng.uniform(20.0, 60.0, d), rng.uniform(15.0, 30.0, d),
                     np.ones(d), rng.uniform(0.3, 0.95, d))
        b = int(np.clip(math.ceil((ab[0] - LAMBDA0) / DLAMBDA - 0.5), 0, N_BINS - 1))
        dyes["eps"] = np.full(d, (1.0 - albedo) * 40.0 / dyes["abs_shape"][:, b].sum(), np.float32)
        med = _medium(d, albedo * 40.0)
        med["conc"] = conc
        out.append(_scene(dyes, med, _source("collimated", (0.5, 0.5, 0.0), (0.0,) * 3, (0.0,) * 3, (0.0, 0.0, 1.0),
                                             [float(ab[0])]),
                          _sensor("none", 0, 0, (0.0,) * 3, (0.0,) * 3, (0.0,) * 3, (0.0,) * 3), n_paths, seed))
    return out


def _beam(lines):
    return _source("collimated", (0.0, 0.0, 0.0), (1.0, 0.0, 0.0), (0.0, 1.0, 0.0), (0.0, 0.0, 1.0), lines)


def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.default_rng(seed)
    top = lambda n: _sensor("ortho", n, n, (0.0, 0.0, 1.0), (1.0, 0.0, 0.0), (0.0, 1.0, 0.0), (0.0, 0.0, 1.0))  # noqa: E731
    grids, st = None, {"case": case}
    if kind == "batch":
        scenes = _batch_scenes(case, seed)
        st["batch"] = fs.Batch(scenes, seed=int(seed) & 0x7FFFFFFF)
        st["paths"] = int(st["batch"].n_paths.sum())
        return st
    if kind == "cube":
        desc = _scene(_dyes([490.0], 15.0, [520.0], 20.0, [2.0], [0.9]), _medium(1, 20.0, conc=1.0),
                      _source("collimated", (0.5, 0.5, 1.0), (0.0,) * 3, (0.0,) * 3, (0.0, 0.0, -1.0), [490.0]),
                      top(case["film"]), case["n_paths"], seed)
    elif kind in ("cornell", "frames"):
        desc, grids = _cornell(case, seed)
    elif kind == "vial":
        med = _medium(1, 20.0, conc=case["conc"], ior=1.33)
        if case["grid"]:
            x = (torch.arange(case["grid"], device="cuda", dtype=torch.float64) + 0.5) / case["grid"] - 0.5
            ins = (x[None, None, :] ** 2 + x[None, :, None] ** 2 <= 0.35 ** 2).expand(case["grid"], -1, -1)
            grids = {"conc": (ins * case["conc"]).float()[None].contiguous(),
                     "solvent": ins.to(torch.uint8).contiguous()}
        y0 = float(rng.uniform(0.4, 0.5))
        desc = _scene(_dyes([495.0], 15.0, [520.0], 20.0, [1.5], [0.9]), med,
                      _source("collimated", (0.0, y0, 0.45), (0.0, 0.1, 0.0), (0.0, 0.0, 0.1), (1.0, 0.0, 0.0), [495.0]),
                      _sensor("ortho", case["film"], case["film"], (0.0, 0.0, 0.0), (1.0, 0.0, 0.0), (0.0, 0.0, 1.0),
                              (0.0, -1.0, 0.0)), case["film"] ** 2 * case["spp"], seed)
    elif kind == "sheet":
        n = case["grid"]
        conc = torch.stack([_blobs(rng, n, 500, n / 128, n / 32) for _ in range(4)])
        ab = [480.0, 495.0, 510.0, 530.0]
        dyes = _dyes(ab, 15.0, [520.0, 560.0, 600.0, 650.0], 20.0, [1.0] * 4, [0.9, 0.7, 0.6, 0.5])
        dyes["eps"] = np.full(4, 0.001 * 63.0 / dyes["abs_shape"][:, 22].sum(), np.float32)
        grids = {"conc": conc}
        desc = _scene(dyes, _medium(4, 0.999 * 63.0),
                      _source("collimated", (0.0, 0.0, 0.475), (0.0, 1.0, 0.0), (0.0, 0.0, 0.05), (1.0, 0.0, 0.0),
                              [488.0]), top(case["film"]), case["film"] ** 2 * case["spp"], seed)
    elif kind == "adjoint":
        n = case["grid"]
        st["conc"] = (torch.stack([_blobs(rng, n, 24, n * 3 / 64, n / 8) for _ in range(2)]) + 0.02).contiguous()
        st["sigma_s"] = torch.tensor(30.0)
        st["target"] = torch.full((case["film"], case["film"], N_BINS), 0.01, device="cuda")
        grids = {"conc": st["conc"]}
        desc = _scene(_dyes([470.0, 560.0], 15.0, [520.0, 610.0], 20.0, [2.0, 2.0], [0.8, 0.6]), _medium(2, 30.0),
                      _beam([470.0, 560.0]), top(case["film"]), case["film"] ** 2 * case["spp"], seed)
    else:
        n = case["grid"]
        grids = {"conc": torch.stack([_blobs(rng, n, 6, n * 1.5 / 16, n * 3 / 16) for _ in range(2)])}
        desc = _scene(_dyes([470.0, 560.0], 20.0, [520.0, 610.0], 25.0, [3.0, 2.0], [0.8, 0.6]),
                      _medium(2, 3.0, walls=0b000011, albedo=0.7), _beam([470.0, 560.0]),
                      _sensor("pinhole", case["film"], case["film"], (0.5, -1.0, 0.5), (1.0, 0.0, 0.0), (0.0, 0.0, 1.0),
                              (0.0, 1.0, 0.0), 50.0), case["film"] ** 2 * case["spp"], seed)
    st["desc"], st["grids"] = desc, grids
    st["scene"] = fs.Scene(desc, grids=grids)
    return st


def _read(s):
    t = s.read()
    t["counters"] = np.array(list(t["counters"].values()), np.int64)
    return t


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "batch":
        state["batch"].launch()
        t = state["batch"].read()
        t["counters"] = np.array(list(t["counters"].values()), np.int64)
        return t
    s = state["scene"]
    if kind == "adjoint":
        conc = state["conc"].detach().requires_grad_(True)
        sig = state["sigma_s"].detach().requires_grad_(True)
        film = fs.FluoroRender.apply(conc, sig, s, {"seed": state["desc"]["params"]["seed"]})
        loss = ((film - state["target"]) ** 2).sum()
        loss.backward()
        return {"film": film.detach(), "loss": loss.detach(), "grad_conc": conc.grad, "grad_sigma_s": sig.grad}
    if kind == "camera":
        film = s.render_camera()
        return {"film": film, "counters": np.array(list(s.read()["counters"].values()), np.int64)}
    if kind == "frames":
        s.set_medium(state["desc"]["medium"], state["grids"], stream=torch.cuda.current_stream())
        film = s.render(form="wavefront_warp", skip_cell=1)
    elif kind == "cornell":
        film = s.render(form=case["form"], skip_cell=case["cell"], hero=case["hero"])
    else:
        film = s.render(form="wavefront_warp")
    return {"film": film, **_read(s)}


def _film_values(case):
    if "width" in case:
        return case["width"] * case["height"] * N_BINS
    return case.get("film", 0) ** 2 * N_BINS


def work(case):
    kind = case["kind"]
    steps, events, conns, marches = UNITS[kind]
    if kind == "cornell" and not case["cell"]:
        steps, marches = 3.6 * steps, 3.5 * marches   # without leaps every null collision is sampled
    if kind == "batch":
        mean_edge = 0.5 * (16 + case["max_edge"])
        n_paths = case["media"] * (1e6 - 1e4) / math.log(100.0) * case["scale"]
        grid = case["media"] * 2 * 4 * mean_edge * (mean_edge ** 2 + (case["max_edge"] - 16) ** 2 / 4.0)
        out = case["media"] * 21 * N_BINS * 8
    else:
        n_paths = case.get("n_paths") or _film_values(case) // N_BINS * case["spp"]
        dyes = {"cornell": 4, "frames": 4, "sheet": 4, "adjoint": 2, "camera": 2, "vial": 1}.get(kind, 0)
        mask = 1 if kind in ("cornell", "frames", "vial") else 0
        grid = case.get("grid", 0) ** 3 * (4 * dyes + mask)
        out = 4 * _film_values(case)
    # operations of the method: a uniform, a logarithm and about ten fp32 operations a free flight; three
    # more uniforms, a direction and the collision type an event; projection and visibility a connection
    flops = n_paths * (26.0 * steps + 78.0 * events + 45.0 * conns + 26.0 * marches)
    if case.get("hero"):
        flops *= 1.3
    if kind == "adjoint":   # forward, then the replay of the contributions and of the scores
        flops, grid, out = 3.0 * flops, 2 * grid, 3 * out + grid
    return {"bytes": float(grid + out), "flops": float(flops)}


# The homogeneous cube in 64 bits ------------------------------------------------------------------


def _philox(pid, step, slot, seed):
    """Philox4x32-10 blocks of the counters (pid, step, slot, 0) under the key (seed, 0), as uniforms."""
    m32 = 0xFFFFFFFF
    c = [pid & m32, torch.full_like(pid, step), torch.full_like(pid, slot), pid >> 32]
    k0, k1 = seed & m32, 0

    def mul(a, x):   # 32 x 32 -> 64 bits in halves, without overflow of int64
        lo, hi = a * (x & 0xFFFF), a * (x >> 16)
        low = lo + ((hi & 0xFFFF) << 16)
        return ((hi >> 16) + (low >> 32)) & m32, low & m32

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return [(v >> 8).double() / 16777216.0 for v in c]


def exact(case, seed):
    """The cube's film and tallies with every quantity in 64 bits: the same random numbers, the closed-form
    transmittance. The other scenes decide on grid values at rounded positions and estimate transmittances by
    random marches: a 64-bit run of theirs leaves the 32-bit paths, and is another sample of the same mean."""
    if case["kind"] != "cube" or case["n_paths"] > 2_000_000:
        return None
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    n, nf, B, key = case["n_paths"], case["film"], N_BINS, int(seed) & 0x7FFFFFFF
    dy = _dyes([490.0], 15.0, [520.0], 20.0, [2.0], [0.9])
    sig_a = torch.from_numpy(2.0 * dy["abs_shape"][0].astype(np.float64)).to(dev)
    em = dy["emit_spec"][0].astype(np.float64)
    cdf, qy = torch.from_numpy(np.cumsum(em) / em.sum()).to(dev), float(dy["qy"][0])
    sig_s = 20.0
    film, face = torch.zeros(nf * nf * B, dtype=torch.float64, device=dev), torch.zeros(2 * 6 * B, dtype=torch.float64, device=dev)
    absorbed, emitted = (torch.zeros(B, dtype=torch.float64, device=dev) for _ in range(2))
    pid = torch.arange(n, device=dev)
    x = torch.tensor([0.5, 0.5, 1.0], dtype=torch.float64, device=dev).repeat(n, 1)
    w = torch.tensor([0.0, 0.0, -1.0], dtype=torch.float64, device=dev).repeat(n, 1)
    b = torch.full((n,), 22, device=dev)
    wt, fl = torch.ones(n, dtype=torch.float64, device=dev), torch.zeros(n, dtype=torch.int64, device=dev)
    for step in range(100_000):
        if pid.numel() == 0:
            break
        u_dist, _, u_event, u_d1 = _philox(pid, step, 0, key)
        u_d2, u_emit, u_rr, _ = _philox(pid, step, 1, key)
        total = sig_s + sig_a[b]
        t = torch.where(w == 0.0, torch.inf, (torch.where(w > 0.0, 1.0, 0.0) - x) / w).clamp_min(0.0)
        te, axis = t.min(1)
        tf = -torch.log1p(-u_dist) / total
        out = tf >= te
        f = 2 * axis + (w.gather(1, axis[:, None])[:, 0] > 0.0).long()
        face.index_add_(0, ((fl * 6 + f) * B + b)[out], wt[out])
        keep = ~out
        x, tf, u_event, u_d1, u_d2, u_emit, u_rr, total, b, wt, fl, pid, w = (
            v[keep] for v in (x, tf, u_event, u_d1, u_d2, u_emit, u_rr, total, b, wt, fl, pid, w))
        x = x + tf[:, None] * w
        dye = u_event * total >= sig_s
        absorbed.index_add_(0, b[dye], wt[dye])
        wt, b = torch.where(dye, wt * qy, wt), torch.where(dye, torch.searchsorted(cdf, u_emit, right=True).clamp_max(B - 1), b)
        emitted.index_add_(0, b[dye], wt[dye])
        fl = torch.where(dye, 1, fl)
        z, phi = 1.0 - 2.0 * u_d1, 2.0 * math.pi * u_d2
        r = torch.sqrt((1.0 - z * z).clamp_min(0.0))
        w = torch.stack([r * torch.cos(phi), r * torch.sin(phi), z], 1)
        tr = torch.exp(-(sig_s + sig_a[b]) * (1.0 - x[:, 2]).clamp_min(0.0))
        px, py = ((x[:, k] * nf).floor().long().clamp(0, nf - 1) for k in (0, 1))
        film.index_add_(0, (py * nf + px) * B + b, wt * tr * (nf * nf / (4.0 * math.pi * n)))
        if step + 1 >= 5:   # every step of a homogeneous medium is an event
            live = u_rr < wt.clamp_max(1.0)
            x, w, b, wt, fl, pid = (v[live] for v in (x, w, b, wt.clamp_min(1.0), fl, pid))
    shape = lambda v, *s: v.cpu().numpy().reshape(s) / n  # noqa: E731
    zero = torch.zeros_like(absorbed)
    return {"film": film.reshape(nf, nf, B).cpu().numpy(), "face": shape(face, 2, 6, B),
            "absorbed": shape(torch.cat([absorbed, zero]), 2, B), "emitted": shape(emitted, 1, B), "counters": None}
