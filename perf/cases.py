"""The work that a user of this package has it do, as cases that can be timed
and whose outputs can be compared.

Every case goes through the public entry points: ``Simulator`` (scene upload
in ``prepare``, frames and maps in ``run``) and ``autograd.echo`` /
``autograd.range_doppler_map``.  Scene and radar sizes are those of
``scenegen``'s workloads, of the tests and of ``bench.py``, scaled up and
down.  ``exact`` restates the method in plain torch, in 64 bits: brute-force
visibility, the flat-facet integral as a divided difference taken over its
best-separated vertices, the delay of every sample.
"""
import math

import numpy as np
import torch

import paper_2208_10939_gb300 as pkg
import scenegen as sg
from paper_2208_10939_gb300 import autograd as bag

PATHS = {"fp64": pkg.PATH_FP64, "mixed": pkg.PATH_MIXED, "spectral": pkg.PATH_SPECTRAL}
DETECT = dict(guard_r=2, guard_d=2, train_r=8, train_d=4, pfa=1e-6, angle_bins=512)
MAX_POINTS = 1024
SNR_DB = 20.0
SCAN = 0.012             # metres
LIT = 0.3                # about the share of a vehicle's facets that a radar sees
DEV = "cuda"


def _car(name, path, ntri, M, N, P, Q, slant=30.0, speed=10.0, lane=0, tdm=False):
    return {"name": name, "kind": "frame", "scene": "car", "path": path, "ntri": ntri, "M": M,
            "N": N, "P": P, "Q": Q, "slant": slant, "speed": speed, "lane": lane, "tdm": tdm}


def listed():
    return [
        # the smallest frame in use: the 200-facet test plate, one TX; a call's latency
        {"name": "plate_frame", "kind": "frame", "scene": "plate", "path": "mixed", "n": 10,
         "M": 128, "N": 64, "P": 1, "Q": 4},
        # the frame of the paper's experiments: one sedan toward a 12-channel radar
        _car("sedan_frame", "mixed", 20_000, 256, 128, 3, 4),
        # the dataset generator's step: a batch of small scenes in one call
        {"name": "dataset_batch", "kind": "frame", "scene": "batch", "path": "mixed", "scenes": 8,
         "tri_max": 12_000, "M": 256, "N": 128},
        # the largest: the intersection with ground and twelve vehicles, 192 channels
        {"name": "intersection_frame", "kind": "frame", "scene": "intersection", "path": "mixed",
         "tri_scale": 0.25, "ground_n": 158, "vehicles": 12, "M": 512, "N": 64, "P": 12, "Q": 16},
        # the same scene by the inverse-FFT route, fewer channels
        {"name": "intersection_spectral", "kind": "frame", "scene": "intersection",
         "path": "spectral", "tri_scale": 0.25, "ground_n": 158, "vehicles": 12, "M": 512, "N": 64,
         "P": 2, "Q": 8},
        # the plain FP64 path, as one runs it to check a scene
        _car("car_fp64", "fp64", 5_000, 256, 32, 3, 4, slant=25.0, speed=8.0, tdm=True),
        # car and road with the two-facet paths
        {"name": "road_bounce", "kind": "frame", "scene": "road", "path": "mixed", "ntri": 20_000,
         "ground_size": 20.0, "ground_n": 40, "M": 256, "N": 128, "P": 3, "Q": 4},
        # one step of a mesh fit: map, loss, gradients of vertices and reflectivities
        {"name": "sedan_gradient", "kind": "gradient", "precision": "mixed", "ntri": 20_000,
         "M": 256, "N": 128, "P": 3, "Q": 4, "slant": 30.0, "speed": 10.0},
        # the same in FP64 on a coarse car
        {"name": "car_gradient_fp64", "kind": "gradient", "precision": "fp64", "ntri": 1_500,
         "M": 128, "N": 32, "P": 2, "Q": 4, "slant": 18.0, "speed": 8.0},
        # the map of a recorded cube: the 192-channel array
        {"name": "rdm_192", "kind": "rdm", "P": 12, "Q": 16, "N": 256, "M": 512, "double": False},
        # and the paper's 384-sample profile on 12 channels, in double precision
        {"name": "rdm_384", "kind": "rdm", "P": 3, "Q": 4, "N": 128, "M": 384, "double": True},
        # noise, CA-CFAR, angles: the point cloud of a recorded cube
        {"name": "point_cloud", "kind": "points", "P": 3, "Q": 4, "N": 128, "M": 256,
         "targets": 24},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plate", "car", "car", "car", "batch", "intersection", "gradient", "rdm",
                       "points", "road"])
    M, N = rng.choice([128, 192, 256, 384, 512]), rng.choice([16, 24, 32, 48, 64, 96, 128, 192])
    P, Q = rng.randint(1, 4), rng.randint(1, 6)
    if kind == "plate":
        return {"kind": "frame", "scene": "plate", "path": rng.choice(["mixed", "fp64"]),
                "n": rng.randint(3, 20), "M": M, "N": N, "P": 1, "Q": 4}
    if kind == "car":
        path = rng.choice(["mixed", "mixed", "spectral", "fp64"])
        small = path == "fp64"
        ntri = _log(rng, 600, 6_000) if small else _log(rng, 14_000, 40_000)
        c = _car("", path, ntri, M, min(N, 24) if small else N, P, Q, rng.uniform(20.0, 45.0),
                 rng.uniform(0.5, 10.0), rng.randint(0, 2), rng.random() < 0.25)
        del c["name"]
        return c
    if kind == "batch":
        return {"kind": "frame", "scene": "batch", "path": rng.choice(["mixed", "mixed", "spectral"]),
                "scenes": rng.randint(2, 12), "tri_max": _log(rng, 5_500, 60_000), "M": 256,
                "N": rng.choice([32, 64, 96, 128])}
    if kind == "intersection":
        return {"kind": "frame", "scene": "intersection", "path": rng.choice(["mixed", "spectral"]),
                "tri_scale": rng.uniform(0.05, 0.25), "ground_n": _log(rng, 79, 158),
                "vehicles": rng.randint(3, 12), "M": rng.choice([256, 384, 512]), "N": N, "P": P,
                "Q": Q}
    if kind == "gradient":
        double = rng.random() < 0.5
        return {"kind": "gradient", "precision": "fp64" if double else "mixed",
                "ntri": _log(rng, 600, 3_000) if double else _log(rng, 14_000, 20_000), "M": M,
                "N": min(N, 24) if double else N, "P": min(P, 2) if double else P, "Q": min(Q, 4),
                "slant": rng.uniform(18.0, 40.0), "speed": rng.uniform(0.5, 10.0)}
    if kind == "rdm":
        return {"kind": "rdm", "P": _log(rng, 1, 12), "Q": _log(rng, 1, 16),
                "N": rng.choice([32, 64, 96, 128, 256]), "M": M, "double": rng.random() < 0.3}
    if kind == "points":
        return {"kind": "points", "P": P, "Q": Q + 1, "N": max(N, 32), "M": M,
                "targets": rng.randint(4, 40)}
    return {"kind": "frame", "scene": "road", "path": "mixed", "ntri": _log(rng, 1_000, 20_000),
            "ground_size": rng.uniform(8.0, 20.0), "ground_n": rng.randint(8, 40), "M": M,
            "N": min(N, 64), "P": min(P, 3), "Q": min(Q, 4)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _scanned(scene, rng):
    """The scene with its surfaces as a scan gives them: the vertices off by
    about a centimetre, so that no panel is flat to a wavelength."""
    for m in scene.meshes:
        m.verts += rng.normal(scale=SCAN, size=m.verts.shape)
    return scene


def _scenes(case, seed):
    """The case's scenes: one, or a batch."""
    rng = np.random.default_rng(seed)
    kind = case.get("scene", "car")
    if kind == "plate":
        s = sg.plate_scene(range_m=float(rng.uniform(18.0, 22.0)), n=case["n"], M=case["M"],
                           N=case["N"])
        s.instances[0].rot = sg.rot_z(float(rng.uniform(-0.02, 0.02)))
        return [s]
    if kind == "batch":
        return [_scanned(sg.batch_scene(i, base_seed=4 + seed, M=case["M"], N=case["N"],
                                        tri_max=case["tri_max"]), rng)
                for i in range(case["scenes"])]
    if kind == "intersection":
        return [_scanned(sg.intersection_scene(
            seed=3 + seed, n_vehicles=case["vehicles"], M=case["M"], N=case["N"], P=case["P"],
            Q=case["Q"], ground_n=case["ground_n"], tri_scale=case["tri_scale"]), rng)]
    if kind == "road":
        return [sg.sedan_ground_scene(ground_size=case["ground_size"], ground_n=case["ground_n"],
                                      seed=2 + seed, ntri=case["ntri"], M=case["M"], N=case["N"],
                                      P=case["P"], Q=case["Q"])]
    # a mesh under fit keeps its topology: the seed moves its vertices
    fit = case["kind"] == "gradient"
    s = sg.car_scene(seed=2 if fit else 2 + seed, ntri=case["ntri"], slant=case["slant"], speed=case["speed"],
                     M=case["M"], N=case["N"], P=case["P"], Q=case["Q"], lane=case.get("lane", 0))
    s.radar.tdm = bool(case.get("tdm", False))
    if fit:
        s.meshes[0].rho[:] = rng.uniform(0.5, 1.0, size=s.meshes[0].rho.shape)
    return [_scanned(s, rng)]


def _recorded(case, seed):
    """A recorded cube: point echoes (beat, Doppler and channel phase
    progressions) over receiver noise."""
    O, N, M, targets = case["P"] * case["Q"], case["N"], case["M"], case.get("targets", 16)
    dtype = torch.complex128 if case.get("double") else torch.complex64
    g = torch.Generator(device=DEV).manual_seed(seed)
    u = torch.rand((targets, 5), generator=g, device=DEV, dtype=torch.float64)
    tone = lambda f, n: torch.exp(2j * math.pi * f[:, None] * torch.arange(n, device=DEV))  # noqa: E731
    amp = torch.exp(2j * math.pi * u[:, 0]) * 10 ** (-1.5 * u[:, 1])
    cube = torch.einsum("k,ko,kn,km->onm", amp, tone(0.4 * (u[:, 2] - 0.5), O),
                        tone(0.9 * (u[:, 3] - 0.5), N), tone(0.05 + 0.8 * u[:, 4], M))
    noise = torch.randn((2, O, N, M), generator=g, device=DEV, dtype=torch.float32)
    return (cube + 0.05 * torch.complex(noise[0], noise[1])).to(dtype).contiguous()


def _map_weights(case, seed):
    """Which range-Doppler cells the gradient cases weigh, and how much."""
    g = torch.Generator(device=DEV).manual_seed(seed + 77)
    return torch.rand((case["M"], case["N"]), generator=g, device=DEV, dtype=torch.float32)


GAIN = 1e8      # brings the echo's powers to the order of one


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "rdm":
        s["cube"] = _recorded(case, seed)
        s["sim"] = pkg.Simulator(0)
        s["sim"].load_scene(sg.car_scene(ntri=200, M=case["M"], N=case["N"], P=case["P"],
                                         Q=case["Q"]))
        return s
    s["sim"] = sim = pkg.Simulator(0)
    if case["kind"] == "points":
        sim.load_scene(sg.car_scene(ntri=200, M=case["M"], N=case["N"], P=case["P"], Q=case["Q"]))
        s["cube"] = _recorded(case, seed)
        s["seed"] = seed
        return s
    scenes = _scenes(case, seed)
    if case["kind"] == "gradient":
        sc = scenes[0]
        s["es"] = bag.EchoScene(sim, sc, case["precision"])
        s["base"] = s["es"].vertex_tensor(sc, DEV)
        fit = torch.float32 if case["precision"] == "mixed" else torch.float64
        s["offset"] = torch.zeros(s["base"].shape, dtype=fit, device=DEV, requires_grad=True)
        s["rho"] = torch.tensor(sc.meshes[0].rho, device=DEV, requires_grad=True)
        s["weights"] = _map_weights(case, seed)
        return s
    if len(scenes) > 1:
        sim.load_scenes(scenes)
    else:
        sim.load_scene(scenes[0])
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    case = state["case"]
    if case["kind"] == "rdm":
        return {"rdm": state["sim"].rdm(state["cube"])}
    sim = state["sim"]
    if case["kind"] == "points":
        noisy = sim.add_noise(state["cube"].clone(), SNR_DB, state["seed"])
        pts, n = sim.detect(noisy, max_points=MAX_POINTS, **DETECT)
        table = np.zeros(MAX_POINTS, pkg.POINT_DTYPE)
        table[:len(pts)] = pts
        return {"cube": noisy, "n": n, **{k: table[k] for k in table.dtype.names}}
    if case["kind"] == "gradient":
        offset, rho = state["offset"], state["rho"]
        offset.grad = rho.grad = None
        adc = bag.echo(state["base"] + offset.double(), rho, state["es"])
        rdm = bag.range_doppler_map(adc * GAIN, sim)
        loss = (state["weights"] * rdm).sum()
        loss.backward()
        return {"loss": loss.detach(), "verts": offset.grad, "rho": rho.grad}
    adc = sim.simulate(PATHS[case["path"]])
    return {"adc": adc, "rdm": sim.rdm(adc)}


def work(case):
    """Bytes: the inputs read once, the outputs written once.  Operations: the
    cube as a fast non-uniform transform of the lit facets (5 log2 per sample
    as in an FFT, and about 100 per lit facet and channel), once more for the
    map; a gradient pass takes both directions."""
    O = case.get("P", 3) * case.get("Q", 4)
    cells = case["N"] * case["M"]
    word = 16 if case.get("double") or "fp64" in (case.get("path"), case.get("precision")) else 8
    fft = 5.0 * math.log2(cells) * O * cells
    if case["kind"] in ("rdm", "points"):
        return {"bytes": word * O * cells * (1 if case["kind"] == "rdm" else 2) + 4 * cells,
                "flops": fft}
    copies = case.get("scenes", 1)
    if case.get("scene") == "plate":
        F = 2 * case["n"] ** 2
    elif case.get("scene") == "intersection":
        F = case["vehicles"] * 95_000 * case["tri_scale"] + 2 * case["ground_n"] ** 2
    elif case.get("scene") == "batch":
        F = copies * 0.5 * (5_000 + case["tri_max"])
    else:
        F = case["ntri"] + (2 * case["ground_n"] ** 2 if "ground_n" in case else 0)
    both = 2 if case["kind"] == "gradient" else 1
    return {"bytes": both * (40.0 * F + copies * (word * O + 4) * cells),
            "flops": both * (2 * copies * fft + 100.0 * LIT * F * O)}


# ---------------------------------------------------------------------------
# the method in plain torch, 64 bits
# ---------------------------------------------------------------------------
C0 = 299_792_458.0


def _t(a):
    return torch.as_tensor(np.asarray(a), dtype=torch.float64, device=DEV)


def _facets(scene, local=None):
    """World vertices at the frame start (F, 3, 3), velocities, reflectivities."""
    tri, vel, rho = [], [], []
    for i, ins in enumerate(scene.instances):
        m = scene.meshes[ins.mesh_id]
        v = _t(m.verts) if local is None else local
        w = v @ _t(ins.rot).T + _t(ins.pos) + _t(ins.vel) * scene.t0
        tri.append(w[torch.as_tensor(m.tris, dtype=torch.int64, device=DEV)])
        vel.append(_t(ins.vel).expand(m.nf, 3))
        rho.append(_t(m.rho) * ins.rho_scale)
    return torch.cat(tri), torch.cat(vel), torch.cat(rho)


def _lit(tri, ants, eps=1e-6, margin=1e-9):
    """(A, F): facets that face the antenna with nothing on the way."""
    c = tri.mean(1)
    e1, e2 = tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0]
    n = torch.linalg.cross(e1, e2)
    out = []
    for p in ants:
        D = p - c
        cos = (n * D).sum(1) / (n.norm(dim=1) * D.norm(dim=1))
        lit = cos >= eps
        for ids in torch.nonzero(lit)[:, 0].split(max(1, 40_000_000 // tri.shape[0])):
            d, o = D[ids][:, None], c[ids][:, None]
            dot = lambda a, b: a[..., 0] * b[..., 0] + a[..., 1] * b[..., 1] + a[..., 2] * b[..., 2]  # noqa: E731
            cross = lambda a, b: (a[..., 1] * b[..., 2] - a[..., 2] * b[..., 1],  # noqa: E731
                                  a[..., 2] * b[..., 0] - a[..., 0] * b[..., 2],
                                  a[..., 0] * b[..., 1] - a[..., 1] * b[..., 0])
            dot3 = lambda a, b: a[0] * b[..., 0] + a[1] * b[..., 1] + a[2] * b[..., 2]  # noqa: E731
            pv = cross(d, e2[None])
            det = dot3(pv, e1[None])
            t = o - tri[None, :, 0]
            u = dot3(pv, t) / det
            qv = cross(t, e1[None])
            v = dot3(qv, d) / det
            w = dot3(qv, e2[None]) / det
            hit = ((det != 0) & (u >= -margin) & (v >= -margin) & (u + v <= 1 + margin)
                   & (w >= -margin) & (w <= 1 + margin))
            hit[torch.arange(len(ids), device=DEV), ids] = False
            lit[ids] &= ~hit.any(1)
        out.append(lit)
    return torch.stack(out)


def _divided_difference(a):
    """Integral of exp(j a) over the unit simplex for the phases a (..., 3),
    ascending in magnitude order along the last axis."""
    spread = a[..., 2] - a[..., 0]
    near = spread.abs() < 1.0
    f = lambda x, y: 1j * torch.exp(0.5j * (x + y)) * torch.sinc((x - y) / (2 * math.pi))  # noqa: E731
    far = (f(a[..., 1], a[..., 2]) - f(a[..., 0], a[..., 1])) / torch.where(
        near, torch.ones_like(spread), spread)
    mean = a.mean(-1)
    y = [torch.where(near, a[..., i] - mean, torch.zeros_like(mean)) for i in range(3)]
    e2, e3 = y[0] * y[1] + y[0] * y[2] + y[1] * y[2], y[0] * y[1] * y[2]
    h = [torch.ones_like(e2), torch.zeros_like(e2), -e2]
    for p in range(3, 18):
        h.append(-e2 * h[p - 2] + e3 * h[p - 3])
    series = sum((1j ** p) * h[p] / math.factorial(p + 2) for p in range(18))
    return torch.where(near, torch.exp(1j * mean) * series, -far)


def _rows(radar, tri, vel, rho, p, q, n):
    """Sum over the facets of Eq. 13 for channel (p, q), chirps n: (len(n), M)."""
    k_m = torch.arange(radar.M, device=DEV, dtype=torch.float64) / radar.fs
    f_m = radar.f0 + radar.slope * k_m
    slots, slot = (radar.P, p) if radar.tdm else (1, 0)
    tn = (n.double() * slots + slot) * radar.Tc
    pt, pr = _t(radar.tx[p]), _t(radar.rx[q])
    c, dv = tri.mean(1), tri - tri.mean(1, keepdim=True)
    nrm = torch.linalg.cross(tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0])
    area2 = nrm.norm(dim=1)
    nrm = nrm / area2[:, None]
    cn = c[:, None] + vel[:, None] * tn[None, :, None]                  # (K, n, 3)
    Rt, Rr = (pt - cn).norm(dim=-1), (pr - cn).norm(dim=-1)
    b = (pt - cn) / Rt[..., None] + (pr - cn) / Rr[..., None]
    g = rho[:, None] * 0.5 * (b * nrm[:, None]).sum(-1) / (Rt * Rr) * area2[:, None]
    u = torch.einsum("knc,kvc->knv", b, dv).sort(dim=-1).values
    J = _divided_difference(-(2 * math.pi / C0) * f_m[None, None, :, None] * u[:, :, None, :])
    at = cn[:, :, None] + vel[:, None, None] * (k_m if radar.intra_chirp_motion else 0 * k_m)[
        None, None, :, None]
    tau = ((pt - at).norm(dim=-1) + (pr - at).norm(dim=-1)) / C0
    th = f_m * tau - 0.5 * radar.slope * tau * tau
    amp = 2 * math.sqrt(math.pi) / (4 * math.pi) ** 1.5
    return amp * (g[..., None] * J * torch.exp(2j * math.pi * (th - th.detach().round()))).sum(0)


def _chunks(radar, K):
    return torch.arange(radar.N, device=DEV).split(max(1, 6_000_000 // max(1, K * radar.M)))


def _echo(scene):
    r = scene.radar
    tri, vel, rho = _facets(scene)
    lit = _lit(tri, _t(r.antennas))
    out = torch.zeros((r.O, r.N, r.M), dtype=torch.complex128, device=DEV)
    for p in range(r.P):
        for q in range(r.Q):
            k = torch.nonzero(lit[p] & lit[r.P + q])[:, 0]
            for n in _chunks(r, len(k)):
                out[p * r.Q + q, n] = _rows(r, tri[k], vel[k], rho[k], p, q, n)
    return out


def _map(cube):
    hann = lambda n: _t(0.5 - 0.5 * np.cos(2 * np.pi * np.arange(n) / (n - 1)))  # noqa: E731
    x = torch.fft.fft(cube.to(torch.complex128) * hann(cube.shape[2]), dim=2)
    y = torch.fft.fftshift(torch.fft.fft(x * hann(cube.shape[1])[:, None], dim=1), dim=1)
    return (y.real ** 2 + y.imag ** 2).sum(0).T


def exact(case, seed):
    if case["kind"] == "rdm":
        return {"rdm": _map(_recorded(case, seed))}
    if case["kind"] == "points" or case.get("scene") in ("intersection", "road"):
        return None             # the noise's own values; two-facet paths and large scenes: too long
    scenes = _scenes(case, seed)
    terms = sum(LIT * s.nf * s.radar.O * s.radar.N * s.radar.M for s in scenes)
    if case["kind"] == "gradient":
        if terms > 3e9:
            return None
        sc = scenes[0]
        r = sc.radar
        cube = (_echo(sc) * GAIN).requires_grad_(True)
        loss = (_map_weights(case, seed).double() * _map(cube)).sum()
        loss.backward()
        G = cube.grad * GAIN
        offset = _t(sc.meshes[0].verts).requires_grad_(True)
        rho = _t(sc.meshes[0].rho).requires_grad_(True)
        lit = _lit(_facets(sc)[0], _t(r.antennas))
        for p in range(r.P):
            for q in range(r.Q):
                k = torch.nonzero(lit[p] & lit[r.P + q])[:, 0]
                for n in _chunks(r, len(k)):
                    tri, vel, _ = _facets(sc, offset)
                    rows = _rows(r, tri[k], vel[k], rho[k], p, q, n)
                    (rows * G[p * r.Q + q, n].conj()).real.sum().backward()
        return {"loss": loss.detach(), "verts": offset.grad, "rho": rho.grad}
    if terms > 1.5e10:
        return None
    cubes = [_echo(s) for s in scenes]
    maps = [_map(c) for c in cubes]
    return {"adc": torch.stack(cubes) if len(cubes) > 1 else cubes[0],
            "rdm": torch.stack(maps) if len(maps) > 1 else maps[0]}
