"""Workloads of the library as its users run them, for timing and for comparing results.

A case is one run of a two-component lattice (or of a batch of them) between two outputs: `prepare` builds the
microstructure and the initial state from the seed and sets the lattice up, `run` advances it by the case's steps through
the C ABI and reads the result back, into pinned host arrays that the caller keeps, as a monitoring loop does. `exact`
states the same steps in 64 bits with plain torch operations (Eqs. 1, 3-7, A.3-A.6 of the method).

Cases are dicts of plain values:
  kind       "lattice" (lbm_step) or "batch" (the batched steps of the serving loop, `graph`: replayed from a CUDA graph)
  nx, ny, nz the lattice; edges: the batch's cubic lattices, "40 36 32"
  storage    population storage (lbm.STORAGES)
  medium     "electrode" solid grains, gray binder and reservoirs on the x faces, the pores half imbibed
             "droplet"   a sphere of fluid 1 in a uniform gray medium, periodic
             "channel"   a uniform gray medium between two reservoirs, the front part of the way in
             "layers"    stratified fluids along a body force, periodic
             "membrane"  bounce-back fractions per component between moving walls
  wave       wavefront shape given to lbm_set_wavefront (0: the library's default step)
  steps      time steps of one pass
  reads      what is read back: "fields", "densities", "populations" or "all" (fields and observables)
"""
import math

import numpy as np
import torch

from paper_2206_11524_gb300 import lbm

HI, LO = 0.99, 0.01          # majority and dissolved density
INLET = (1.04, 0.01)         # densities of the inlet and the outlet reservoir
OUTLET = (0.01, 0.99)
LAYERS = 4


def lattice(name, nx, ny, nz, storage, medium, steps, wave=0, reads="fields"):
    return {"name": name, "kind": "lattice", "nx": nx, "ny": ny, "nz": nz, "storage": storage, "medium": medium,
            "wave": wave, "steps": steps, "reads": reads}


def batch(name, edges, storage, steps, graph):
    return {"name": name, "kind": "batch", "edges": " ".join(str(e) for e in edges), "storage": storage,
            "steps": steps, "graph": graph}


def listed():
    return [
        # imbibition of a 1D gray medium, the front read every few hundred steps (Washburn study): pure launch latency
        lattice("capillary_500", 500, 1, 1, "f32", "channel", 200),
        # stratified 2D flow whose component fluxes come from the populations (relative permeability study)
        lattice("layers_50x50", 50, 50, 1, "f32", "layers", 200, reads="populations"),
        # a run monitored at every other step: the smallest call that moves a 3D lattice and reads everything back
        lattice("monitor_32x16x16", 32, 16, 16, "f32", "electrode", 2, reads="all"),
        # Laplace droplet at the study's size
        lattice("droplet_128", 128, 128, 128, "f32", "droplet", 20),
        # the benchmark's imbibition lattice in the library's default step
        lattice("electrode_256", 256, 256, 256, "f32", "electrode", 16),
        # and in the wavefront step, which the tuner picks for it
        lattice("electrode_256_wave", 256, 256, 256, "f32", "electrode", 16, wave=2),
        # the same lattice in local half offsets, the storage that keeps float32's saturation curve
        lattice("electrode_256_f16l", 256, 256, 256, "f16l", "electrode", 16),
        # the large domain in half offsets, the front read from the densities
        lattice("large_512x512x384", 512, 512, 384, "f16", "electrode", 8, reads="densities"),
        # membranes and porous obstacles: a fraction per component, moving walls, ragged edges
        lattice("membrane_150x90x70", 150, 90, 70, "f32", "membrane", 16),
        # ragged crop in the 16-bit format with float32's range
        lattice("ragged_97x131x61_bf16l", 97, 131, 61, "bf16l", "electrode", 16),
        # one tick of the serving loop, lattices of mixed sizes in a captured graph
        batch("serve_mixed", (160, 132, 112, 96, 80, 76, 64, 60, 52, 44, 40, 36), "f16l", 16, True),
        # the first steps of newly admitted small requests
        batch("serve_small", (48, 44, 40, 36, 32, 32), "f16l", 8, False),
    ]


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["thin", "box", "box", "batch"])
    if kind == "thin":           # the 1D and 2D studies
        nx, ny = spread(40, 640), rng.choice([1, 1, 5, spread(16, 100)])
        return {k: v for k, v in lattice("", nx, ny, 1, "f32", "channel" if ny == 1 else rng.choice(["channel", "layers"]),
                                         spread(20, 300), reads=rng.choice(["fields", "populations"])).items() if k != "name"}
    if kind == "batch":
        n = rng.randint(3, 12)
        edges = [4 * round(spread(32, 160) / 4) + rng.choice([0, 0, 0, 1, 2]) for _ in range(n)]
        return {k: v for k, v in batch("", edges, rng.choice(["f16l", "f16l", "f16", "f32"]), 2 * spread(2, 10),
                                       rng.random() < 0.6).items() if k != "name"}
    nodes = math.exp(rng.uniform(math.log(2e4), math.log(2e7)))
    storage = rng.choice(["f32", "f32", "f16", "f16l", "bf16", "bf16l"])
    a = nodes ** (1 / 3)
    nx, ny = (max(16, int(round(a * rng.uniform(0.6, 1.6)))) for _ in range(2))
    if rng.random() < 0.4:
        nx = 32 * max(1, round(nx / 32))
    nz = max(3, int(round(nodes / (nx * ny))))
    medium = rng.choice(["electrode", "electrode", "droplet", "membrane" if storage == "f32" else "electrode"])
    wave = rng.choice([0, 0, 0, 2]) if storage == "f32" else 0
    steps = max(2, min(spread(4, 40), int((3e8 if storage == "f32" else 6e8) / (nx * ny * nz))))
    return {k: v for k, v in lattice("", nx, ny, nz, storage, medium, steps, wave=wave).items() if k != "name"}


# ---- inputs ----------------------------------------------------------------------------------------------------------

def smooth_noise(shape, sigma, gen):
    """White noise under a periodic Gaussian of `sigma` nodes, scaled to unit variance."""
    a = torch.fft.rfftn(torch.randn(shape, generator=gen, device="cuda"))
    for d, n in enumerate(shape):
        k = torch.fft.rfftfreq(n, device="cuda") if d == 2 else torch.fft.fftfreq(n, device="cuda")
        a *= torch.exp(-2 * (math.pi * sigma * k) ** 2).reshape([-1 if e == d else 1 for e in range(3)])
    a = torch.fft.irfftn(a, s=shape)
    return a / a.std().clamp_min(1e-20) if a.numel() > 1 else a


def threshold(a, share):
    """The value that `share` of `a` lies above (from a strided sample)."""
    flat = a.flatten()
    flat = flat[::max(1, flat.numel() // 1_000_000)]
    return torch.quantile(flat, 1.0 - share)


def problem(medium, nx, ny, nz, seed):
    """Geometry, initial densities, faces and parameters: device float32 arrays [nz, ny, nx]."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    shape = (nz, ny, nx)

    def rand():
        return float(torch.rand((), generator=gen, device="cuda"))

    x = torch.arange(nx, device="cuda", dtype=torch.float32).expand(shape)
    y = torch.arange(ny, device="cuda", dtype=torch.float32)[None, :, None].expand(shape)
    z = torch.arange(nz, device="cuda", dtype=torch.float32)[:, None, None].expand(shape)
    full = torch.full(shape, 0.0, device="cuda")
    p = {"shape": shape, "tau": (1.0, 1.0), "G": 1.75, "F": (0.0, 0.0, 0.0), "faces": {}, "ns2": None, "gads": full}
    ripple = smooth_noise(shape, 2.0, gen)
    if medium == "electrode":
        # 60 % solid grains a dozen nodes wide, a fifth gray binder in patches of one fraction each
        grain = smooth_noise(shape, 3.5, gen)
        solid = grain > threshold(grain, 0.6)
        patch = smooth_noise(shape, 3.0, gen)
        gray = ~solid & (patch > threshold(patch, 0.5))
        frac = 0.2 + 0.7 * torch.sigmoid(2.0 * smooth_noise(shape, 6.0, gen))
        frac = torch.round(frac * 16) / 16
        open_ = (x < LAYERS) | (x >= nx - LAYERS)
        p["ns"] = torch.where(open_, full, torch.where(solid, full + 1.0, torch.where(gray, frac, full)))
        p["gads"] = torch.where(gray & ~open_, full + 0.214375, full)
        p["G"] = 1.5 + 0.5 * rand()
        wet = (x < nx * (0.3 + 0.3 * rand()) + 2.0 * ripple)
        p["faces"] = {0: (LAYERS, *INLET, None), 1: (LAYERS, *OUTLET, None)}
    elif medium == "droplet":
        c = [(n - 1) / 2 + rand() - 0.5 for n in (nz, ny, nx)]
        wet = (x - c[2]) ** 2 + (y - c[1]) ** 2 + (z - c[0]) ** 2 < (0.25 * min(s for s in shape if s > 1)) ** 2
        p["ns"] = full + 0.6 * rand()
    elif medium == "channel":
        inner = (x >= LAYERS) & (x < nx - LAYERS)
        p["ns"] = torch.where(inner, full + 0.1 + 0.8 * rand(), full)
        p["gads"] = torch.where(inner, full + 0.05 + 0.35 * rand(), full)
        wet = x < LAYERS + (nx - 2 * LAYERS) * (0.2 + 0.4 * rand())
        p["faces"] = {0: (LAYERS, HI, LO, None), 1: (LAYERS, LO, HI, None)}
    elif medium == "layers":
        p["ns"] = full + 0.1 + 0.8 * rand()
        p["F"] = (1e-5, 0.0, 0.0)
        wet = y < ny * (0.2 + 0.6 * rand())
    else:                        # "membrane": a slab only fluid 1 crosses, sheared by the y faces
        slab = ((x > 0.45 * nx) & (x < 0.55 * nx)).float()
        p["ns"] = 0.3 * rand() * torch.sigmoid(ripple)
        p["ns2"] = torch.maximum(p["ns"], slab)
        p["gads"] = 0.1 * slab
        p["tau"] = (1.0, 0.8)
        wet = x < 0.5 * nx
        p["faces"] = {2: (1, 0.5, 0.5, (0.0, 0.0, 0.0)), 3: (1, 0.5, 0.5, (0.02, 0.0, 0.01))}
    p["rho"] = (torch.where(wet, HI, LO) * (1.0 + 0.02 * torch.tanh(ripple)),
                torch.where(wet, LO, HI) * (1.0 - 0.02 * torch.tanh(ripple)))
    return p


def pinned(shape):
    return torch.empty(shape, dtype=torch.float32, pin_memory=True).numpy()


def set_up(p, storage, wave, reads, stream=None):
    """A lattice with geometry, boundaries and state, and the host arrays its results are read into."""
    nz, ny, nx = p["shape"]
    lat = lbm.Lattice(nx, ny, nz, tau=p["tau"], G=p["G"], F_ext=p["F"], storage=storage, rho0=(0.5, 0.5),
                      ns_per_component=p["ns2"] is not None, stream=stream)
    host = {k: p[k].cpu().numpy() for k in ("ns", "gads")}
    lat.set_geometry(host["ns"], host["gads"], None if p["ns2"] is None else p["ns2"].cpu().numpy())
    for face, (layers, a, b, u) in p["faces"].items():
        lat.set_bc(face, layers, a, b, u)
    lat.init_equilibrium(*(r.float().cpu().numpy() for r in p["rho"]))
    if wave:
        lat.set_wavefront(wave)
    out = {}
    if reads == "populations":
        out["f"] = np.zeros((2, 19) + lat.shape, np.float32)
    else:
        out = {"rho_a": pinned(lat.shape), "rho_b": pinned(lat.shape)}
        if reads != "densities":
            out |= {"u": pinned((3,) + lat.shape), "p": pinned(lat.shape)}
    return lat, out


def read(lat, out):
    if "f" in out:
        lbm.lbm_get_populations(lat.ctx, out["f"])
    else:
        lbm.lbm_read_fields(lat.ctx, out["rho_a"], out["rho_b"], out.get("u"), out.get("p"))


def batch_problems(case, seed):
    return [problem("electrode", int(e), int(e), int(e), seed * 64 + k) for k, e in enumerate(case["edges"].split())]


class Batch:
    def __init__(self, case, seed):
        self.stream, self.steps, self.graph = torch.cuda.Stream(), case["steps"], None
        made = [set_up(p, case["storage"], 0, "fields", self.stream) for p in batch_problems(case, seed)]
        self.lats, self.out = [m[0] for m in made], [m[1] for m in made]
        self.ctxs = [lat.ctx for lat in self.lats]
        if case["graph"]:        # a graph needs the reservoirs in force: the serving loop takes two plain steps first
            lbm.lbm_batch_step(self.ctxs, 2, self.stream.cuda_stream)
            self.graph = lbm.lbm_batch_graph_create(self.ctxs, self.steps, self.stream.cuda_stream)

    def __del__(self):
        if getattr(self, "graph", None):
            lbm.lbm_batch_graph_destroy(self.graph)


def prepare(case, seed):
    if case["kind"] == "batch":
        return Batch(case, seed)
    p = problem(case["medium"], case["nx"], case["ny"], case["nz"], seed)
    lat, out = set_up(p, case["storage"], case["wave"], case["reads"])
    return {"lat": lat, "out": out, "steps": case["steps"], "observe": case["reads"] == "all"}


def run(state):
    if isinstance(state, Batch):
        if state.graph:
            lbm.lbm_batch_graph_launch(state.graph, state.stream.cuda_stream)
        else:
            lbm.lbm_batch_step(state.ctxs, state.steps, state.stream.cuda_stream)
        for lat, out in zip(state.lats, state.out):
            read(lat, out)
        return state.out
    lat, out = state["lat"], state["out"]
    lbm.lbm_step(lat.ctx, state["steps"])
    read(lat, out)
    if state["observe"]:
        return {**out, "observables": lat.observables()}
    return out


# ---- cost ------------------------------------------------------------------------------------------------------------

def work(case):
    """Per pass: every step reads and writes each population once and reads the geometry; the outputs are written once."""
    size = 4 if case["storage"] == "f32" else 2
    if case["kind"] == "batch":
        nodes, medium, reads = sum(int(e) ** 3 for e in case["edges"].split()), "electrode", "fields"
    else:
        nodes, medium, reads = case["nx"] * case["ny"] * case["nz"], case["medium"], case["reads"]
    per_step = 2 * 38 * size + (12 if medium == "membrane" else 8)
    out = {"populations": 152, "densities": 8}.get(reads, 24)
    return {"bytes": nodes * (case["steps"] * per_step + out), "flops": nodes * case["steps"] * 600}


# ---- the same steps in 64 bits ---------------------------------------------------------------------------------------

# D3Q19 in the order of the populations: direction i + 9 is opposite to direction i, i = 1 .. 9
HALF = [(-1, 0, 0), (0, -1, 0), (0, 0, -1), (-1, -1, 0), (-1, 1, 0), (-1, 0, -1), (-1, 0, 1), (0, -1, -1), (0, -1, 1)]
C = [(0, 0, 0)] + HALF + [tuple(-v for v in c) for c in HALF]
W = [1 / 3 if not any(c) else 1 / 18 if sum(map(abs, c)) == 1 else 1 / 36 for c in C]


def shifted(a, c):
    """a at x - c (periodic)."""
    return torch.roll(a, (c[2], c[1], c[0]), (0, 1, 2)) if any(c) else a


def gradient(a):
    """sum_i w_i a(x + c_i) c_i."""
    g = [torch.zeros_like(a) for _ in range(3)]
    for c, w in zip(HALF, W[1:]):
        d = w * (shifted(a, tuple(-v for v in c)) - shifted(a, c))
        for k in range(3):
            if c[k]:
                g[k] += c[k] * d
    return g


def equilibrium(i, rho, u):
    cu = sum(C[i][k] * u[k] for k in range(3))
    return W[i] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * sum(v * v for v in u))


class Exact:
    def __init__(self, p):
        d = {k: p[k].double() for k in ("ns", "gads")}
        ns2 = d["ns"] if p["ns2"] is None else p["ns2"].double()
        self.ns, self.p = (d["ns"], ns2), p
        a1 = gradient(d["gads"] * d["ns"])
        self.adhesion = (a1, a1 if p["ns2"] is None else gradient(d["gads"] * ns2))
        self.rest = [r.float().double() for r in p["rho"]]
        self.f = [[W[i] * r for i in range(19)] for r in self.rest]

    def moments(self):
        """Densities, momenta and forces per unit mass."""
        rho = [torch.stack(f).sum(0) for f in self.f]
        j = [[sum(c[k] * f[i] for i, c in enumerate(C) if c[k]) for k in range(3)] for f in self.f]
        s = [gradient(r) for r in rho]
        total, G, F = rho[0] + rho[1], self.p["G"], self.p["F"]
        g = ([-G * s[1][k] + self.adhesion[0][k] + F[k] / total for k in range(3)],
             [-G * s[0][k] - self.adhesion[1][k] + F[k] / total for k in range(3)])
        return rho, j, g

    def step(self):
        rho, j, g = self.moments()
        tau, ns = self.p["tau"], self.ns
        den = rho[0] / tau[0] + rho[1] / tau[1]
        common = [(j[0][k] / tau[0] + j[1][k] / tau[1]) / den for k in range(3)]
        for s in range(2):
            u = [common[k] + tau[s] * g[s][k] for k in range(3)]
            f, new = self.f[s], [None] * 19
            for i in range(19):
                back = f[i] if i == 0 else f[i + 9] if i <= 9 else f[i - 9]
                post = (1 - ns[s]) * (f[i] - (f[i] - equilibrium(i, rho[s], u)) / tau[s]) + ns[s] * back
                new[i] = shifted(post, C[i]).contiguous()
            self.f[s] = new
        n = self.p["shape"]
        for face, (layers, a, b, u) in sorted(self.p["faces"].items()):
            axis = 2 - face // 2
            at = [slice(None)] * 3
            at[axis] = slice(0, layers) if face % 2 == 0 else slice(n[axis] - layers, n[axis])
            for s, r in enumerate((a, b)):
                for i in range(19):
                    self.f[s][i][tuple(at)] = equilibrium(i, r, u or (0.0, 0.0, 0.0))

    def fields(self):
        rho, j, g = self.moments()
        total = rho[0] + rho[1]
        u = [sum((1 - self.ns[s]) * (j[s][k] + 0.5 * rho[s] * g[s][k]) for s in range(2)) / total for k in range(3)]
        return {"rho_a": rho[0], "rho_b": rho[1], "u": torch.stack(u), "p": (total + self.p["G"] * rho[0] * rho[1]) / 3}


def exact_of(p, steps, reads):
    if p["shape"][0] * p["shape"][1] * p["shape"][2] * steps > 3e8:
        return None
    sim = Exact(p)
    for _ in range(steps):
        sim.step()
    if reads == "populations":
        return {"f": torch.stack([torch.stack(f) for f in sim.f])}
    out = sim.fields()
    if reads == "densities":
        return {k: out[k] for k in ("rho_a", "rho_b")}
    if reads == "all":           # observables: FP64 sums of the densities (Eq. 19, Eq. A.6)
        a, b, n = out["rho_a"], out["rho_b"], p["shape"]
        inner = torch.ones(n, dtype=torch.bool, device="cuda")
        face = np.full(6, np.nan)
        for k, (layers, *_) in p["faces"].items():
            axis = 2 - k // 2
            at = [slice(None)] * 3
            at[axis] = slice(0, layers) if k % 2 == 0 else slice(n[axis] - layers, n[axis])
            inner[tuple(at)] = False
            face[k] = float(out["p"][tuple(at)].mean())
        fluid = (1 - sim.ns[0]) * inner
        out["observables"] = {"mass": np.array([float(a.sum()), float(b.sum())]), "nonfinite": None, "p_face": face,
                              "sat1": float((fluid * (a >= 0.5)).sum() / fluid.sum())}
    return out


def exact(case, seed):
    if case["kind"] == "batch":
        steps = case["steps"] + (2 if case["graph"] else 0)
        return [exact_of(p, steps, "fields") for p in batch_problems(case, seed)]
    return exact_of(problem(case["medium"], case["nx"], case["ny"], case["nz"], seed), case["steps"], case["reads"])
