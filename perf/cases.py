"""The calls that a user of the library spends time in, as measured cases.

Four kinds of work, each through the public binding:

* ``ladder``  -- one pore throat from rest: reset the densities, run a pressure
  ladder, read its rows and the density field back (FP32 or 16-bit storage).
* ``box``     -- a domain that lives on: new reservoir densities, a stretch of
  time steps, the measurements and the density field.
* ``batch``   -- the per-throat simulations of a packing in one call.
* ``train``, ``predict``, ``throats`` -- the surrogate network: training an
  ensemble, evaluating it on prepared inputs, and on throats given as spheres.

``exact`` restates the time step and the network in 64-bit torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1906_04722_gb300 as lbm
from paper_1906_04722_gb300 import surrogate as lbm_surrogate

MAJOR, MINOR, G = 2.0, 0.06, 0.9
G_ADS = (-0.3, 0.3)
SOLID, ADHESIVE, MEMBRANE, INLET, OUTLET = 1, 2, 4, 8, 16
ROW_KEYS = ("p_c", "p_c_res", "S_w", "p_w", "p_nw", "phi_probe")
MEASURED = ("p_w", "p_nw", "p_c", "p_in", "p_out", "p_c_res", "S_w")
COUNTED = ("n_fluid", "n_w", "n_interface", "n_bulk_w", "n_bulk_nw")
N_IN, N_OUT = 24, 33  # a throat's network inputs; p_c^e and a 32-increment curve


def listed():
    return [
        # the single pore throat of the tests and of the plain per-throat loop: 32^3, three
        # touching spheres, 20 increments of 25 steps; about 500 launches of a few microseconds
        {"name": "throat32 fp32", "kind": "ladder", "precision": 0, "incr": 20, "steps": 25},
        # the same throat in 16-bit deviation storage
        {"name": "throat32 fp16", "kind": "ladder", "precision": 1, "incr": 20, "steps": 25},
        # a static drop in a periodic box (interfacial tension by Laplace's law)
        {"name": "drop 48", "kind": "box", "scene": "drop", "nx": 48, "ny": 48, "nz": 48, "precision": 0,
         "steps": 200, "tuned": False},
        # body-force-driven flow through a packing, periodic along z, ragged box, unequal
        # relaxation times, the kernel a new domain starts with
        {"name": "flow 101x90x77", "kind": "box", "scene": "flow", "nx": 101, "ny": 90, "nz": 77, "precision": 0,
         "steps": 100, "tuned": False},
        # the drainage sample of the benchmark, tuned on the domain as the README shows:
        # one stretch of a pressure increment
        {"name": "sample192 fp32", "kind": "box", "scene": "drain", "nx": 192, "ny": 192, "nz": 192, "precision": 0,
         "steps": 100, "tuned": True},
        # the same in FP16 deviations
        {"name": "sample192 fp16", "kind": "box", "scene": "drain", "nx": 192, "ny": 192, "nz": 192, "precision": 1,
         "steps": 100, "tuned": True},
        # per-throat simulations of a packing: a handful (a rank's share, or the throats the
        # surrogate is unsure of), a few hundred, and the benchmark's 1024
        {"name": "batch 16", "kind": "batch", "n": 16, "incr": 10, "steps": 50},
        {"name": "batch 256", "kind": "batch", "n": 256, "incr": 4, "steps": 100},
        {"name": "batch 1024", "kind": "batch", "n": 1024, "incr": 4, "steps": 100},
        # the benchmark's ensemble on about the throats of six packings, a few epochs of it
        {"name": "train 6000", "kind": "train", "n": 6000, "epochs": 4, "batch": 256, "n_in": N_IN, "n_out": N_OUT,
         "hidden": 256, "layers": 4, "members": 5, "half": False},
        # inference on the throats of four 2000-sphere packings, inputs at hand
        {"name": "predict 100000", "kind": "predict", "n": 100000, "n_in": N_IN, "n_out": N_OUT, "hidden": 256,
         "layers": 4, "members": 5, "half": False},
        # inference from sphere triples: the lattice description of each box, then the network
        {"name": "throats 2000", "kind": "throats", "n": 2000, "half": False},
    ]


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["ladder", "box", "box", "box", "batch", "batch", "train", "predict", "throats"])
    if kind == "ladder":
        return {"kind": kind, "precision": rng.choice([0, 1, 2]), "incr": spread(4, 24), "steps": spread(10, 60)}
    if kind == "box":
        nx, ny, nz = spread(24, 180), spread(24, 180), spread(24, 180)
        if rng.random() < 0.5:
            nx = nx // 4 * 4
        scene = rng.choice(["drain", "drain", "drop", "flow"])
        steps = max(20, min(spread(40, 400), 100 * 192 ** 3 // (nx * ny * nz)))
        return {"kind": kind, "scene": scene, "nx": nx, "ny": ny, "nz": nz,
                "precision": rng.choice([0, 0, 0, 1, 2]), "steps": steps, "tuned": nx * ny * nz >= 1 << 20}
    if kind == "batch":
        n = spread(1, 700)
        return {"kind": kind, "n": n, "incr": spread(2, 8), "steps": spread(15, 60)}
    net = {"n_in": rng.choice([7, N_IN]), "n_out": rng.choice([17, N_OUT]), "hidden": rng.choice([64, 96, 128, 256]),
           "layers": rng.choice([2, 3, 4]), "members": rng.choice([1, 2, 3, 5, 8]), "half": rng.random() < 0.5}
    if kind == "train":
        n = spread(500, 6000)
        return {"kind": kind, "n": n, "epochs": rng.choice([1, 2, 3]), "batch": min(n, rng.choice([64, 100, 128, 256, 300])),
                **net}
    if kind == "predict":
        return {"kind": kind, "n": spread(100, 100000), **net, "members": rng.choice([2, 3, 5])}
    return {"kind": kind, "n": spread(30, 2000), "half": rng.random() < 0.5}


# ------------------------------------------------------------------- inputs
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _packing(rng, n, box, rmin, rmax):
    """n non-overlapping spheres (fewer if the box will not take them), one after another."""
    box = np.asarray(box, dtype=float)
    got = np.empty((0, 4))
    for _ in range(200 * n):
        r = rng.uniform(rmin, rmax)
        c = r + rng.uniform(size=3) * np.maximum(box - 2 * r, 0.0)
        if len(got) == 0 or np.all(((got[:, :3] - c) ** 2).sum(1) >= (got[:, 3] + r) ** 2):
            got = np.vstack([got, [*c, r]])
            if len(got) == n:
                break
    return got


def _throats(seed, n):
    """n throats of a 192^3 packing of 300 spheres (several packings where one has too few)."""
    rng = np.random.default_rng(seed)
    out = []
    while n > 0:
        sp = _packing(rng, 300, (192, 192, 192), 10.0, 14.0)
        take = min(n, 1500)
        out.append(lbm.packing_throat_sample(sp, take, int(rng.integers(1 << 30))))
        n -= take
    return np.concatenate(out)


def _grain(shape, spheres, origin=(0.0, 0.0, 0.0), dev="cpu"):
    """Cells whose centre lies in a sphere."""
    nz, ny, nx = shape
    ax = [torch.arange(m, dtype=torch.float64, device=dev) + o for m, o in zip((nx, ny, nz), origin)]
    out = torch.zeros(shape, dtype=torch.bool, device=dev)
    for cx, cy, cz, r in np.asarray(spheres).tolist():
        lo = [max(0, math.floor(c - r - o) - 1) for c, o in zip((cx, cy, cz), origin)]
        hi = [min(m, math.ceil(c + r - o) + 2) for c, o, m in zip((cx, cy, cz), origin, (nx, ny, nz))]
        if any(h <= l for l, h in zip(lo, hi)):
            continue
        dx, dy, dz = (ax[d][lo[d]:hi[d]] - c for d, c in enumerate((cx, cy, cz)))
        d2 = (dx * dx)[None, None, :] + (dy * dy)[None, :, None] + (dz * dz)[:, None, None]
        out[lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]] |= d2 <= r * r
    return out


def _outside_prism(shape, c, origin=(0.0, 0.0, 0.0)):
    """Cells outside the triangular prism through the centres c (3 x 3)."""
    nz, ny, nx = shape
    p = np.stack(np.meshgrid(*[np.arange(m) + o for m, o in zip((nx, ny, nz), origin)], indexing="ij"), -1)
    n = np.cross(c[1] - c[0], c[2] - c[0])
    out = np.zeros(p.shape[:3], dtype=bool)
    for i in range(3):
        inward = np.cross(n, c[(i + 1) % 3] - c[i])
        rel = p - c[i]
        out |= (rel[..., 0] * inward[0] + rel[..., 1] * inward[1]) + rel[..., 2] * inward[2] < 0.0
    return out.transpose(2, 1, 0)


def _throat32():
    R = 20.0 / math.sqrt(3.0)
    return np.array([(16.0 + R * math.cos(t), 16.0 + R * math.sin(t), 16.0, 10.0)
                     for t in map(math.radians, (90.0, 210.0, 330.0))])


def _noise(shape, seed):
    g = torch.Generator(device=_device()).manual_seed(int(seed))
    return 1.0 + 1e-3 * torch.randn((2,) + tuple(shape), generator=g, device=_device(), dtype=torch.float64)


def _two_phase(non_wetting, seed):
    """Densities (wetting, non-wetting) of a phase map, with a little noise."""
    hi, lo = torch.full_like(non_wetting, MAJOR, dtype=torch.float64), torch.full_like(non_wetting, MINOR, dtype=torch.float64)
    rho = torch.stack([torch.where(non_wetting, lo, hi), torch.where(non_wetting, hi, lo)])
    return rho * _noise(non_wetting.shape, seed)


def _box_scene(case, seed):
    """(mask, densities, make_params arguments) of a box case."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    shape, dev = (nz, ny, nx), _device()
    rng = np.random.default_rng(seed)
    mask = torch.zeros(shape, dtype=torch.uint8, device=dev)
    z, y, x = torch.meshgrid(*[torch.arange(m, device=dev) for m in shape], indexing="ij")
    par = {}
    if case["scene"] == "drop":
        r = 0.25 * min(shape)
        phase = (x - nx / 2) ** 2 + (y - ny / 2) ** 2 + (z - nz / 2) ** 2 < r * r
        par = {"G_ads": (0.0, 0.0), "periodic": (1, 1, 1)}
    else:
        rmax = min(14.0, 0.3 * min(shape))
        spheres = _packing(rng, max(1, round(300 * nx * ny * nz / 192 ** 3)), (nx, ny, nz), rmax * 10 / 14, rmax)
        mask[_grain(shape, spheres, dev=dev)] = SOLID | ADHESIVE
        if case["scene"] == "flow":
            phase = (x + y + z) % 40 < 16  # slugs of both fluids
            par = {"periodic": (0, 0, 1), "body_force": (0.0, 0.0, 2e-5), "tau": (1.0, 1.2)}
        else:
            phase = z < 0.4 * nz  # the front of a drainage under way
            open_ = mask == 0
            mask[0][open_[0]] = INLET
            mask[nz - 1][open_[nz - 1]] = OUTLET
            mask[nz - 4:nz - 1][open_[nz - 4:nz - 1]] = MEMBRANE
    return mask, _two_phase(phase, seed), par


def _he_normal(case, seed):
    """Parameters of each member, flat (W_0, b_0, W_1, ...), He-normal weights and small biases."""
    rng = np.random.default_rng(seed)
    sizes = [case["n_in"]] + [case["hidden"]] * case["layers"] + [case["n_out"]]
    out = []
    for _ in range(case["members"]):
        flat = []
        for a, b in zip(sizes[:-1], sizes[1:]):
            flat += [rng.standard_normal(a * b) * math.sqrt(2.0 / a), 0.05 * rng.standard_normal(b)]
        out.append(np.concatenate(flat).astype(np.float32))
    return out, sizes


def _samples(case, seed):
    """Standardised inputs and smooth targets of them."""
    rng = np.random.default_rng(seed + 1)
    X = rng.standard_normal((case["n"], case["n_in"])).astype(np.float32)
    mix = rng.standard_normal((case["n_in"], case["n_out"])) / math.sqrt(case["n_in"])
    return X, np.tanh(X @ mix).astype(np.float32)


def _ladder(case, step):
    return [MAJOR + step * i for i in range(case["incr"])]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ladder":
        shape = (32, 32, 32)
        par = lbm.make_params(reservoirs=True, prism_clip=True, precision=case["precision"])
        inlet = torch.zeros(shape, dtype=torch.bool, device=_device())
        inlet[0] = True
        return {"kind": kind, "dom": lbm.Domain(par, _throat32(), (32, 32, 32)),
                "rho": _two_phase(inlet, seed).cpu().numpy(), "ladder": _ladder(case, 0.01), "steps": case["steps"]}
    if kind == "box":
        mask, rho, par = _box_scene(case, seed)
        dom = lbm.Domain(lbm.make_params(precision=case["precision"], **par), mask=mask.cpu().numpy())
        dom.set_densities(rho.cpu().numpy())
        if case["tuned"]:
            dom.autotune(8)
        return {"kind": kind, "dom": dom, "steps": case["steps"], "drain": case["scene"] == "drain"}
    if kind == "batch":
        return {"kind": kind, "throats": _throats(seed, case["n"]), "params": lbm.make_params(),
                "ladder": _ladder(case, 0.06), "steps": case["steps"]}
    if kind == "throats":
        known = _throats(seed, 200)
        r = np.maximum(lbm.lbm_throat_incircle(known), 0.5)
        net = lbm_surrogate.ThroatSurrogate(n_incr=N_OUT - 1, theta=0.8, half=case["half"], seed=seed)
        level = np.linspace(0.2, 2.0, N_OUT - 1)
        blank = {k: 0.0 for k in ("rho_in_nw", "p_c", "p_c_res", "p_w", "p_nw", "phi_probe")}
        net.fit(known, [{"p_ce": 0.1 / v, "invaded_at": 3, "n_fluid": 1000} for v in r],
                [[{**blank, "S_w": float(1.0 / (1.0 + level[k] * v)), "n_interface": 0} for k in range(N_OUT - 1)]
                 for v in r], epochs=10, batch=64)
        return {"kind": kind, "net": net, "throats": _throats(seed + 1, case["n"])}
    params, _ = _he_normal(case, seed)
    net = lbm.Surrogate(case["n_in"], case["n_out"], n_hidden=case["hidden"], n_layers=case["layers"],
                        n_members=case["members"], half=case["half"], seed=seed)
    for m, flat in enumerate(params):
        net.set_params(m, flat)
    X, T = _samples(case, seed)
    return {"kind": kind, "net": net, "X": X, "T": T, "members": case["members"],
            "epochs": case.get("epochs"), "batch": case.get("batch")}


# --------------------------------------------------------------------- runs
def run(state):
    kind = state["kind"]
    if kind == "ladder":
        dom = state["dom"]
        dom.set_densities(state["rho"])
        got = dom.drainage(state["ladder"], state["steps"], MAJOR, (16, 16, 29))
        return {"rows": np.array([[r[k] for k in ROW_KEYS] for r in got["rows"]]),
                "n_interface": np.array([r["n_interface"] for r in got["rows"]]),
                "p_ce": got["p_ce"], "invaded_at": got["invaded_at"], "density": dom.density()}
    if kind == "box":
        dom = state["dom"]
        if state["drain"]:
            dom.set_pressure_bc(2.1, MAJOR)
        dom.step(state["steps"])
        m = dom.measure(allow_nonfinite=True)
        return {"mass": np.array(m["mass"]), "measured": np.array([m[k] for k in MEASURED]),
                "counted": np.array([m[k] for k in COUNTED]), "density": dom.density()}
    if kind == "batch":
        res, rows = lbm.lbm_run_throat_batch(state["throats"], state["params"], state["ladder"], state["steps"], MAJOR)
        return {"rows": np.array([[[r[k] for k in ROW_KEYS] for r in t] for t in rows]),
                "n_interface": np.array([[r["n_interface"] for r in t] for t in rows]),
                "p_ce": np.array([r["p_ce"] for r in res]), "invaded_at": np.array([r["invaded_at"] for r in res]),
                "n_fluid": np.array([r["n_fluid"] for r in res])}
    if kind == "throats":
        pce, rel, curves = state["net"].predict(state["throats"])
        return {"p_ce": pce, "spread": rel, "curves": curves}
    net = state["net"]
    if kind == "train":
        loss = net.train(state["X"], state["T"], state["epochs"], state["batch"], 1e-3, seed=3)
        return {"loss": loss, "params": np.stack([net.get_params(m) for m in range(state["members"])])}
    mean, spread = net.predict(state["X"])
    return {"mean": mean, "spread": spread}


def work(case):
    """Time steps: every population of a non-solid cell read once and written once a step (2 x 19 values, or 19
    pair words and the density pair in 16-bit storage), about 500 operations each.  The networks: inputs and outputs
    (and a step's parameters, gradients and moments), two operations a weight and sample, three times that in training."""
    kind = case["kind"]
    if kind in ("ladder", "box", "batch"):
        if kind == "ladder":
            cells, steps = 3342, case["incr"] * case["steps"]  # open cells of the throat
        elif kind == "batch":
            cells, steps = 8300 * case["n"], case["incr"] * case["steps"]  # an average throat's open cells
        else:
            cells, steps = case["nx"] * case["ny"] * case["nz"], case["steps"]
            cells = cells if case["scene"] == "drop" else 0.73 * cells
        per = 168 if case.get("precision") else 304
        return {"bytes": float(per * cells * steps), "flops": 500.0 * cells * steps}
    n = case["n"]
    if kind == "throats":  # the boxes' cells, and the network of "predict"
        net, io, members = 24 * 256 + 3 * 65536 + 256 * N_OUT, n * (96 + 8 * 2 + 4 * (N_OUT - 1)), 5
        return {"bytes": float(io), "flops": 2.0 * members * net * n}
    net = case["n_in"] * case["hidden"] + (case["layers"] - 1) * case["hidden"] ** 2 + case["hidden"] * case["n_out"]
    members = case["members"]
    if kind == "predict":
        return {"bytes": float(4 * n * (case["n_in"] + 2 * case["n_out"]) + 4 * members * net),
                "flops": 2.0 * members * net * n}
    batches = case["epochs"] * (n // case["batch"])
    # a batch reads and writes the parameters and both Adam moments (the gradient is its own)
    return {"bytes": float(batches * members * (24 * net + 4 * case["batch"] * (case["n_in"] + case["n_out"]))),
            "flops": 6.0 * members * net * batches * case["batch"]}


# ------------------------------------------------------------ 64-bit values
E = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
              (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
              (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)])
WEIGHT = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
OPPOSITE = [0] + [k + 1 if k % 2 else k - 1 for k in range(1, 19)]


class _Reference:
    """Two-component Shan-Chen step in 64 bits on a mask, closed or periodic axes; a wall
    layer at the end of a closed axis stands for the neutral walls beyond the box."""

    def __init__(self, mask, rho, tau=(1.0, 1.0), G_ads=G_ADS, body_force=(0.0, 0.0, 0.0), periodic=(0, 0, 0)):
        pad = [v for p in periodic for v in (0, 0 if p else 1)]  # x, y, z: torch pads the last axis first
        self.inner = tuple(slice(0, m) for m in mask.shape)
        self.mask = torch.nn.functional.pad(mask, pad, value=SOLID)
        rho = torch.nn.functional.pad(rho, pad)
        self.tau, self.G_ads, self.g = tau, G_ads, body_force
        solid = (self.mask & SOLID) != 0
        self.wall = (solid, solid | ((self.mask & MEMBRANE) != 0))
        self.inlet, self.outlet = (self.mask & (SOLID | INLET)) == INLET, (self.mask & (SOLID | OUTLET)) == OUTLET
        grain = ((self.mask & (SOLID | ADHESIVE)) == (SOLID | ADHESIVE)).double()
        self.adhesion = self._gradient(grain)
        self.f = [[w * torch.where(self.wall[s], 0.0, rho[s]) for w in WEIGHT] for s in (0, 1)]

    @staticmethod
    def _at(a, e):  # the value at x - e
        dims = [(d, int(v)) for d, v in zip((2, 1, 0), e) if v]
        return torch.roll(a, [v for _, v in dims], [d for d, _ in dims]) if dims else a

    def _gradient(self, a):
        out = [torch.zeros_like(a) for _ in range(3)]
        for k in range(1, 19):
            v = WEIGHT[k] * self._at(a, -E[k])
            for d in range(3):
                if E[k][d]:
                    out[d] += int(E[k][d]) * v
        return out

    def density(self):
        return [sum(f[1:], f[0]) for f in self.f]

    def step(self, rho_in=(MINOR, MAJOR), rho_out=(MAJOR, MINOR)):
        rho = self.density()
        den = rho[0] / self.tau[0] + rho[1] / self.tau[1]
        den = torch.where(den == 0, 1.0, den)
        common = []
        for d in range(3):
            j = [sum(int(E[k][d]) * self.f[s][k] for k in range(1, 19) if E[k][d]) for s in (0, 1)]
            common.append((j[0] / self.tau[0] + j[1] / self.tau[1]) / den)
        force = [self._gradient(rho[1]), self._gradient(rho[0])]
        for s in (0, 1):
            u = [common[d] + self.tau[s] * (-G * force[s][d] - self.G_ads[s] * self.adhesion[d] + self.g[d])
                 for d in range(3)]
            uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
            post = []
            for k in range(19):
                eu = sum(int(E[k][d]) * u[d] for d in range(3) if E[k][d])
                eq = WEIGHT[k] * rho[s] * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * uu)
                v = self.f[s][k] + (eq - self.f[s][k]) / self.tau[s]
                v = torch.where(self.inlet, WEIGHT[k] * rho_in[s], v)
                post.append(torch.where(self.outlet, WEIGHT[k] * rho_out[s], v))
            self.f[s] = [torch.where(self.wall[s], 0.0, torch.where(self._at(self.wall[s], E[k]), post[OPPOSITE[k]],
                                                                    self._at(post[k], E[k]))) for k in range(19)]

    def measure(self, where=None):
        """Observables over the cells `where` (a box of slices of the mask)."""
        at = self.inner if where is None else where
        m, (a, b) = self.mask[at], [r[at] for r in self.density()]
        p = (a + b) / 3.0 + G * a * b / 3.0
        phi = (a - b) / (a + b)
        fluid = m == 0

        def mean(sel):
            return float(p[sel].mean()) if bool(sel.any()) else math.nan

        out = {"mass": [float(a.sum()), float(b.sum())], "p_w": mean(fluid & (phi > 0.9)),
               "p_nw": mean(fluid & (phi < -0.9)), "p_in": mean(self.inlet[at]), "p_out": mean(self.outlet[at]),
               "S_w": float((fluid & (a > b)).sum()) / float(fluid.sum())}
        return {**out, "p_c": out["p_nw"] - out["p_w"], "p_c_res": out["p_in"] - out["p_out"]}


def _rows(ref, boxes, probes, ladder, steps):
    """Rows of a pressure ladder for each box, and their entry pressures."""
    rows = np.zeros((len(boxes), len(ladder), len(ROW_KEYS)))
    for i, level in enumerate(ladder):
        for _ in range(steps):
            ref.step(rho_in=(MINOR, level))
        a, b = ref.density()
        for t, (box, probe) in enumerate(zip(boxes, probes)):
            m = ref.measure(box)
            rw, rn = float(a[probe]), float(b[probe])
            m["phi_probe"] = (rw - rn) / (rw + rn) if rw + rn else 0.0
            rows[t, i] = [m[k] for k in ROW_KEYS]
    p_ce = []
    for r in rows:
        hit = np.flatnonzero(r[:, ROW_KEYS.index("phi_probe")] < 0.0)
        p_ce.append(math.inf if len(hit) == 0 else float(np.nanmax(r[:hit[0] + 1, ROW_KEYS.index("p_c")], initial=-math.inf)))
    return rows, np.array(p_ce)


def _throat_box(s3):
    """Mask and probe (z, y, x) of one throat: the frame of its three centres."""
    c, r = s3[:, :3], s3[:, 3]

    def dot(a, b):  # term by term: rows of cells lie on the prism's walls, where a rounding decides
        return (a[..., 0] * b[..., 0] + a[..., 1] * b[..., 1]) + a[..., 2] * b[..., 2]

    a, n = c[1] - c[0], np.cross(c[1] - c[0], c[2] - c[0])
    e1, e3 = a / np.sqrt(dot(a, a)), n / np.sqrt(dot(n, n))
    local = np.stack([dot(c - c[0], e) for e in (e1, np.cross(e3, e1), e3)], -1)
    lo, h = np.floor(local[:, :2].min(0)), math.ceil(r.max())
    nx, ny = (np.ceil(local[:, :2].max(0)) - lo).astype(int) + 1
    shape, origin = (2 * h + 1, int(ny), int(nx)), (lo[0], lo[1], -float(h))
    grain = _grain(shape, np.c_[local, r], origin).numpy()
    mask = np.where(grain, SOLID | ADHESIVE, np.where(_outside_prism(shape, local, origin), SOLID, 0)).astype(np.uint8)
    mask[0][mask[0] == 0] = INLET
    mask[-1][mask[-1] == 0] = OUTLET
    k = shape[0] - 3
    p = np.stack(np.meshgrid(np.arange(nx) + origin[0], np.arange(ny) + origin[1], [k + origin[2]], indexing="ij"), -1)
    gap = np.min([np.linalg.norm(p - q, axis=-1) - v for q, v in zip(local, r)], axis=0)[..., 0].T
    gap[(mask[k] & SOLID) != 0] = -np.inf
    return mask, (k, *(int(v) for v in np.unravel_index(np.argmax(gap), gap.shape)))


def _forward(params, sizes, X):
    """Network output in 64 bits and the input of each layer."""
    at, h, kept = 0, X, []
    for i, (a, b) in enumerate(zip(sizes[:-1], sizes[1:])):
        W, c = params[at:at + a * b].view(b, a), params[at + a * b:at + a * b + b]
        at += a * b + b
        kept.append(h)
        h = h @ W.T + c
        if i < len(sizes) - 2:
            h = torch.relu(h)
    return h, kept


def _shuffled(seed, member, n, epochs):
    """Seeded Fisher-Yates orders of one member, an epoch after another."""
    mask = (1 << 64) - 1
    st = (seed * 0x9E3779B97F4A7C15 + member * 0xD1B54A32D192ED03 + 7) & mask
    for _ in range(epochs):
        o = list(range(n))
        for i in range(n - 1, 0, -1):
            st = (st + 0x9E3779B97F4A7C15) & mask
            z = ((st ^ (st >> 30)) * 0xBF58476D1CE4E5B9) & mask
            z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
            j = (z ^ (z >> 31)) % (i + 1)
            o[i], o[j] = o[j], o[i]
        yield o


def exact(case, seed):
    kind, dev = case["kind"], _device()
    if kind == "ladder":
        shape, s3 = (32, 32, 32), _throat32()
        mask = np.where(_grain(shape, s3).numpy(), SOLID | ADHESIVE,
                        np.where(_outside_prism(shape, s3[:, :3]), SOLID, 0)).astype(np.uint8)
        mask[0][mask[0] == 0] = INLET
        mask[-1][mask[-1] == 0] = OUTLET
        inlet = torch.zeros(shape, dtype=torch.bool, device=dev)
        inlet[0] = True
        ref = _Reference(torch.from_numpy(mask).to(dev), _two_phase(inlet, seed))
        rows, p_ce = _rows(ref, [ref.inner], [(29, 16, 16)], _ladder(case, 0.01), case["steps"])
        return {"rows": rows[0], "n_interface": None, "p_ce": float(p_ce[0]), "invaded_at": None,
                "density": torch.stack([r[ref.inner] for r in ref.density()]).cpu().numpy()}
    if kind == "box":
        if case["nx"] * case["ny"] * case["nz"] * case["steps"] > 1.5e9:
            return None
        mask, rho, par = _box_scene(case, seed)
        ref = _Reference(mask, rho, **par)
        for _ in range(case["steps"]):
            ref.step(rho_in=(MINOR, 2.1))
        m = ref.measure()
        return {"mass": np.array(m["mass"]), "measured": np.array([m[k] for k in MEASURED]), "counted": None,
                "density": torch.stack([r[ref.inner] for r in ref.density()]).cpu().numpy()}
    if kind == "batch":
        if case["n"] * case["incr"] * case["steps"] > 16 * 500:
            return None
        boxes = [_throat_box(s3) for s3 in _throats(seed, case["n"])]
        ny, nx = (max(m.shape[d] for m, _ in boxes) for d in (1, 2))
        whole, where, probes, z = [], [], [], 0
        for m, p in boxes:  # one above the other, a wall plane between
            t = np.full((m.shape[0] + 1, ny + 1, nx + 1), SOLID, dtype=np.uint8)
            t[:m.shape[0], :m.shape[1], :m.shape[2]] = m
            where.append((slice(z, z + m.shape[0]), slice(0, m.shape[1]), slice(0, m.shape[2])))
            probes.append((z + p[0], p[1], p[2]))
            whole.append(t)
            z += t.shape[0]
        mask = torch.from_numpy(np.concatenate(whole)).to(dev)
        inlet = mask == INLET
        hi, lo = torch.full(mask.shape, MAJOR, dtype=torch.float64, device=dev), MINOR
        rho = torch.stack([torch.where(inlet, lo, hi), torch.where(inlet, hi, lo)])
        rows, p_ce = _rows(_Reference(mask, rho), where, probes, _ladder(case, 0.06), case["steps"])
        return {"rows": rows, "n_interface": None, "p_ce": p_ce, "invaded_at": None, "n_fluid": None}
    if kind == "throats":
        return None  # the network is what the library trained
    params, sizes = _he_normal(case, seed)
    X, T = (torch.from_numpy(v).double().to(dev) for v in _samples(case, seed))
    params = [torch.from_numpy(p).double().to(dev) for p in params]
    if kind == "predict":
        Y = torch.stack([_forward(p, sizes, X)[0] for p in params])
        return {"mean": Y.mean(0).cpu().numpy(), "spread": Y.std(0, unbiased=True).cpu().numpy()}
    epochs, batch, n = case["epochs"], case["batch"], case["n"]
    loss = np.zeros((len(params), epochs))
    for m, p in enumerate(params):
        m1, m2, t = torch.zeros_like(p), torch.zeros_like(p), 0
        for ep, order in enumerate(_shuffled(3, m, n, epochs)):
            order = torch.tensor(order, device=dev)
            for b in range(0, n - batch + 1, batch):
                x, y = X[order[b:b + batch]], T[order[b:b + batch]]
                p = p.detach().requires_grad_(True)
                err = ((_forward(p, sizes, x)[0] - y) ** 2).mean()
                grad, = torch.autograd.grad(err, p)
                loss[m, ep] += float(err) / (n // batch)
                t += 1
                m1 = 0.9 * m1 + 0.1 * grad
                m2 = 0.999 * m2 + 0.001 * grad * grad
                p = p.detach() - 1e-3 * (m1 / (1 - 0.9 ** t)) / (torch.sqrt(m2 / (1 - 0.999 ** t)) + 1e-8)
        params[m] = p
    return {"loss": loss, "params": torch.stack(params).cpu().numpy()}
