"""Performance cases of the lattice Boltzmann framework: what a user's program has it do.

Each case is one pass through the public binding (paper_2009_04604_gb300.lbm): a
number of time steps and the read-out that follows them. The families:

  couette  circular Couette flow on D2Q9, the convergence studies' grids
  rigid    Jeffery's orbit on D2Q9: a body turning freely under the fluid's torque
  duct     the sphere in a duct (D3Q19, D3Q27), fields and drag after the steps
  monitor  the same duct, its drag read back after every step
  porous   a periodic box of spheres under a body force, with or without one
           sphere moving on a prescribed path
  batch    many ducts of uneven sizes advanced by one launch per step

exact() integrates the same equations in 64 bits with plain torch, from the
method's definition: dense arrays, one direction after another.
"""
import functools
import itertools
import math

import numpy as np
import torch

FLUID, SOLID, OPEN = 0, 1, 2


def listed():
    return [
        # The smallest calls: a validation grid in FP64, as in a convergence sweep. Latency and launches.
        dict(name="couette_64_f64", family="couette", L=64, dtype="f64", bc="elibb_f", tau=0.8, steps=100),
        # The sweep's larger grids in FP32 storage, an odd size, with the Bouzidi rule for comparison.
        dict(name="couette_301_f32_bfl", family="couette", L=301, dtype="f32", bc="bfl", tau=0.6, steps=100),
        # Fluid-structure coupling: the body's links are rebuilt after every step, on a small grid.
        dict(name="jeffery_128x98_f64", family="rigid", nx=128, ny=98, ra=8.0, rb=4.0, dtype="f64", tau=0.8,
             steps=100),
        # The reference-precision run on the downscaled benchmark, against which the others are judged.
        dict(name="duct_64x32x32_f64", family="duct", nx=64, ny=32, nz=32, lattice=19, dtype="f64", bc="elibb_f",
             collision="bgk", tau=0.7, steps=60, tuned=False),
        # The sphere-in-duct benchmark at full size: the framework's main path, autotuned, FP32 and FP16 storage.
        dict(name="duct_256x128x128_f32", family="duct", nx=256, ny=128, nz=128, lattice=19, dtype="f32",
             bc="elibb_f", collision="bgk", tau=0.7, steps=100, tuned=True),
        dict(name="duct_256x128x128_f16", family="duct", nx=256, ny=128, nz=128, lattice=19, dtype="f16",
             bc="elibb_f", collision="bgk", tau=0.7, steps=100, tuned=True),
        # Another lattice, collision and rule, an odd size, at the default launch.
        dict(name="duct_151x67x71_q27_trt", family="duct", nx=151, ny=67, nz=71, lattice=27, dtype="f32",
             bc="elibb_fq", collision="trt", tau=0.7, steps=60, tuned=False),
        # A controlled run: the drag is read back after every step (a synchronising call), default launch.
        dict(name="monitor_128x96x80_f32", family="monitor", nx=128, ny=96, nz=80, dtype="f32", bc="elibb_f",
             tau=0.7, steps=20),
        # The porous medium with a moving sphere (FP16, autotuned), where every fifth fluid node is a boundary node.
        dict(name="porous_256_moving_f16", family="porous", n=256, rmin=6.0, rmax=12.0, moving=True, dtype="f16",
             bc="elibb_f", tau=0.65, steps=40, tuned=True, geo=7),
        # The same medium without it, an odd size, the quadratic rule, FP32.
        dict(name="porous_150_f32_fq", family="porous", n=150, rmin=6.0, rmax=12.0, moving=False, dtype="f32",
             bc="elibb_fq", tau=0.65, steps=60, tuned=True, geo=8),
        # A parameter study: many small grids, and fewer larger ones, advanced by one launch per step.
        dict(name="batch_96_small_f32", family="batch", count=96, lo=16, hi=48, dtype="f32", tau=0.7, steps=64,
             geo=11),
        dict(name="batch_16_large_f16", family="batch", count=16, lo=48, hi=144, dtype="f16", tau=0.7, steps=40,
             geo=12),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    family = rng.choice(["couette", "rigid", "duct", "duct", "monitor", "porous", "porous", "batch"])
    if family == "couette":
        dtype = rng.choice(["f64", "f32"])
        return dict(family=family, L=log(48, 512 if dtype == "f32" else 160), dtype=dtype,
                    bc=rng.choice(["elibb_f", "elibb_fq", "bfl", "hwbb"]), tau=rng.choice([0.6, 0.8, 1.0]), steps=100)
    if family == "rigid":
        rb = rng.uniform(3.0, 5.0)
        ny = log(66, 130)
        return dict(family=family, nx=log(96, 192), ny=ny, ra=2.0 * rb, rb=rb, dtype=rng.choice(["f64", "f32"]),
                    tau=rng.choice([0.7, 0.8]), steps=100)
    if family == "duct":
        dtype = rng.choice(["f32", "f16", "bf16"])
        lattice = rng.choice([19, 19, 27])
        top = 1 if lattice == 19 else 0.7
        return dict(family=family, nx=log(48, int(256 * top)), ny=log(32, int(128 * top)), nz=log(32, int(128 * top)),
                    lattice=lattice, dtype=dtype, bc=rng.choice(["elibb_f", "elibb_fq"]),
                    collision=rng.choice(["bgk", "bgk", "trt"]), tau=rng.choice([0.6, 0.7, 0.9]), steps=60,
                    tuned=rng.random() < 0.5)
    if family == "monitor":
        return dict(family=family, nx=log(48, 200), ny=log(32, 110), nz=log(32, 110), dtype=rng.choice(["f32", "f16"]),
                    bc=rng.choice(["elibb_f", "elibb_fq"]), tau=rng.choice([0.6, 0.7]), steps=20)
    if family == "porous":
        n, rmax = log(96, 224), rng.uniform(8.0, 12.0)
        return dict(family=family, n=n, rmin=0.5 * rmax, rmax=rmax, moving=rng.random() < 0.5,
                    dtype=rng.choice(["f32", "f16"]), bc=rng.choice(["elibb_f", "elibb_fq"]), tau=0.65, steps=40,
                    tuned=rng.random() < 0.5, geo=rng.randrange(1, 100))
    lo = log(16, 40)
    hi = lo + rng.randint(16, 48)
    return dict(family=family, count=min(96, max(12, int(4e6 / ((lo + hi) / 2.0) ** 3))), lo=lo, hi=hi,
                dtype=rng.choice(["f32", "f16"]), tau=0.7, steps=40, geo=rng.randrange(1, 100))


# ---------------------------------------------------------------- inputs
# A workload: dims, base node kinds and their velocities (host arrays), shapes, and the initial state.

def _duct_base(dims, u_in):
    """Side walls at y, z = 0 and n-1, the inlet plane x = 0 moving with u_in, the open outlet plane x = nx-1."""
    nx, ny, nz = dims
    base = np.zeros((nz, ny, nx), np.uint8)
    base_u = np.zeros((nz, ny, nx, 3))
    base[:, :, 0] = SOLID
    base_u[1:-1, 1:-1, 0, 0] = u_in
    base[1:-1, 1:-1, nx - 1] = OPEN
    base[:, (0, ny - 1), :] = SOLID
    base[(0, nz - 1), :, :] = SOLID
    return base.reshape(-1), base_u.reshape(-1, 3)


def _duct(dims, seed, lattice, tau):
    r = np.random.default_rng(seed)
    u_in = 0.02 * r.uniform(0.7, 1.3)
    base, base_u = _duct_base(dims, u_in)
    R = min(dims[1], dims[2]) / 8.0
    c = (dims[0] / 4.0, dims[1] / 2.0, dims[2] / 2.0)
    return dict(lattice=lattice, dims=dims, tau=tau, force=(0.0, 0.0, 0.0), base=base, base_u=base_u,
                shapes=[dict(type="sphere", tag=1, c=c, r=(R, 0, 0))], rho=1.0,
                u=tuple(0.01 * r.uniform(-0.2, 1.0, 3) * (1.0, 0.2, 0.2)), body=None)


def _couette(case, seed):
    r = np.random.default_rng(seed)
    L = case["L"]
    om = 0.01 * r.uniform(0.8, 1.2) / (0.25 * L)
    c = (L / 2.0, L / 2.0, 0.0)
    shapes = [dict(type="sphere", tag=1, c=c, r=(0.25 * L, 0, 0), om=(0, 0, om), om1=(0, 0, om)),
              dict(type="sphere_out", tag=2, c=c, r=(0.45 * L, 0, 0))]
    N = L * L
    u = np.zeros((N, 3))
    u[:, :2] = 1e-3 * r.standard_normal((N, 2))
    return dict(lattice=9, dims=(L, L, 1), tau=case["tau"], force=(0.0, 0.0, 0.0), base=None, base_u=None,
                shapes=shapes, rho=1.0 + 1e-3 * r.standard_normal(N), u=u, body=None)


def _rigid(case, seed):
    r = np.random.default_rng(seed)
    nx, ny, ra, rb = case["nx"], case["ny"], case["ra"], case["rb"]
    U, H = 0.04 * r.uniform(0.8, 1.2), ny - 2
    y = np.arange(nx * ny) // nx
    base = np.zeros(nx * ny, np.uint8)
    base[(y == 0) | (y == ny - 1)] = SOLID
    base_u = np.zeros((nx * ny, 3))
    base_u[y == 0, 0] = -0.5 * U
    base_u[y == ny - 1, 0] = 0.5 * U
    u = np.zeros((nx * ny, 3))
    u[:, 0] = -0.5 * U + U * (y - 0.5) / H
    u[base == SOLID] = 0.0
    body = dict(type="ellipsoid", tag=1, c=(nx / 2.0 - 0.3, (ny - 1) / 2.0, 0.0), r=(rb, ra, 1.0),
                ang=float(r.uniform(0.0, 0.5)), om=(0.0, 0.0, 0.0))
    return dict(lattice=9, dims=(nx, ny, 1), tau=case["tau"], force=(0.0, 0.0, 0.0), base=base, base_u=base_u,
                shapes=[], rho=np.ones(nx * ny), u=u, body=body,
                inertia=math.pi * ra * rb * (ra * ra + rb * rb) / 4.0)


@functools.lru_cache(maxsize=8)
def _packing(n, rmin, rmax, moving, geo):
    """Non-overlapping spheres in a periodic box of side n, by random sequential addition, the largest first; with
    `moving`, the box around the moving sphere's path is kept free. Spheres across the edge come once per image."""
    r = np.random.default_rng(geo)
    L = float(n)
    want = 0.4 * L ** 3 / (math.pi / 3.0 * (rmax ** 4 - rmin ** 4) / (rmax - rmin))
    radii = np.sort(r.uniform(rmin, rmax, int(want) + 1))[::-1]
    R, A = _moving_sizes(n)
    half = np.array([A + R + 4.0, R + 4.0, R + 4.0])
    P, S = np.zeros((len(radii), 3)), np.zeros(len(radii))
    k = 0
    for rad in radii:
        p = r.uniform(0, L, (48, 3))
        d = p[:, None, :] - P[None, :k, :]
        d -= L * np.round(d / L)
        ok = ((d * d).sum(2) >= (rad + S[:k]) ** 2).all(1)
        if moving:
            gap = np.maximum(np.abs(p - L / 2) - half, 0.0)
            ok &= (gap * gap).sum(1) >= rad * rad
        hit = np.nonzero(ok)[0]
        if len(hit):
            P[k], S[k] = p[hit[0]], rad
            k += 1
    shapes = []
    for p, rad in zip(P[:k], S[:k]):
        for o in itertools.product((-L, 0.0, L), repeat=3):
            c = p + np.array(o)
            if np.all(c + rad >= -1.0) and np.all(c - rad <= L):
                shapes.append(dict(type="sphere", tag=0, c=tuple(float(v) for v in c), r=(float(rad), 0, 0)))
    return shapes


def _moving_sizes(n):
    """Radius and amplitude of the moving sphere's path: 10 and 20 on 384 nodes."""
    return max(4.0, 10.0 * n / 384.0), max(4.0, 20.0 * n / 384.0)


def _porous(case, seed):
    r = np.random.default_rng(seed)
    n = case["n"]
    shapes = _packing(n, case["rmin"], case["rmax"], case["moving"], case["geo"])
    w = dict(lattice=19, dims=(n, n, n), tau=case["tau"], force=(1e-6 * r.uniform(0.8, 1.2), 0.0, 0.0), base=None,
             base_u=None, shapes=shapes, rho=1.0, u=tuple(2e-3 * r.uniform(-1.0, 1.0, 3)), body=None)
    if case["moving"]:
        R, A = _moving_sizes(n)
        period = 5000
        om, ph = 2.0 * math.pi / period, r.uniform(0.0, 2.0 * math.pi)
        t = np.arange(period)
        traj = np.zeros((period, 9))
        traj[:, :3] = n / 2.0
        traj[:, 0] += A * np.sin(om * t + ph)
        traj[:, 3] = A * om * np.cos(om * t + ph)
        w.update(body=dict(type="sphere", tag=1, r=(R, 0, 0)), traj=traj)
    return w


def _batch(case, seed):
    """Ducts of uneven sizes, each with a sphere or an ellipsoid; sizes and obstacles by case["geo"], flow by seed."""
    g, r = np.random.default_rng(case["geo"]), np.random.default_rng(seed)
    out = []
    for _ in range(case["count"]):
        d = tuple(int(v) for v in g.integers(case["lo"], case["hi"] + 1, 3))
        top = (min(d) - 2) / 2.0 - 4.0
        axes = np.clip(g.uniform(case["lo"] / 8.0, case["lo"] / 2.5, 3), 1.0, max(1.0, top))
        c = tuple(float(v) for v in (np.array(d) - 1) / 2.0 + g.uniform(-0.5, 0.5, 3))
        shape = dict(type="sphere", tag=1, c=c, r=(float(axes[0]), 0, 0)) if g.random() < 0.5 else \
            dict(type="ellipsoid", tag=1, c=c, r=tuple(float(v) for v in axes))
        base, base_u = _duct_base(d, float(r.uniform(0.005, 0.03)))
        out.append(dict(lattice=19, dims=d, tau=case["tau"], force=(0.0, 0.0, 0.0), base=base, base_u=base_u,
                        shapes=[shape], rho=1.0, u=tuple(0.01 * r.uniform(0.0, 1.0, 3) * (1.0, 0.1, 0.1)), body=None))
    return out


def _workload(case, seed):
    family = case["family"]
    if family == "couette":
        return _couette(case, seed)
    if family == "rigid":
        return _rigid(case, seed)
    if family == "porous":
        return _porous(case, seed)
    return _duct((case["nx"], case["ny"], case["nz"]), seed, case.get("lattice", 19), case["tau"])


# ---------------------------------------------------------------- the framework
def _start(s, w):
    """The initial state: equilibrium at the workload's density and velocity."""
    if np.ndim(w["rho"]) == 0:
        s.init(w["rho"], w["u"])
        return
    from paper_2009_04604_gb300 import lbm
    c, wt = lbm.lattice_info(s.lattice)
    s.set_populations(_feq(torch.as_tensor(w["rho"]), torch.as_tensor(w["u"]).T, torch.as_tensor(c).double(),
                           torch.as_tensor(wt)).T.contiguous().numpy())


def _sim(w, case, stream=None):
    from paper_2009_04604_gb300 import lbm
    s = lbm.Simulation({9: lbm.D2Q9, 19: lbm.D3Q19, 27: lbm.D3Q27}[w["lattice"]], w["dims"], w["tau"], case["dtype"],
                       stream=stream)
    s.set_options(case.get("bc", "elibb_f"), 1.0, w["force"], 0)
    if case.get("collision", "bgk") == "trt":
        s.set_collision("trt")
    s.build_geometry(w["base"], w["base_u"], w["shapes"])
    if case.get("tuned"):
        s.init(1.0)
        s.autotune(6)
    if w["body"] is not None:
        if "traj" in w:
            s.set_moving_body(w["body"], w["traj"], 0)
        else:
            s.set_free_body(w["body"], w["inertia"], case["steps"])
    _start(s, w)
    return s


def prepare(case, seed):
    if case["family"] == "batch":
        from paper_2009_04604_gb300 import lbm
        stream = torch.cuda.Stream()
        ws = _batch(case, seed)
        sims = [_sim(w, case, stream) for w in ws]
        b = lbm.Batch(sims)
        b.autotune(4)
        for s, w in zip(sims, ws):
            _start(s, w)
        N = [s.N for s in sims]
        return dict(case=case, batch=b, sims=sims, at=np.concatenate([[0], np.cumsum(N)]),
                    rho=torch.zeros(sum(N), dtype=torch.float64, device="cuda"),
                    u=torch.zeros((sum(N), 3), dtype=torch.float64, device="cuda"))
    return dict(case=case, sim=_sim(_workload(case, seed), case))


def run(state):
    case = state["case"]
    if case["family"] == "batch":
        state["batch"].step(case["steps"])
        at = state["at"]
        for k, s in enumerate(state["sims"]):
            s.macros(state["rho"][at[k]:at[k + 1]], state["u"][at[k]:at[k + 1]])
        return dict(rho=state["rho"], u=state["u"])
    s = state["sim"]
    if case["family"] == "monitor":
        drag = []
        for _ in range(case["steps"]):
            s.step(1)
            drag.append(s.wall_force(1))
        rho, u = s.macros()
        return dict(rho=rho, u=u, drag=np.stack(drag))
    s.step(case["steps"])
    rho, u = s.macros()
    out = dict(rho=rho, u=u)
    if case["family"] == "duct" or case.get("moving"):
        out["force"] = s.wall_force(1)
    if case["family"] == "rigid":
        out["orbit"] = s.body_history()
    return out


def work(case):
    """Each step reads and writes every fluid node's populations once; the read-out reads them and writes the fields."""
    family, Q = case["family"], case.get("lattice", 19)
    if family == "couette":
        Q, N = 9, case["L"] ** 2
        fluid = math.pi * (0.45 ** 2 - 0.25 ** 2) * N
    elif family == "rigid":
        Q, N = 9, case["nx"] * case["ny"]
        fluid = case["nx"] * (case["ny"] - 2) - math.pi * case["ra"] * case["rb"]
    elif family == "porous":
        N = case["n"] ** 3
        fluid = 0.66 * N
    elif family == "batch":
        mean = 0.5 * (case["lo"] + case["hi"])
        N = case["count"] * mean ** 3
        fluid = case["count"] * (mean - 2) ** 3
    else:
        N = case["nx"] * case["ny"] * case["nz"]
        fluid = (case["nx"] - 2) * (case["ny"] - 2) * (case["nz"] - 2)
    size = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}[case["dtype"]]
    per_node = {9: 90, 19: 190, 27: 270}[Q]
    return dict(bytes=fluid * size * Q * (2 * case["steps"] + 1) + 32.0 * N, flops=fluid * per_node * case["steps"])


# ---------------------------------------------------------------- the same in 64 bits, by plain torch
def _velocities(Q):
    c = [(x, y, z) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)]
    if Q == 9:
        c = [v for v in c if v[2] == 0]
    if Q == 19:
        c = [v for v in c if abs(v[0]) + abs(v[1]) + abs(v[2]) < 3]
    w = {9: (4 / 9, 1 / 9, 1 / 36), 19: (1 / 3, 1 / 18, 1 / 36), 27: (8 / 27, 2 / 27, 1 / 54, 1 / 216)}[Q]
    return c, [w[sum(a * a for a in v)] for v in c]  # the opposite of direction i is Q - 1 - i


def _feq(rho, u, c, w):
    """Second-order equilibrium, [Q, N]; u: [3, N]."""
    usq = (u * u).sum(0)
    out = torch.empty((len(w),) + tuple(rho.shape), dtype=torch.float64, device=rho.device)
    for i in range(len(w)):
        cu = c[i][0] * u[0] + c[i][1] * u[1] + c[i][2] * u[2]
        out[i] = w[i] * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * usq)
    return out


def _feq_i(rho, ux, uy, uz, c, w):
    cu = c[0] * ux + c[1] * uy + c[2] * uz
    return w * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * (ux * ux + uy * uy + uz * uz))


class _Exact:
    """Dense FP64 integration of one workload, or of a list of workloads side by side in one node array."""

    def __init__(self, ws, case):
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.w0, self.case, self.bc = ws[0], case, case.get("bc", "elibb_f")
        self.Q = ws[0]["lattice"]
        self.D = 2 if self.Q == 9 else 3
        self.c, self.wt = _velocities(self.Q)
        self.om = 1.0 / ws[0]["tau"]
        self.trt = case.get("collision", "bgk") == "trt"
        self.om_m = 1.0 / (0.5 + (3.0 / 16.0) / (ws[0]["tau"] - 0.5)) if self.trt else self.om
        self.F = ws[0]["force"]
        parts = [self.geometry(w) for w in ws]
        off = np.concatenate([[0], np.cumsum([len(p["kind"]) for p in parts])])
        self.N = int(off[-1])
        self.kind = torch.cat([p["kind"] for p in parts])
        self.up = [torch.cat([p["up"][i] + int(o) for p, o in zip(parts, off)]) for i in range(self.Q)]
        self.links = [tuple(torch.cat([p["links"][i][j] + (int(o) if j == 0 else 0) for p, o in zip(parts, off)])
                            for j in range(5)) for i in range(self.Q)]
        self.find_open()
        rho = torch.cat([torch.as_tensor(np.broadcast_to(w["rho"], (int(np.prod(w["dims"])),)).copy()) for w in ws])
        u = torch.cat([torch.as_tensor(np.broadcast_to(w["u"], (int(np.prod(w["dims"])), 3)).copy()) for w in ws])
        self.f = _feq(rho.to(self.dev), u.to(self.dev).T, self.c, self.wt)
        self.force = None

    def find_open(self):
        self.open = []
        for i in range(self.Q):
            self.open.append(torch.nonzero((self.kind == FLUID) & (self.kind[self.up[i]] == OPEN)).reshape(-1))

    # ---- geometry: kinds, upstream indices, and per direction the links (node, q, u_w(t), u_w(t+1), tag)
    def scaled(self, s, X):
        """Offsets from the shape's centre, turned and scaled to its unit (or radius) sphere, and that radius squared."""
        d = [X[a] - s["c"][a] if a < self.D else torch.zeros_like(X[a]) for a in range(3)]
        if s["type"] != "ellipsoid":
            return d, s["r"][0] ** 2
        return self.turned(s, d), 1.0

    def turned(self, s, d):
        ca, sa = math.cos(s.get("ang", 0.0)), math.sin(s.get("ang", 0.0))
        b = [(ca * d[0] + sa * d[1]) / s["r"][0], (ca * d[1] - sa * d[0]) / s["r"][1]]
        return b + [d[2] / s["r"][2] if self.D == 3 else 0.0 * d[2]]

    def inside(self, s, X):
        d, r2 = self.scaled(s, X)
        v = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
        return v >= r2 if s["type"] == "sphere_out" else v <= r2

    def crossing(self, s, X, c):
        """The smallest t in (0, 1] at which X - t c enters the shape; 2 where there is none."""
        d, r2 = self.scaled(s, X)
        e = [float(c[a]) if a < self.D else 0.0 for a in range(3)]
        if s["type"] == "ellipsoid":
            e = [float(v) for v in self.turned(s, [torch.tensor(v, dtype=torch.float64) for v in e])]
        A = e[0] ** 2 + e[1] ** 2 + e[2] ** 2
        B = d[0] * e[0] + d[1] * e[1] + d[2] * e[2]
        C = d[0] * d[0] + d[1] * d[1] + d[2] * d[2] - r2
        disc = B * B - A * C
        sq = torch.sqrt(disc.clamp_min(0.0))
        if s["type"] == "sphere_out":
            t, ok = (B + sq) / A, C < 0
        else:
            t, ok = C / (B + sq), (C > 0) & (B > 0)
        return torch.where(ok & (disc >= 0) & (t > 0) & (t <= 1.0), t, torch.full_like(t, 2.0))

    def box(self, s, dims):
        """Slices (z, y, x) of the nodes that the shape can touch."""
        if s["type"] == "sphere_out":
            return (slice(0, dims[2]), slice(0, dims[1]), slice(0, dims[0]))
        out = []
        for a in (2, 1, 0):
            r = max(s["r"]) if s["type"] == "ellipsoid" else s["r"][0]
            lo, hi = (s["c"][a] - r - 2.0, s["c"][a] + r + 2.0) if a < self.D else (0, 0)
            out.append(slice(min(dims[a], max(0, math.floor(lo))), max(0, min(dims[a], math.ceil(hi) + 1))))
        return tuple(out)

    def coords(self, b):
        z, y, x = (torch.arange(s.start, s.stop, dtype=torch.float64, device=self.dev) for s in b)
        return torch.broadcast_tensors(x[None, None, :], y[None, :, None], z[:, None, None])

    def geometry(self, w):
        nx, ny, nz = dims = w["dims"]
        N = nx * ny * nz
        base = torch.zeros((nz, ny, nx), dtype=torch.uint8, device=self.dev) if w["base"] is None else \
            torch.as_tensor(w["base"]).to(self.dev).reshape(nz, ny, nx)
        kind = base.clone()
        for s in w["shapes"]:
            b = self.box(s, dims)
            k = kind[b]
            kind[b] = torch.where((k == FLUID) & self.inside(s, self.coords(b)), torch.full_like(k, SOLID), k)
        z, y, x = torch.meshgrid(*(torch.arange(n, device=self.dev) for n in (nz, ny, nx)), indexing="ij")
        up = [(((z - c[2]) % nz * ny + (y - c[1]) % ny) * nx + (x - c[0]) % nx).reshape(-1) for c in self.c]
        kf, bf = kind.reshape(-1), base.reshape(-1)
        bu = None if w["base_u"] is None else torch.as_tensor(w["base_u"]).to(self.dev)
        links = []
        for i, c in enumerate(self.c):
            best = torch.full((nz, ny, nx), 2.0, dtype=torch.float64, device=self.dev)
            own = torch.zeros((nz, ny, nx), dtype=torch.int32, device=self.dev)
            if any(c):
                for k, s in enumerate(w["shapes"]):
                    b = self.box(s, dims)
                    t = self.crossing(s, self.coords(b), c)
                    own[b] = torch.where(t < best[b], torch.full_like(own[b], k), own[b])
                    best[b] = torch.minimum(t, best[b])
            n = torch.nonzero((kf == FLUID) & (kf[up[i]] == SOLID)).reshape(-1)
            wall = bf[up[i][n]] != FLUID
            q = torch.where(wall, 0.5, best.reshape(-1)[n].clamp_max(1.0))
            own = own.reshape(-1)[n]
            uw = torch.zeros((len(n), 3), dtype=torch.float64, device=self.dev)
            tag = torch.zeros(len(n), dtype=torch.int32, device=self.dev)
            if bu is not None:
                uw[wall] = bu[up[i][n[wall]]]
            for k, s in enumerate(w["shapes"]):
                if s["tag"] or s.get("om"):
                    m = ~wall & (own == k)
                    tag[m] = s["tag"]
                    if s.get("om"):
                        uw[m] = self.rigid(s, n[m], q[m], c, dims, (0.0, 0.0, 0.0), s["om"])
            links.append((n, q, uw, uw, tag))
        return dict(kind=kf, up=up, links=links)

    def rigid(self, s, n, q, c, dims, v, om):
        """v + om x (x_W - c) at the wall points of links (om along z)."""
        x = n % dims[0] - q * c[0] - s["c"][0]
        y = n // dims[0] % dims[1] - q * c[1] - s["c"][1]
        u = torch.zeros((len(n), 3), dtype=torch.float64, device=self.dev)
        u[:, 0] = v[0] - om[2] * y
        u[:, 1] = v[1] + om[2] * x
        u[:, 2] = v[2]
        return u

    # ---- one step
    def macros(self):
        rho = self.f.sum(0)
        u = torch.zeros((3, self.N), dtype=torch.float64, device=self.dev)
        for i, c in enumerate(self.c):
            for a in range(3):
                if c[a]:
                    u[a] += c[a] * self.f[i]
        for a in range(3):
            u[a] = (u[a] + 0.5 * self.F[a]) / rho
        return rho, u

    def step(self, body=()):
        """body: per direction the moving body's links, in the layout of self.links, or nothing."""
        rho, u = self.macros()
        usq, uF = (u * u).sum(0), u[0] * self.F[0] + u[1] * self.F[1] + u[2] * self.F[2]
        Q, c, wt, f = self.Q, self.c, self.wt, self.f
        post = torch.empty_like(f)
        for i in range(Q // 2 + 1):
            j = Q - 1 - i
            cu = c[i][0] * u[0] + c[i][1] * u[1] + c[i][2] * u[2]
            cF = sum(c[i][a] * self.F[a] for a in range(3))
            ep = wt[i] * rho * (1.0 + 4.5 * cu * cu - 1.5 * usq)
            em = 3.0 * wt[i] * rho * cu
            dp = self.om * (ep - 0.5 * (f[i] + f[j])) + (1 - 0.5 * self.om) * wt[i] * (9.0 * cu * cF - 3.0 * uF)
            dm = self.om_m * (em - 0.5 * (f[i] - f[j])) + (1 - 0.5 * self.om_m) * 3.0 * wt[i] * cF
            post[i] = f[i] + dp + dm
            post[j] = f[j] + dp - dm
        new = torch.empty_like(f)
        self.exchange = []
        for i in range(Q):
            new[i] = post[i][self.up[i]]
            n = self.open[i]
            if len(n):
                un, j = u[:, n], Q - 1 - i
                new[i][n] = _feq_i(torch.ones_like(rho[n]), *un, c[i], wt[i]) + f[j][n] - \
                    _feq_i(rho[n], *un, c[j], wt[j])
            for links in ([self.links[i]] + ([body[i]] if body else [])):
                if len(links[0]):
                    val = self.wall(i, links, rho, u, post)
                    new[i][links[0]] = val
                    self.exchange.append((i, links, post[Q - 1 - i][links[0]], val))
        self.f = new

    def wall(self, i, links, rho, u, post):
        n, q, uw, uw1, _ = links
        j, c, w, r = self.Q - 1 - i, self.c[i], self.wt[i], rho[n]
        me = 6.0 * w * r * (c[0] * uw[:, 0] + c[1] * uw[:, 1] + c[2] * uw[:, 2])
        g, h = post[j][n] + me, post[i][n]
        if self.bc == "hwbb":
            return g
        if self.bc == "bfl":
            ff = self.up[j][n]  # the second node along the link
            near = torch.where(self.kind[ff] == FLUID, 2 * q * post[j][n] + me + (1 - 2 * q) * post[j][ff], g)
            return torch.where(q < 0.5, near, ((2 * q - 1) * h + g) / (2 * q))
        fneq = self.f[j][n] - _feq_i(r, *u[:, n], self.c[j], w)
        f0 = _feq_i(r, *uw1.T, c, w) + fneq
        f1 = _feq_i(r, *uw.T, c, w) + (1 - self.om) * fneq
        near, far = ((1 - 2 * q) * f0 + q * g) / (1 - q).clamp_min(1e-300), ((1 - q) * g + (2 * q - 1) * f1) / q
        if self.bc == "elibb_fq":
            near = torch.where(q >= 0.01, (1 - 2 * q) * f0 + g + (2 * q - 1) * f1, near)
            far = ((1 - q) * g + 2 * (2 * q - 1) * f1 + (2 * q - 1) * (q - 1) * h) / (2 * q * q)
        return torch.where(q < 0.5, near, far)

    def wall_force(self, tag, centre=None):
        """Momentum exchange of the last step over the links with this tag, and with a centre its torque about z."""
        F, T = torch.zeros(3, dtype=torch.float64, device=self.dev), 0.0
        for i, (n, q, uw, _, tg), out, back in self.exchange:
            m = tg == tag
            ci = torch.tensor(self.c[i], dtype=torch.float64, device=self.dev)
            one = (-ci - uw[m]) * out[m, None] - (ci - uw[m]) * back[m, None]
            F += one.sum(0)
            if centre is not None:
                dims = self.w0["dims"]
                x = n[m] % dims[0] - q[m] * self.c[i][0] - centre[0]
                y = n[m] // dims[0] % dims[1] - q[m] * self.c[i][1] - centre[1]
                T = T + (x * one[:, 1] - y * one[:, 0]).sum()
        return F, T

    # ---- a moving body: its nodes and links at a pose, and the refill of nodes it leaves
    def place(self, s, v, v1, om, refill):
        dims = self.w0["dims"]
        b = self.box(s, dims)
        kind = self.static.clone().reshape(dims[2], dims[1], dims[0])
        kind[b] = torch.where(self.inside(s, self.coords(b)), torch.full_like(kind[b], SOLID), kind[b])
        kind = kind.reshape(-1)
        if refill:
            n = torch.nonzero((kind == FLUID) & (self.kind != FLUID)).reshape(-1)
            if len(n):
                zero = torch.zeros_like(n, dtype=torch.float64)
                u = self.rigid(s, n, zero, (0, 0, 0), dims, v, om)
                self.f[:, n] = _feq(torch.ones_like(zero), u.T, self.c, self.wt)
        self.kind = kind
        body = []
        z, y, x = (torch.arange(t.start, t.stop, device=self.dev) for t in b)
        near = ((z[:, None, None] * dims[1] + y[None, :, None]) * dims[0] + x[None, None, :]).reshape(-1)
        for i, c in enumerate(self.c):
            m = self.up[i][near]
            n = near[(kind[near] == FLUID) & (kind[m] == SOLID) & (self.static[m] == FLUID)]
            X = [(n % dims[0]).double(), (n // dims[0] % dims[1]).double(), (n // (dims[0] * dims[1])).double()]
            q = self.crossing(s, X, c).clamp_max(1.0)
            body.append((n, q, self.rigid(s, n, q, c, dims, v, om), self.rigid(s, n, q, c, dims, v1, om),
                         torch.full_like(n, s["tag"])))
        return body


def exact(case, seed):
    if case["family"] == "batch":
        e = _Exact(_batch(case, seed), case)
        for _ in range(case["steps"]):
            e.step()
        return _fields(e)
    w = _workload(case, seed)
    e = _Exact([w], case)
    drag, orbit, body = [], [], ()
    moving = w["body"] is not None
    if moving:
        e.static, s = e.kind, dict(w["body"])
        om, zero = (0.0, 0.0, 0.0), (0.0, 0.0, 0.0)

        def place(k, refill):
            if "traj" not in w:
                return e.place(s, zero, zero, om, refill)
            p, p1 = w["traj"][k % len(w["traj"])], w["traj"][(k + 1) % len(w["traj"])]
            return e.place(dict(s, c=tuple(float(v) for v in p[:3])), p[3:6], p1[3:6], zero, refill)

        body = place(0, False)
    for k in range(case["steps"]):
        e.step(body)
        if case["family"] == "monitor" or k == case["steps"] - 1:
            drag.append(e.wall_force(1)[0].cpu().numpy())
        if case["family"] == "rigid":
            T = float(e.wall_force(1, s["c"])[1])
            om = (0.0, 0.0, om[2] + T / w["inertia"])
            s["ang"] += om[2]
            orbit.append((s["ang"], om[2], T))
        if moving:
            body = place(k + 1, True)
    out = _fields(e)
    if case["family"] == "monitor":
        out["drag"] = np.stack(drag)
    elif case["family"] == "duct" or case.get("moving"):
        out["force"] = drag[-1]
    if case["family"] == "rigid":
        out["orbit"] = np.array(orbit)
    return out


def _fields(e):
    rho, u = e.macros()
    fluid = e.kind == FLUID
    return dict(rho=torch.where(fluid, rho, torch.zeros_like(rho)),
                u=torch.where(fluid, u, torch.zeros_like(u)).T.contiguous())
