"""The work whose speed is measured: what a program does through the public
entry points of ``paper_2003_07968_gb300.capi`` over the range of lattices
the library is used for.

A pass advances lattices by a number of time steps and reads the fields back
(a solve also initialises them first), for
  - one lattice, from the 64 x 64 band of a first experiment, where launches
    and latency count, to the 8192 x 8192 droplet, where memory does;
  - a batch of lattices of one handle, uneven ones and a parameter sweep;
  - requests to a server.
Storage (FP32, FP32 deviations, FP16 deviations), collision (BGK, MRT) and
equation of state (Carnahan-Starling, van der Waals) vary as the paper's
experiments and the batched and served workloads have them.
"""
from __future__ import annotations

import math
import random
import time

import numpy as np
import torch

from paper_2003_07968_gb300 import capi as P

STORAGE = {"f32": P.LBM_STORE_F32, "f32dev": P.LBM_STORE_F32_DEV, "f16dev": P.LBM_STORE_F16_DEV}
# coexistence densities (vapour, liquid) that the initial fields start from
COEX = {"cs": {0.6: (0.023623, 3.114014), 0.65: (0.04283, 2.931034), 0.7: (0.07125, 2.745479),
               0.75: (0.111359, 2.554674), 0.8: (0.166533, 2.355003), 0.85: (0.24211, 2.14086),
               0.9: (0.348205, 1.901846)},
        "vdw": {0.85: (0.31973, 1.80714), 0.9: (0.42574, 1.65727)}}
EOS = {"cs": (3.852462257, 0.1304438842, 2.785855166), "vdw": (3.0, 1.0 / 3.0, 8.0 / 3.0)}

SINGLE = dict(kind="single", nx=256, ny=256, T=0.8, tau=1.0, sigma=1.0, storage="f32dev",
              collision="bgk", eos="cs", shape="droplet", solve=False, velocity=False, steps=100)


def listed():
    def one(name, **kw):
        return dict(SINGLE, name=name, **kw)

    return [
        # a whole small solve: the flat band on 64 x 64 from its field to its
        # result, 2000 steps
        one("band64_solve", nx=64, ny=64, shape="band", storage="f32", solve=True, velocity=True,
            steps=2000),
        # the static droplet of the Young-Laplace test on its way to the steady
        # state: densities and velocities looked at every 500 steps
        one("droplet256", T=0.7, velocity=True, steps=500),
        # the oscillating ellipse with MRT: the density field every 100 steps
        one("mrt200", nx=200, ny=200, T=0.6, tau=0.65, collision="mrt", shape="ellipse"),
        # the surface-tension sweep: six droplets that differ in sigma, one handle
        dict(name="sweep6x200", kind="batch", count=6, lo=200, hi=200, sides_seed=0, T=0.8, tau=0.8,
             sweep=True, storage="f32dev", steps=500),
        # an ordinary lattice of odd sizes, another equation of state
        one("ragged777", nx=777, ny=611, T=0.85, tau=0.9, sigma=0.5, eos="vdw", velocity=True,
            steps=200),
        # the large oscillating ellipse: its extremity sampled every 500 steps
        one("ellipse1024", nx=1024, ny=1024, T=0.6, tau=0.8, shape="ellipse", steps=500),
        # half the bytes: FP16 deviations on a lattice larger than L2
        one("f16_4096", nx=4096, ny=4096, storage="f16dev", steps=100),
        # a short job end to end: host fields with a velocity in, 20 steps,
        # every field and the mass out
        one("job4096", nx=4096, ny=4096, T=0.7, solve=True, velocity=True, steps=20),
        # the largest lattice, many steps between two looks at the density
        one("droplet8192", nx=8192, ny=8192, steps=100),
        # the uneven batch of droplets, sides 64 to 512, in FP32 and FP16 storage
        dict(name="batch512", kind="batch", count=512, lo=64, hi=512, sides_seed=4, T=0.0, tau=1.0,
             sweep=False, storage="f32dev", steps=100),
        dict(name="batch128_f16", kind="batch", count=128, lo=64, hi=512, sides_seed=4, T=0.0,
             tau=1.0, sweep=False, storage="f16dev", steps=100),
        # a server with a burst of requests of many sizes and lengths
        dict(name="served40", kind="served", count=40, lo=128, hi=1024, sides_seed=5, T=0.0,
             tau=1.0, min_steps=10, max_steps=500, storage="f32dev"),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["single", "single", "single", "single", "batch", "served"])
    storage = rng.choice(["f32dev", "f32dev", "f32", "f16dev"])
    if kind == "single":
        eos = rng.choice(["cs", "cs", "cs", "vdw"])
        nx, ny = log_int(33, 5000), log_int(33, 5000)
        T = rng.choice(sorted(COEX[eos]))
        return dict(SINGLE, nx=nx, ny=ny, T=T, eos=eos, tau=rng.choice([0.8, 0.9, 1.0, 1.1]),
                    sigma=rng.choice([0.5, 1.0, 2.0]) if T >= 0.75 else 1.0,
                    storage=storage, collision=rng.choice(["bgk", "bgk", "mrt"]),
                    shape=rng.choice(["droplet", "ellipse", "band"]), solve=rng.random() < 0.3,
                    velocity=rng.random() < 0.5,
                    steps=min(log_int(8, 1500), max(8, int(2.5e9 / (nx * ny)))))
    if kind == "batch":
        hi = log_int(80, 512)
        lo = rng.randint(40, hi)
        count = log_int(2, 200)
        return dict(kind="batch", count=count, lo=lo, hi=hi, sides_seed=rng.randrange(1000),
                    T=0.0, tau=rng.choice([0.8, 1.0]), sweep=False, storage=storage,
                    steps=min(log_int(10, 400), max(10, int(2.5e9 / (count * hi * hi)))))
    hi = log_int(200, 1024)
    return dict(kind="served", count=rng.randint(3, 40), lo=rng.randint(64, hi), hi=hi,
                sides_seed=rng.randrange(1000), T=0.0, tau=1.0, min_steps=5,
                max_steps=log_int(30, 500), storage=storage)


def lattices(case):
    """The lattices of a case: one dict of sizes and parameters each."""
    if case["kind"] == "single":
        return [dict(case)]
    r = random.Random(case["sides_seed"])
    out = []
    for k in range(case["count"]):
        side = r.randint(case["lo"], case["hi"])
        T = case["T"] or r.choice([0.6, 0.65, 0.7, 0.75, 0.8, 0.85, 0.9])
        shape = "droplet" if case["kind"] == "batch" else r.choice(["droplet", "band"])
        steps = case["steps"] if case["kind"] == "batch" else r.randint(case["min_steps"], case["max_steps"])
        out.append(dict(SINGLE, nx=side, ny=side, T=T, tau=case["tau"], shape=shape, steps=steps,
                        sigma=4.0 / 2 ** k if case.get("sweep") else 1.0, storage=case["storage"]))
    return out


def field(lat, rng, velocity=False):
    """Initial density (and velocity) of a lattice, FP64 on the GPU: liquid in
    vapour with a tanh interface of width 5; where it sits and how large it
    is comes from ``rng``."""
    nx, ny = lat["nx"], lat["ny"]
    rg, rl = COEX[lat["eos"]][lat["T"]]
    x = torch.arange(nx, dtype=torch.float64, device="cuda")[None, :]
    y = torch.arange(ny, dtype=torch.float64, device="cuda")[:, None]
    side = min(nx, ny)
    if lat["shape"] == "band":
        mid, half = ny * rng.uniform(0.4, 0.6), ny * rng.uniform(0.2, 0.28)
        prof = 0.5 * (torch.tanh(0.4 * (y - mid + half)) - torch.tanh(0.4 * (y - mid - half)))
        gen = torch.Generator(device="cuda").manual_seed(rng.randrange(1 << 30))
        noise = torch.rand((ny, nx), dtype=torch.float64, device="cuda", generator=gen)
        rho = rg + (rl - rg) * prof + min(1e-3, 0.02 * rg) * (2.0 * noise - 1.0)
    else:
        stretch = 1.2 if lat["shape"] == "ellipse" else 1.0
        cx, cy = nx * rng.uniform(0.4, 0.6), ny * rng.uniform(0.4, 0.6)
        R = side * rng.uniform(0.2, 0.3)
        r = torch.sqrt(((x - cx) / stretch) ** 2 + ((y - cy) * stretch) ** 2)
        rho = 0.5 * (rl + rg) - 0.5 * (rl - rg) * torch.tanh(0.4 * (r - R))
    if not velocity:
        return rho, None, None
    a, ph = 2.0 * math.pi, rng.uniform(0.0, 6.0)
    ux = (1e-3 * torch.sin(a * y / ny + ph)).expand(ny, nx)
    uy = (1e-3 * torch.sin(a * x / nx - ph)).expand(ny, nx)
    return rho, ux, uy


def pinned(t):
    """A host copy of a device field in page-locked memory, as numpy."""
    h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    h.copy_(t)
    return h.numpy()


def host_fields(case, seed):
    """Per lattice (rho, ux, uy) on the host, from the seed alone."""
    rng = random.Random(seed)
    out = []
    for lat in lattices(case):
        f = field(lat, rng, velocity=case["kind"] == "single" and case["solve"])
        out.append(tuple(None if v is None else pinned(v.contiguous()) for v in f))
    return out


def descriptor(lat):
    kw = {}
    if lat["collision"] == "mrt":
        kw = dict(collision=P.LBM_COLL_MRT, mrt_rates=[1.0] * 7 + [1.0 / lat["tau"]] * 2)
    if lat["eos"] == "vdw":
        kw["eos_kind"] = P.LBM_EOS_KIND_VDW
    return P.lbm_desc_default(lat["nx"], lat["ny"], T=lat["T"], tau=lat["tau"], sigma=lat["sigma"],
                              storage=STORAGE[lat["storage"]], **kw)


def out_array(shape):
    return torch.empty(shape, dtype=torch.float64, pin_memory=True).numpy()


def prepare(case, seed):
    lats = lattices(case)
    fields = host_fields(case, seed)
    descs = [descriptor(lat) for lat in lats]
    s = {"case": case, "fields": fields, "descs": descs, "lats": lats}
    if case["kind"] == "served":
        s["server"] = P.lbm_server_create(P.lbm_server_opts_default(
            arena_bytes=3 << 30, max_request_sites=1024 * 1024, max_width=1024,
            storage=STORAGE[case["storage"]], with_velocity=0))
        return s
    s["handle"] = P.lbm_create(descs)
    for k, (rho, ux, uy) in enumerate(fields):
        P.lbm_init(s["handle"], k, rho, ux, uy)
    # the program's own result arrays: a batch's fields one after another
    if case["kind"] == "single":
        keys = ("rho", "ux", "uy") if case["velocity"] else ("rho",)
        s["out"] = {k: out_array((case["ny"], case["nx"])) for k in keys}
    else:
        s["rho"] = out_array(sum(lat["nx"] * lat["ny"] for lat in lats))
        s["out"], at = [], 0
        for lat in lats:
            n = lat["nx"] * lat["ny"]
            s["out"].append({"rho": s["rho"][at:at + n].reshape(lat["ny"], lat["nx"])})
            at += n
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "served":
        tickets = [P.lbm_submit(s["server"], d, f[0], lat["steps"])
                   for d, f, lat in zip(s["descs"], s["fields"], s["lats"])]
        got = [None] * len(tickets)
        left = list(range(len(tickets)))
        while left:
            for k in left:
                got[k] = P.lbm_poll(s["server"], tickets[k], u=False)
            left = [k for k in left if got[k] is None]
            if left:
                time.sleep(0.0002)
        return [g["rho"] for g in got]
    h = s["handle"]
    if case["kind"] == "batch":
        P.lbm_step(h, case["steps"])
        for k, out in enumerate(s["out"]):
            P.lbm_moments(h, k, u=False, mass=False, out=out)
        return s["rho"]
    if case["solve"]:
        P.lbm_init(h, 0, *s["fields"][0])
    P.lbm_step(h, case["steps"])
    return P.lbm_moments(h, 0, u=case["velocity"], mass=case["velocity"], out=s["out"])


def work(case):
    """The state (nine populations a site) in and out once a pass, the host
    fields in and out; 200 floating-point operations a site and step (density
    8, psi 17, its moments and the force 50, velocity, equilibria, source and
    relaxation 125)."""
    lats = lattices(case)
    sites = sum(lat["nx"] * lat["ny"] for lat in lats)
    updates = sum(lat["nx"] * lat["ny"] * lat["steps"] for lat in lats)
    es = 2 if case["storage"] == "f16dev" else 4
    fields_in = 0 if case["kind"] == "batch" else 1 if case["kind"] == "served" else 3 * case["solve"]
    fields_out = 3 if case["kind"] == "single" and case["velocity"] else 1
    state = 0 if case["kind"] == "served" or (case["kind"] == "single" and case["solve"]) else 18 * es
    return {"bytes": float(sites * (state + 8 * (fields_in + fields_out))), "flops": 200.0 * updates}


# ---- what a pass returns, in plain 64-bit torch ------------------------------
CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
W = (4 / 9, 1 / 9, 1 / 9, 1 / 9, 1 / 9, 1 / 36, 1 / 36, 1 / 36, 1 / 36)


class Solver:
    """The method's time step for lattices of one tau and collision, their
    sites one after another in flat arrays."""

    def __init__(self, lats, fields):
        self.tau = lats[0]["tau"]
        self.mrt = lats[0]["collision"] == "mrt"
        self.vdw = lats[0]["eos"] == "vdw"
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        idx, at = [], 0
        for lat in lats:
            nx, ny = lat["nx"], lat["ny"]
            x = torch.arange(nx, dtype=torch.int32, device=dev)[None, :]
            y = torch.arange(ny, dtype=torch.int32, device=dev)[:, None]
            idx.append([(at + ((y + CY[i]) % ny) * nx + (x + CX[i]) % nx).reshape(-1) for i in range(9)])
            at += nx * ny
        self.to = [torch.cat([v[i] for v in idx]) for i in range(9)]  # site x + c_i
        self.opp = (0, 3, 4, 1, 2, 7, 8, 5, 6)

        def flat(k):
            return torch.cat([torch.from_numpy(np.ascontiguousarray(f[k])).to(dev).reshape(-1) for f in fields])

        def per_site(key):
            if len({lat[key] for lat in lats}) == 1:
                return lats[0][key]
            return torch.cat([torch.full((lat["nx"] * lat["ny"],), lat[key], dtype=torch.float64, device=dev)
                              for lat in lats])

        self.T, self.sigma = per_site("T"), per_site("sigma")
        rho = flat(0)
        zero = torch.zeros_like(rho)
        ux, uy = (flat(1), flat(2)) if fields[0][1] is not None else (zero, zero)
        self.f = [self.equilibrium(i, rho, ux, uy) for i in range(9)]

    def equilibrium(self, i, rho, ux, uy):
        cu = CX[i] * ux + CY[i] * uy
        return W[i] * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * (ux * ux + uy * uy))

    def psi(self, rho):
        a, b, c = EOS["vdw" if self.vdw else "cs"]
        eta = b * rho
        q = 1.0 / (1.0 - eta) if self.vdw else (1.0 + eta + eta ** 2 - eta ** 3) / (1.0 - eta) ** 3
        p = 0.01 * (c * rho * self.T * q - a * rho * rho)
        return torch.sqrt(rho / 3.0 - p)  # G = -1

    def moments(self):
        """rho, the force-shifted velocity and the force."""
        rho = sum(self.f)
        s = self.psi(rho)
        m1x, m1y, xx, yy, xy = (torch.zeros_like(s) for _ in range(5))
        for i in range(9):
            p = s if i == 0 else s[self.to[i]]
            if CX[i]:
                m1x.add_(p, alpha=W[i] * CX[i])
            if CY[i]:
                m1y.add_(p, alpha=W[i] * CY[i])
            xx.add_(p, alpha=W[i] * (CX[i] ** 2 - 1 / 3))
            yy.add_(p, alpha=W[i] * (CY[i] ** 2 - 1 / 3))
            if CX[i] * CY[i]:
                xy.add_(p, alpha=W[i] * CX[i] * CY[i])
        G, eps = -1.0, 1.73
        k1, k2 = 13.5 * eps * G, 9.0 * (self.sigma - 1.0) * G
        lead = -6.0 * G * s + k2 * (xx + yy)
        Fx = lead * m1x + (k1 - k2) * (m1x * xx + m1y * xy)
        Fy = lead * m1y + (k1 - k2) * (m1x * xy + m1y * yy)
        jx = self.f[1] - self.f[3] + self.f[5] - self.f[6] - self.f[7] + self.f[8]
        jy = self.f[2] - self.f[4] + self.f[5] + self.f[6] - self.f[7] - self.f[8]
        return rho, (jx + 0.5 * Fx) / rho, (jy + 0.5 * Fy) / rho, Fx, Fy

    def step(self):
        rho, ux, uy, Fx, Fy = self.moments()
        Fu = Fx * ux + Fy * uy
        om = 1.0 / self.tau
        dn, src = [], []
        for i in range(9):
            cu, cF = CX[i] * ux + CY[i] * uy, CX[i] * Fx + CY[i] * Fy
            dn.append(self.f[i] - self.equilibrium(i, rho, ux, uy))
            src.append(W[i] * (3.0 * cF + 9.0 * cF * cu - 3.0 * Fu))
        if self.mrt:
            dn, src = torch.stack(dn), torch.stack(src)
            M = self.matrix().to(dn.device)
            rates = torch.tensor([1.0] * 7 + [om] * 2, dtype=torch.float64, device=dn.device)
            inv = torch.linalg.inv(M)
            dn = inv @ (rates[:, None] * (M @ dn))
            src = inv @ ((1.0 - 0.5 * rates)[:, None] * (M @ src))
            post = [self.f[i] - dn[i] + src[i] for i in range(9)]
        else:
            post = [self.f[i] - om * dn[i] + (1.0 - 0.5 * om) * src[i] for i in range(9)]
        self.f = [post[0]] + [post[i][self.to[self.opp[i]]] for i in range(1, 9)]

    @staticmethod
    def matrix():
        """The Gram-Schmidt moments 1, e, e^2, j_x, q_x, j_y, q_y, p_xx, p_xy."""
        c = torch.tensor([CX, CY], dtype=torch.float64)
        x, y = c[0], c[1]
        r = x * x + y * y
        return torch.stack([torch.ones(9, dtype=torch.float64), 3 * r - 4, 4.5 * r * r - 10.5 * r + 4,
                            x, (3 * r - 5) * x, y, (3 * r - 5) * y, x * x - y * y, x * y])


def exact(case, seed):
    lats, fields = lattices(case), host_fields(case, seed)
    if case["kind"] == "served":
        out = []
        for lat, f in zip(lats, fields):
            one = Solver([lat], [f])
            for _ in range(lat["steps"]):
                one.step()
            out.append(one.moments()[0].reshape(lat["ny"], lat["nx"]))
        return out
    s = Solver(lats, fields)
    for _ in range(case["steps"]):
        s.step()
    rho, ux, uy = s.moments()[:3]
    if case["kind"] == "batch":
        return rho
    shape = (case["ny"], case["nx"])
    out = {"rho": rho.reshape(shape)}
    if case["velocity"]:
        out.update(ux=ux.reshape(shape), uy=uy.reshape(shape), mass=float(rho.sum()))
    return out
