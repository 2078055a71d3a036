"""What this library is used for, as cases that can be timed.

Every case is a call sequence of a user's program: a simulation that is already set up is
advanced by a number of steps and read out (flow field on the GPU, states and forces of the
bodies on the host), a batch of requests is served, or fields are taken in and out through
host arrays.  The sizes are those of the paper's set-ups (workloads.py) and of the ranges the
serving mix draws from: boxes with edges 32 to 256, squirmers with radii 3 to 16, every storage.

``exact`` is an independent restatement of the method in plain torch FP64 (compressible
equilibrium, TRT / BGK, link bounce-back at the link midpoint, conversions, partially saturated
cells, the contact force with a round tube).
"""
import math

import numpy as np
import torch

from paper_1903_04799_gb300 import lbsq, workloads

BYTES = {"f64": 8, "f32": 4, "f16dev": 2, "bf16dev": 2}

# Velocity order of the library's public header: opposite pairs are adjacent.
C = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
              (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
              (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)], dtype=np.int64)
W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
OPP = [0] + [i + 1 if i % 2 else i - 1 for i in range(1, 19)]
MAGIC = 3.0 / 16.0


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # smallest call: the paper's fixed squirmer in a 32^3 box, where launches and the body
        # kernels' latency are the whole time
        {"name": "fixed_32_f64", "kind": "swim", "nx": 32, "ny": 32, "nz": 32, "storage": "f64", "collision": "bgk",
         "R": 4.0, "B1": 0.01, "beta": 0.0, "mobile": False, "psm": False, "steps": 200},
        # one free swimmer in the box of the swim-speed runs
        {"name": "swimmer_128_f32", "kind": "swim", "nx": 128, "ny": 128, "nz": 128, "storage": "f32",
         "collision": "trt", "R": 8.0, "B1": 0.005, "beta": 5.0, "mobile": True, "psm": False, "steps": 200},
        # odd edges (the serving mix draws any edge): neither paired loads nor whole-row blocks fit
        {"name": "swimmer_odd_f32", "kind": "swim", "nx": 125, "ny": 99, "nz": 111, "storage": "f32",
         "collision": "trt", "R": 6.5, "B1": 0.004, "beta": -2.0, "mobile": True, "psm": False, "steps": 150},
        # the 256^3 pusher of the precision study, in FP64 and in 16 bits
        {"name": "pusher_256_f64", "kind": "swim", "nx": 256, "ny": 256, "nz": 256, "storage": "f64",
         "collision": "trt", "R": 16.0, "B1": 0.002, "beta": -3.0, "mobile": True, "psm": False, "steps": 40},
        {"name": "pusher_256_f16", "kind": "swim", "nx": 256, "ny": 256, "nz": 256, "storage": "f16dev",
         "collision": "trt", "R": 16.0, "B1": 0.002, "beta": -3.0, "mobile": True, "psm": False, "steps": 64},
        # the same in partially saturated cells, the coupling without speed fluctuations
        {"name": "psm_256_f32", "kind": "swim", "nx": 256, "ny": 256, "nz": 256, "storage": "f32",
         "collision": "trt", "R": 16.0, "B1": 0.002, "beta": -3.0, "mobile": True, "psm": True, "steps": 48},
        # two squirmers passing each other: 250 is even but no multiple of four
        {"name": "pair_250_bf16", "kind": "pair", "n": 250, "storage": "bf16dev", "R": 9.0, "beta": 5.0, "steps": 60},
        # the dense suspension: 200 squirmers, every one's state read for its trajectory
        {"name": "suspension_256_f32", "kind": "suspension", "n": 256, "count": 200, "storage": "f32", "R": 6.0,
         "steps": 60},
        # a squirmer in a round tube, the long oscillation run
        {"name": "tube_f32", "kind": "tube", "R": 9.0, "storage": "f32", "steps": 200},
        # a flow without bodies and with another viscosity (the general relaxation)
        {"name": "flow_160_f64", "kind": "flow", "nx": 160, "ny": 144, "nz": 130, "storage": "f64", "lambda_e": 1.4,
         "steps": 50},
        # a batch of requests served together: boxes, tubes and obstacles of many sizes
        {"name": "serve_24", "kind": "serve", "count": 24, "lo": 32, "hi": 160, "steps": 256},
        # initial fields in, diagnostics, populations and fields out, all through host arrays
        {"name": "readout_128_f32", "kind": "readout", "nx": 128, "ny": 128, "nz": 128, "storage": "f32", "steps": 4},
    ]


def _edge(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _steps(rng, step_bytes, most):
    """A number of steps for which a pass stays well below the largest listed case."""
    return max(4, min(most, rng.randint(8, 200), int(1.2e11 / step_bytes)))


def draw(rng):
    kind = rng.choice(["swim", "swim", "swim", "pair", "suspension", "tube", "flow", "flow", "serve", "readout"])
    storage = rng.choice(["f64", "f32", "f16dev", "bf16dev"])
    if kind in ("swim", "flow", "readout"):
        hi = {"swim": 256, "flow": 224, "readout": 150}[kind]
        n = _edge(rng, 32, hi)
        nx, ny, nz = (max(30, min(hi, n + rng.randint(-n // 6, n // 6))) for _ in range(3))
        c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "storage": storage,
             "steps": _steps(rng, 38 * BYTES[storage] * nx * ny * nz, 200 if kind != "readout" else 8)}
        if kind == "flow":
            c["lambda_e"] = rng.choice([1.0, 1.0, round(rng.uniform(0.6, 1.7), 3)])
        if kind == "swim":
            c.update(collision=rng.choice(["trt", "trt", "bgk"]), B1=round(rng.uniform(0.002, 0.01), 4),
                     R=round(rng.uniform(3.0, min(16.0, (min(nx, ny, nz) - 10) / 4)), 2),
                     beta=round(rng.uniform(-5, 5), 2), mobile=rng.random() < 0.85, psm=rng.random() < 0.2)
        return c
    if kind == "pair":
        R = round(rng.uniform(4.0, 9.0), 1)
        n = max(40, int(R * rng.uniform(22, 28)))
        return {"kind": kind, "n": n, "storage": storage, "R": R, "beta": round(rng.uniform(-5, 5), 2),
                "steps": _steps(rng, 38 * BYTES[storage] * n ** 3, 100)}
    if kind == "suspension":
        n, R = rng.randint(120, 256), round(rng.uniform(4.0, 6.0), 1)
        count = max(4, int(200 * (n / 256) ** 3 * rng.uniform(0.5, 1.0)))
        return {"kind": kind, "n": n, "count": count, "storage": rng.choice(["f32", "f32", "f16dev"]), "R": R,
                "steps": _steps(rng, 152 * n ** 3, 48)}
    if kind == "tube":
        return {"kind": kind, "R": float(rng.randint(4, 12)), "storage": storage, "steps": rng.randint(20, 200)}
    return {"kind": "serve", "count": rng.randint(3, 24), "lo": 32, "hi": rng.randint(48, 150),
            "steps": rng.randint(64, 256)}


# ------------------------------------------------------------------ inputs

def _rng(seed):
    return np.random.default_rng(190304799 + int(seed))


def _unit(rng):
    v = rng.standard_normal(3)
    return tuple(float(a) for a in v / np.linalg.norm(v))


def _shape(case):
    kind = case["kind"]
    if kind in ("pair", "suspension"):
        return (case["n"],) * 3
    if kind == "tube":
        return workloads.tube_oscillation(R=case["R"]).shape
    return (case["nx"], case["ny"], case["nz"])


def _bodies(case, seed):
    """The spheres of a case, as workloads.Body."""
    rng, kind = _rng(seed), case["kind"]
    if kind == "swim":
        pos = tuple(float(n / 2 + d) for n, d in zip(_shape(case), rng.uniform(-1.5, 1.5, 3)))
        return [workloads.Body(pos, _unit(rng), case["R"], case["B1"], case["beta"], case["mobile"])]
    if kind == "pair":
        w = workloads.two_squirmers_passing(d=float(3 * case["R"] + rng.uniform(-2, 2)), n=case["n"], R=case["R"],
                                            beta=case["beta"])
        return w.bodies
    if kind == "suspension":
        return workloads.c4_suspension(case["n"], case["count"], case["R"], min_dist=34.0, seed=int(seed)).bodies
    if kind == "tube":
        t = workloads.tube_oscillation(y0_over_R=float(rng.uniform(-1.1, 1.1)), R=case["R"])
        b = t.body
        return [workloads.Body((b.pos[0], b.pos[1], b.pos[2] + float(rng.uniform(-3, 3))), b.e, b.R, b.B1, -1.5, True)]
    return []


def _fields(case, seed, amplitude):
    """Smooth periodic density and velocity (three low Fourier modes each), FP64, [z, y, x] / [3, z, y, x]."""
    nx, ny, nz = _shape(case)
    rng = _rng(seed + 7)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    ax = [torch.arange(n, dtype=torch.float64, device=dev) * (2 * math.pi / n) for n in (nx, ny, nz)]

    def modes():
        t = torch.zeros((nz, ny, nx), dtype=torch.float64, device=dev)
        for _ in range(3):
            k, ph = rng.integers(-2, 3, 3), float(rng.uniform(0, 2 * math.pi))
            a = [torch.polar(torch.ones_like(x), x * int(kk)) for x, kk in zip(ax, k)]
            t += (a[2][:, None, None] * a[1][None, :, None] * a[0][None, None, :] * complex(math.cos(ph), math.sin(ph))).real
        return t

    return 1.0 + 0.2 * amplitude * modes(), torch.stack([amplitude / 3 * modes() for _ in range(3)])


def _initial(case, seed):
    """(rho, u) a case starts from, or None: a fluid at rest."""
    amplitude = {"swim": 0.004, "flow": 0.02, "readout": 0.02}.get(case["kind"])
    return None if amplitude is None else _fields(case, seed, amplitude)


def _lambda_e(case):
    return float(case.get("lambda_e", 1.0))


def _requests(case, seed):
    mix = workloads.serving_mix(case["count"], seed=1903 + int(seed), steps_range=(case["steps"] // 2, case["steps"]),
                                edge_range=(case["lo"], case["hi"]))
    return [lbsq.make_request(q.geometry, q.shape, q.storage, pos=q.pos, e=q.e, R=q.R, B1=q.B1, beta=q.beta,
                              obstacle=q.obstacle, wca=q.wca, steps=q.steps) for q in mix]


# ------------------------------------------------------------------ a user's program

class _Sim:
    """A lattice, the ids of its spheres and the buffers its fields are read into."""

    def __init__(self, case, seed):
        shape = _shape(case)
        self.lat = lbsq.Lattice(shape, collision=case.get("collision", "trt"), lambda_e=_lambda_e(case),
                                storage=case["storage"])
        if case["kind"] == "tube":
            t = workloads.tube_oscillation(R=case["R"])
            self.lat.add_round_tube(*t.axis, t.radius)
            self.lat.set_contact(*t.contact)
        if case.get("psm"):
            self.lat.set_coupling("psm")
        self.ids = [self.lat.add_squirmer(b.pos, b.e, b.R, b.B1, b.beta, b.mobile) for b in _bodies(case, seed)]
        init = _initial(case, seed)
        self.host = None
        if init is not None:
            self.host = [t.cpu().numpy() for t in init]
            self.lat.set_fields(*self.host)
        self.steps = case["steps"]
        nx, ny, nz = shape
        self.rho = torch.zeros((nz, ny, nx), dtype=torch.float64, device="cuda")
        self.u = torch.zeros((3, nz, ny, nx), dtype=torch.float64, device="cuda")


def prepare(case, seed):
    if case["kind"] == "serve":
        srv = lbsq.Server(budget_bytes=6 << 30, max_resident=32)
        return {"kind": "serve", "srv": srv, "requests": _requests(case, seed)}
    return {"kind": case["kind"], "sim": _Sim(case, seed)}


def run(state):
    if state["kind"] == "serve":
        return _serve(state["srv"], state["requests"])
    if state["kind"] == "readout":
        return _readout(state["sim"])
    sim = state["sim"]
    lat = sim.lat
    lat.step(sim.steps)
    lbsq.lb_get_fields_device(lat.ctx, sim.rho.data_ptr(), sim.u.data_ptr())
    out = {"rho": sim.rho, "u": sim.u}
    if sim.ids:
        out["state"] = np.array([np.concatenate(lat.state(k)) for k in sim.ids])
        if len(sim.ids) <= 2:  # a trajectory run of a few bodies logs their forces too
            out["force"] = np.array([np.concatenate([*lat.force_torque(k), lat.stresslet(k)]) for k in sim.ids])
    return out


def _serve(srv, requests):
    left = {srv.submit(q): k for k, q in enumerate(requests)}
    rows, steps = [None] * len(requests), [0] * len(requests)
    while left:
        srv.advance()
        for t in list(left):
            r = srv.poll(t)
            if r.state in (lbsq.LB_REQ_DONE, lbsq.LB_REQ_FAILED):
                k = left.pop(t)
                rows[k] = np.concatenate([r.pos, r.vel, r.e, r.omega, r.F, r.T, [r.mean_speed], r.mean_vel])
                steps[k] = int(r.steps_done)
    return {"result": np.array(rows), "steps": np.array(steps)}


def _readout(sim):
    lat = sim.lat
    lat.set_fields(*sim.host)
    lat.step(sim.steps)
    mass, mom = lat.mass()
    rho, u = lat.fields()
    return {"totals": np.array([mass, *mom]), "rho": rho, "u": u, "f": lat.populations()}


def work(case):
    """Bytes and operations of one pass.  A step reads and writes every population once (neighbours
    couple every cell in every step) and takes about 250 operations per cell; then the outputs."""
    if case["kind"] == "serve":
        q = _requests(case, 0)
        upd = [(r.nx * r.ny * r.nz * r.steps, 4 if r.storage == lbsq.LB_F32 else 2) for r in q]
        return {"bytes": float(sum(38 * b * n for n, b in upd)), "flops": float(sum(250 * n for n, _ in upd))}
    n, b = math.prod(_shape(case)), BYTES[case["storage"]]
    if case["kind"] == "readout":
        # set-up: 32 B read and 19 b written; mass, fields, populations: 19 b read each, 32 + 152 B written
        return {"bytes": float(n * (38 * b * case["steps"] + 32 + 19 * b + 3 * 19 * b + 32 + 152)),
                "flops": float(n * (250 * case["steps"] + 400))}
    return {"bytes": float(n * (38 * b * case["steps"] + 19 * b + 32)), "flops": float(n * (250 * case["steps"] + 80))}


# ------------------------------------------------------------------ 64-bit reference

def _equilibrium(i, rho, u, uu):
    cu = sum(float(C[i, a]) * u[a] for a in range(3) if C[i, a])
    if i == 0:
        return W[0] * rho * (1.0 - 1.5 * uu)
    return W[i] * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu)


class _Exact:
    """The method in plain torch FP64: f[i, z, y, x], two arrays, one step after another."""

    def __init__(self, shape, le, lo, device):
        self.n = shape
        nx, ny, nz = shape
        self.le, self.lo, self.dev = le, lo, device
        self.zyx = (nz, ny, nx)
        self.N = nx * ny * nz
        w = torch.tensor(W, device=device)
        self.f = w[:, None, None, None].expand(19, nz, ny, nx).contiguous()
        self.owner = torch.zeros(self.N, dtype=torch.int32, device=device)
        self.c = torch.tensor(C, device=device)
        self.w = w
        self.opp = torch.tensor(OPP, device=device)
        self.walls, self.bodies, self.tube, self.contact = [], [], None, None
        self.psm = False

    def t(self, v):
        return torch.tensor(v, dtype=torch.float64, device=self.dev)

    def set_fields(self, rho, u):
        rho, u = rho.to(self.dev), u.to(self.dev)
        uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
        for i in range(19):
            self.f[i] = _equilibrium(i, rho, u, uu)

    def flat(self, xyz):
        nx, ny, _ = self.n
        return xyz[..., 0] + nx * (xyz[..., 1] + ny * xyz[..., 2])

    def coords(self, m):
        nx, ny, _ = self.n
        return torch.stack([m % nx, (m // nx) % ny, m // (nx * ny)], -1)

    def wrap(self, xyz):
        return torch.remainder(xyz, torch.tensor(self.n, device=self.dev))

    def image(self, d):
        n = self.t(self.n)
        return torch.where(d > n / 2, d - n, torch.where(d <= -n / 2, d + n, d))

    def add_tube(self, cx, cy, r):
        nx, ny, nz = self.n
        x = torch.arange(nx, dtype=torch.float64, device=self.dev)
        y = torch.arange(ny, dtype=torch.float64, device=self.dev)
        solid = ((x[None, :] - cx) ** 2 + (y[:, None] - cy) ** 2 >= r * r).expand(nz, ny, nx).reshape(-1)
        self.walls.append((1, torch.nonzero(solid).squeeze(1)))
        self.owner[solid] = 1
        self.tube = (cx, cy, r)

    def box(self, b):
        lo = torch.floor(self.t(b["pos"]) - b["R"]).long() - 2
        k = torch.arange(int(math.ceil(2 * b["R"])) + 6, device=self.dev)
        return self.wrap(lo + torch.stack(torch.meshgrid(k, k, k, indexing="ij"), -1).reshape(-1, 3))

    def inside(self, b):
        x = self.box(b)
        d = self.image(x.double() - self.t(b["pos"]))
        d2 = (d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2]
        return self.flat(x[d2 < b["R"] * b["R"]])

    def add_sphere(self, body):
        m = 4.0 / 3.0 * math.pi * body.R ** 3
        b = {"pos": [p - math.floor(p / n) * n for p, n in zip(body.pos, self.n)], "R": body.R, "B1": body.B1,
             "B2": body.beta * body.B1, "mobile": body.mobile, "M": m, "I": 0.4 * m * body.R ** 2,
             "e": np.array(body.e) / np.linalg.norm(body.e), "v": np.zeros(3), "w": np.zeros(3), "Fc": np.zeros(6),
             "out": np.zeros(12), "id": 2 + len(self.bodies)}
        b["pos"] = np.array(b["pos"])
        if not self.psm:
            b["cells"] = self.inside(b)
            self.owner[b["cells"]] = b["id"]
        self.bodies.append(b)

    def surface_velocity(self, b, d):
        e, v, w = self.t(b["e"]), self.t(b["v"]), self.t(b["w"])
        r = d.norm(dim=-1, keepdim=True)
        n = torch.where(r > 0, d / r, torch.zeros_like(d))
        ct = (n * e).sum(-1, keepdim=True)
        slip = torch.where(r > 0, (b["B1"] + b["B2"] * ct) * (ct * n - e), torch.zeros_like(d))
        return v + torch.linalg.cross(w.expand_as(d), d) + slip

    def moments(self, d, dF):
        """Force, torque and stresslet of momentum dF given to the body at offsets d."""
        F, T = dF.sum(0), torch.linalg.cross(d, dF).sum(0)
        tr = (d * dF).sum(-1) / 3
        S = [-(d[:, a] * dF[:, a] - tr).sum() for a in range(3)]
        S += [-0.5 * (d[:, a] * dF[:, b] + d[:, b] * dF[:, a]).sum() for a, b in ((0, 1), (0, 2), (1, 2))]
        return torch.cat([F, T, torch.stack(S)]).cpu().numpy()

    def collide(self):
        f = self.f
        rho = f.sum(0)
        j = [sum(float(C[i, a]) * f[i] for i in range(19) if C[i, a]) for a in range(3)]
        u = [x / rho for x in j]
        uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
        f[0] += self.le * (_equilibrium(0, rho, u, uu) - f[0])
        for i in range(1, 19, 2):
            a, b = f[i], f[i + 1]
            ea, eb = _equilibrium(i, rho, u, uu), _equilibrium(i + 1, rho, u, uu)
            even = self.le * 0.5 * ((ea + eb) - (a + b))
            odd = self.lo * 0.5 * ((ea - eb) - (a - b))
            f[i], f[i + 1] = a + even + odd, b + even - odd

    def links(self, cells):
        """(fluid node, direction) of every link into the solid cells."""
        i = torch.arange(1, 19, device=self.dev)
        src = self.flat(self.wrap(self.coords(cells)[:, None, :] - self.c[None, 1:, :]))
        keep = self.owner[src] == 0
        return src[keep], i[None, :].expand(len(cells), 18)[keep]

    def bounce(self):
        """Reflected populations (slots and values) and the bodies' forces, from the post-collision state."""
        f, hits = self.f.view(19, -1), []
        for _, cells in self.walls:
            n, i = self.links(cells)
            hits.append((n, self.opp[i], f[i, n]))
        for b in self.bodies:
            n, i = self.links(b["cells"])
            ci = self.c[i].double()
            d = self.image(self.coords(n).double() + 0.5 * ci - self.t(b["pos"]))
            out = f[i, n]
            back = out - 6.0 * self.w[i] * (ci * self.surface_velocity(b, d)).sum(-1)
            hits.append((n, self.opp[i], back))
            b["out"] = self.moments(d, ci * (out + back)[:, None])
        return hits

    def psm_cover(self):
        """Partially saturated cells: solid fraction, blended collision and forces, from the state before the step."""
        k = (torch.arange(8, dtype=torch.float64, device=self.dev) + 0.5) / 8 - 0.5
        pts = torch.stack(torch.meshgrid(k, k, k, indexing="ij"), -1).reshape(-1, 3)
        f, hits = self.f.view(19, -1), []
        th = 1.0 / self.le - 0.5
        for b in self.bodies:
            x = self.box(b)
            d = self.image(x.double() - self.t(b["pos"]))
            eps = torch.cat([((c[:, None, :] + pts).square().sum(-1) < b["R"] ** 2).double().mean(-1)
                             for c in d.split(4096)])
            x, d, eps = x[eps > 0], d[eps > 0], eps[eps > 0]
            n = self.flat(x)
            g = f[:, n]
            rho = g.sum(0)
            u = (self.c.double().T @ g) / rho
            us = self.surface_velocity(b, d).T
            uu, ss = u.square().sum(0), us.square().sum(0)
            eq = torch.stack([_equilibrium(i, rho, u, uu) for i in range(19)])
            es = torch.stack([_equilibrium(i, rho, us, ss) for i in range(19)])
            solid = (g[self.opp] - eq[self.opp]) - (g - es)
            neq = eq - g
            fluid = self.le * 0.5 * (neq + neq[self.opp]) + self.lo * 0.5 * (neq - neq[self.opp])
            B = eps * th / ((1 - eps) + th)
            hits.append((n, g + (1 - B) * fluid + B * solid))
            b["out"] = self.moments(d, -(B * (self.c.double().T @ solid)).T)
        return hits

    def contact_force(self, b):
        F = np.zeros(3)
        if self.contact and self.tube:
            sigma, eps = self.contact
            cx, cy, r = self.tube
            dx, dy = b["pos"][0] - cx, b["pos"][1] - cy
            rho = math.hypot(dx, dy)
            gap = (r - 0.5) - rho - b["R"]
            if gap < 2 ** (1 / 6) * sigma and rho > 0:
                s = sigma / max(gap, 0.05 * sigma)
                k = 24 * eps / max(gap, 0.05 * sigma) * (2 * s ** 12 - s ** 6)
                F[:2] -= k * np.array([dx, dy]) / rho
        return F

    def advance(self, b):
        """Symplectic Euler and rotation; the force that entered, with torque and stresslet, in b["log"]."""
        FT = b["out"][:6] + b["Fc"]
        b["log"] = np.concatenate([FT, b["out"][6:]])
        b["Fc"] = np.zeros(6)
        if not b["mobile"]:
            return
        b["v"] = b["v"] + (FT[:3] + self.contact_force(b)) / b["M"]
        b["w"] = b["w"] + FT[3:] / b["I"]
        x = b["pos"] + b["v"]
        n = np.array(self.n, dtype=np.float64)
        b["pos"] = np.where(x >= n, x - n, np.where(x < 0, x + n, x))
        th = np.linalg.norm(b["w"])
        if th > 0:
            k, e = b["w"] / th, b["e"]
            e = e * math.cos(th) + np.cross(k, e) * math.sin(th) + k * (k @ e) * 2 * math.sin(th / 2) ** 2
            b["e"] = e / np.linalg.norm(e)

    def remap(self, b):
        before = b["cells"]
        after = self.inside(b)
        b["cells"] = after
        if len(before) == len(after) and torch.equal(before.sort().values, after.sort().values):
            return
        f, pos = self.f.view(19, -1), self.t(b["pos"])
        covered, opened = after[~torch.isin(after, before)], before[~torch.isin(before, after)]
        fluid = self.owner == 0  # before the change
        self.owner[opened] = 0
        self.owner[covered] = b["id"]

        def book(cells, mom, sign):
            d = self.image(self.coords(cells).double() - pos)
            tot = torch.cat([mom.sum(0), torch.linalg.cross(d, mom).sum(0)]).cpu().numpy()
            b["Fc"] = b["Fc"] + sign * tot

        if len(covered):
            book(covered, (self.c.double().T @ f[:, covered]).T, 1.0)
        if len(opened):
            near = self.flat(self.wrap(self.coords(opened)[:, None, :] + self.c[None, 1:, :]))
            ok = (self.owner[near] == 0) & fluid[near]
            rho = (f[:, near].sum(0) * ok).sum(-1) / ok.sum(-1).clamp(min=1)
            rho = torch.where(ok.any(-1), rho, torch.ones_like(rho))
            d = self.image(self.coords(opened).double() - pos)
            u = (self.t(b["v"]) + torch.linalg.cross(self.t(b["w"]).expand_as(d), d)).T
            uu = u.square().sum(0)
            new = torch.stack([_equilibrium(i, rho, u, uu) for i in range(19)])
            f[:, opened] = new
            book(opened, (self.c.double().T @ new).T, -1.0)

    def step(self):
        covered = self.psm_cover() if self.psm else []
        self.collide()
        f = self.f.view(19, -1)
        for n, g in covered:
            f[:, n] = g
        hits = [] if self.psm else self.bounce()
        for i in range(1, 19):
            self.f[i] = torch.roll(self.f[i], tuple(int(a) for a in C[i][::-1]), (0, 1, 2))
        for n, i, back in hits:
            f[i, n] = back
        for b in self.bodies:
            self.advance(b)
        if not self.psm:
            for b in self.bodies:
                if b["mobile"]:
                    self.remap(b)

    def fields(self):
        fluid = (self.owner == 0).view(self.zyx)
        rho = self.f.sum(0)
        u = torch.stack([sum(float(C[i, a]) * self.f[i] for i in range(19) if C[i, a]) / rho for a in range(3)])
        return rho * fluid, u * fluid


def exact(case, seed):
    if case["kind"] == "serve":
        return None  # a batch of whole simulations
    shape = _shape(case)
    if math.prod(shape) * case["steps"] > 1.2e9:
        return None  # over about 20 seconds
    le = _lambda_e(case)
    lo = le if case.get("collision") == "bgk" else 1.0 / (0.5 + MAGIC / (1.0 / le - 0.5))
    x = _Exact(shape, le, lo, "cuda" if torch.cuda.is_available() else "cpu")
    if case["kind"] == "tube":
        t = workloads.tube_oscillation(R=case["R"])
        x.add_tube(*t.axis, t.radius)
        x.contact = t.contact
    x.psm = bool(case.get("psm"))
    for b in _bodies(case, seed):
        x.add_sphere(b)
    init = _initial(case, seed)
    if init is not None:
        x.set_fields(*init)
    for _ in range(case["steps"]):
        x.step()
    rho, u = x.fields()
    if case["kind"] == "readout":
        totals = torch.stack([rho.sum(), *((u[a] * rho).sum() for a in range(3))])
        return {"totals": totals, "rho": rho.reshape(-1), "u": u.reshape(3, -1),
                "f": x.f.reshape(19, -1)}
    out = {"rho": rho, "u": u}
    if x.bodies:
        out["state"] = np.array([np.concatenate([b["pos"], b["v"], b["e"], b["w"]]) for b in x.bodies])
        if len(x.bodies) <= 2:
            out["force"] = np.array([b["log"] for b in x.bodies])
    return out
