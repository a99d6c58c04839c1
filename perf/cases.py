"""What a program does with this library, as timed cases: simulations of the paper's setups
(arXiv:1909.04166, Secs. 6.1 - 7) advanced through the public calls, over the grid sizes, storage
precisions, side kinds and operator forms that the library offers.

A case of kind "run" is one simulation in a caller-supplied device buffer: initialise it from
device fields, advance it, and read its state in place (lbm_init_fields_device, lbm_step,
lbm_state_device).  A "session" is the same through host arrays (init, step, diagnostics, fields),
and a "batch" advances many independent drops together and reads every case's fields.

``exact`` restates the scheme in float64 torch: moments by moment matrices, streaming by an index
map; it shares nothing with the library but the problem statement and the documented state layout.
"""
import math

import numpy as np
import torch

from paper_1909_04166_gb300 import lbm

E_X = (0, 1, 0, -1, 0, 1, -1, -1, 1)
E_Y = (0, 0, 1, 0, -1, 1, 1, -1, -1)
WEIGHTS = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
BYTES_PER_NODE = {"fp64": 144, "fp32": 72, "fp16": 44, "bf16": 44}
# floating-point operations of one node update (both collisions, forces, stencils, sums): about
# 600 counted from the formulas; the interface lattice alone about 200
FLOPS_PER_NODE = 600
FLOPS_PER_NODE_SHEAR = 200
FIELDS = ("phi", "p", "ux", "uy", "rho")
EXACT_CASES = 2   # cases of a batch that exact() restates


def listed():
    return [
        # the static drop of Sec. 6.2 in the library's correctness precision
        {"name": "laplace_fp64", "kind": "run", "setup": "laplace", "nx": 64, "ny": 64,
         "precision": "fp64", "steps": 200},
        # the same drop in FP32 watched closely: a short call between two looks at the state
        {"name": "laplace_fp32_short", "kind": "run", "setup": "laplace", "nx": 64, "ny": 64,
         "precision": "fp32", "steps": 20},
        # surfactant-driven drop (Sec. 6.7): a narrow odd channel, Langmuir isotherm, long runs
        {"name": "young_fp32", "kind": "run", "setup": "young", "nx": 51, "ny": 201,
         "precision": "fp32", "steps": 1000},
        # rising bubble (Sec. 6.5): odd sides, free-slip walls beside no-slip ends
        {"name": "bubble_fp32", "kind": "run", "setup": "bubble", "nx": 161, "ny": 481,
         "precision": "fp32", "steps": 500},
        # thermocapillary drop (Sec. 6.7) with 16-bit storage
        {"name": "marangoni_bf16", "kind": "run", "setup": "marangoni", "nx": 512, "ny": 256,
         "precision": "bf16", "steps": 500},
        # Rayleigh-Taylor (Sec. 6.3) as a program with host arrays runs it between two samples
        {"name": "rt_session_fp32", "kind": "session", "setup": "rt", "nx": 256, "ny": 1024,
         "precision": "fp32", "steps": 1600},
        # the bandwidth headline: drop impact at density ratio 1000 (Sec. 6.6)
        {"name": "impact_fp32", "kind": "run", "setup": "impact", "nx": 2048, "ny": 1024,
         "precision": "fp32", "steps": 500},
        # the same with 16-bit storage
        {"name": "impact_fp16", "kind": "run", "setup": "impact", "nx": 2048, "ny": 1024,
         "precision": "fp16", "steps": 500},
        # a large impact: several gigabytes of state traffic per step
        {"name": "impact_large_fp32", "kind": "run", "setup": "impact", "nx": 4096, "ny": 4096,
         "precision": "fp32", "steps": 100},
        # a ragged impact channel of the paper's own size (1501 x 501), short of one full wave
        {"name": "impact_ragged_fp32", "kind": "run", "setup": "impact", "nx": 1501, "ny": 501,
         "precision": "fp32", "steps": 300},
        # the interface lattice alone in the reversing vortex (Sec. 6.1)
        {"name": "shear_fp32", "kind": "run", "setup": "shear", "nx": 800, "ny": 800,
         "precision": "fp32", "steps": 500},
        # many independent drops of uneven sizes, read out at a checkpoint (Sec. 7 style sweep)
        {"name": "batch_fp32", "kind": "batch", "setup": "drops", "ncases": 192, "side_min": 32,
         "side_max": 256, "precision": "fp32", "steps": 2000},
    ]


# setup -> (grid ranges, precisions it is run in)
RANGES = {
    "laplace": ((32, 256), (32, 256), ("fp64", "fp32", "fp32")),
    "young": ((40, 160), (150, 400), ("fp32",)),
    "bubble": ((100, 400), (300, 900), ("fp32", "fp32", "fp16")),
    "marangoni": ((200, 800), (120, 500), ("fp32", "fp16", "bf16", "fp64")),
    "rt": ((100, 600), (400, 1600), ("fp32",)),
    "impact": ((900, 4096), (400, 4096), ("fp32", "fp32", "fp16", "bf16")),
    "shear": ((128, 2048), (128, 2048), ("fp32",)),
    "drops": (None, None, ("fp32", "fp16")),
}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    setup = rng.choice(sorted(RANGES))
    xs, ys, precisions = RANGES[setup]
    precision = rng.choice(precisions)
    if setup == "drops":
        n = _log_int(rng, 16, 192)
        return {"kind": "batch", "setup": setup, "ncases": n, "side_min": 32, "side_max": 256,
                "precision": precision, "steps": _log_int(rng, 100, 1000)}
    nx, ny = _log_int(rng, *xs), _log_int(rng, *ys)
    if setup == "shear":
        ny = nx                                   # the vortex fills a square box
    if setup in ("laplace", "rt", "impact") and rng.random() < 0.5:
        nx, ny = 32 * max(1, nx // 32), 32 * max(1, ny // 32)
    # no dearer than the largest listed case: steps within its node updates (FP64 runs about 15
    # times slower)
    most = 4096 * 4096 * 100 // (15 if precision == "fp64" else 1)
    steps = max(2, min(_log_int(rng, 20, 1000), most // (nx * ny)))
    kind = "session" if setup in ("rt", "marangoni") and rng.random() < 0.25 else "run"
    return {"kind": kind, "setup": setup, "nx": nx, "ny": ny, "precision": precision,
            "steps": steps}


# ---- inputs --------------------------------------------------------------------------------------

def _tanh(zeta, width):
    return 0.5 + 0.5 * torch.tanh(2.0 * zeta / width)


def _problem(case, seed):
    """Parameters (keys of lbm.make_params) and initial device fields of a single-grid case; the
    seed moves the drop and adds a velocity perturbation of about 1 % of the flow's scale."""
    setup, nx, ny = case["setup"], case["nx"], case["ny"]
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    host = np.random.default_rng(int(seed))
    jx, jy = host.uniform(-0.5, 0.5), host.uniform(-0.5, 0.5)
    f64 = dict(dtype=torch.float64, device="cuda")
    x = torch.arange(nx, **f64)[None, :]
    y = torch.arange(ny, **f64)[:, None]
    c = dict(nx=nx, ny=ny, wall_x=0, wall_y=0, rho_a=1.0, rho_b=1.0, mu_a=0.1, mu_b=0.1,
             mobility=0.02, width=4.0)
    uy0 = None
    if setup == "laplace":
        c.update(rho_b=1e-3, mu_a=0.1, mu_b=1e-4, sigma0=1e-3, width=5.0)
        phi = _tanh(0.25 * min(nx, ny) - torch.hypot(x - nx / 2 - jx, y - ny / 2 - jy), 5.0)
        scale = 1e-4
    elif setup == "young":
        c.update(wall_y=1, mu_a=0.05, mu_b=0.05, sigma0=0.0244 / 5.0, sigma_model=1, beta=5.0,
                 gradpsi_y=min(9.95e-5, 0.02 / ny))
        phi = _tanh(15.0 - torch.hypot(x - nx // 2 - jx, y - 45.0 - jy), 4.0)
        scale = 1e-4
    elif setup == "bubble":
        d, ug = 0.4 * min(nx, 200), 0.02
        mu_a = ug * d / 35.0
        c.update(wall_x=2, wall_y=1, rho_b=0.1, mu_a=mu_a, mu_b=mu_a / 10.0,
                 sigma0=ug * ug * d / 10.0, gy=-ug * ug / d, rho_ref=1.0)
        phi = _tanh(torch.hypot(x - nx / 2 - jx, y - 0.25 * ny - jy) - d / 2, 4.0)
        scale = 0.01 * ug
    elif setup == "marangoni":
        c.update(wall_y=1, rho_b=0.1, mu_a=0.05, mu_b=0.05, sigma0=1e-3, dsigma_dT=-2e-6,
                 gradT_x=0.01)
        phi = _tanh(0.125 * min(nx, ny) - torch.hypot(x - nx / 2 - jx, y - ny / 2 - jy), 4.0)
        scale = 1e-5
    elif setup == "rt":
        uc = 0.04
        nu, rho_b = uc * nx / 3000.0, 1.0 / 3.0
        c.update(wall_y=1, rho_b=rho_b, mu_a=nu, mu_b=nu * rho_b, sigma0=5e-5, mobility=0.1,
                 width=5.0, gy=-uc * uc / nx, rho_ref=0.5 * (1.0 + rho_b))
        yi = ny / 2 + jy + 0.1 * nx * torch.cos(2 * math.pi * (x - jx) / nx)
        phi = _tanh(y - yi, 5.0)
        scale = 0.01 * uc
    elif setup == "impact":
        u, d = 0.05, 0.2 * min(nx, ny)
        mu_a = u * d / 100.0
        c.update(wall_y=1, rho_b=1e-3, mu_a=mu_a, mu_b=mu_a / 10.0, sigma0=u * u * d / 8000.0,
                 mobility=0.1, width=5.0)
        film = 0.1 * d
        drop = _tanh(d / 2 - torch.hypot(x - nx / 2 - jx, y - film - d / 2), 5.0)
        phi = torch.maximum(_tanh(film - y, 5.0).expand(ny, nx), drop)
        uy0 = -u * drop
        scale = 0.01 * u
    elif setup == "shear":
        c.update(mobility=0.02 * 3.0 / 60.0, width=3.0, flow=1, u0=0.02,
                 reverse_step=int(round(nx / 0.02)))
        phi = _tanh(0.2 * nx - torch.hypot(x - nx / 2 - jx, y - 0.3 * ny - jy), 3.0)
        scale = 0.0
    else:
        raise ValueError(setup)
    phi = phi.expand(ny, nx).contiguous()
    # the perturbation sits in the heavy phase, as a stirred liquid's would
    ux = scale * torch.randn(ny, nx, generator=gen, **f64) * phi
    uy = scale * torch.randn(ny, nx, generator=gen, **f64) * phi
    if uy0 is not None:
        uy = uy + uy0
    return c, (phi, torch.zeros_like(phi), ux, uy)


def _drops(case, seed):
    """The cases of a batch: drops of uneven grids, density ratios, surface tensions."""
    host = np.random.default_rng(int(seed))
    out = []
    for i in range(case["ncases"]):
        # the grids belong to the case (every seed runs the same work), the physics to the seed
        g = np.random.default_rng(1000 + i)
        nx = int(g.integers(case["side_min"], case["side_max"] + 1))
        ny = int(g.integers(case["side_min"], case["side_max"] + 1))
        r = float(host.uniform(0.2, 0.35)) * min(nx, ny)
        rho_b = 1.0 / math.exp(host.uniform(math.log(10.0), math.log(1000.0)))
        sigma = math.exp(host.uniform(math.log(1e-4), math.log(1e-2)))
        a, b = (r, r) if i % 2 == 0 else (r * math.sqrt(5 / 3), r * math.sqrt(3 / 5))
        c = dict(nx=nx, ny=ny, wall_x=0, wall_y=0, rho_a=1.0, rho_b=rho_b, mu_a=0.1,
                 mu_b=0.1 * rho_b, sigma0=sigma, mobility=0.02, width=5.0)
        y, x = np.mgrid[0:ny, 0:nx].astype(np.float64)
        d = (np.hypot((x - nx / 2) / a, (y - ny / 2) / b) - 1.0) * min(a, b)
        amp = 0.01 * math.sqrt(sigma / r)
        phi = 0.5 + 0.5 * np.tanh(-2.0 * d / 5.0)
        c["fields"] = dict(phi=phi, p=np.zeros_like(phi),
                           ux=amp * host.standard_normal((ny, nx)),
                           uy=amp * host.standard_normal((ny, nx)))
        out.append(c)
    return out


class _Run:
    """A context in a torch buffer with its initial device fields."""

    def __init__(self, case, seed):
        self.steps = case["steps"]
        self.problem, self.fields = _problem(case, seed)
        self.ny = case["ny"]
        self.params = lbm.make_params(self.problem, case["precision"],
                                      stream=torch.cuda.current_stream().cuda_stream)
        nbytes = lbm.lbm_state_bytes(self.params)
        self.buffer = torch.zeros(nbytes, dtype=torch.uint8, device="cuda")
        self.ctx = lbm.lbm_create_with_buffer(self.params, self.buffer.data_ptr(), nbytes)
        self.precision = case["precision"]
        self.shear = case["setup"] == "shear"

    def state(self):
        """The current state as views of the buffer (layout of lbm_state_device)."""
        ptr, nstrips, _ = lbm.lbm_state_device(self.ctx)
        half = self.buffer.numel() // 2
        raw = self.buffer.narrow(0, ptr - self.buffer.data_ptr(), half)
        if self.precision in ("fp16", "bf16"):
            raw = raw.view(self.ny, nstrips, 1408)
            dtype = torch.float16 if self.precision == "fp16" else torch.bfloat16
            return {"z": raw[..., :256].view(torch.float32).view(self.ny, nstrips, 2, 32),
                    "d": raw[..., 256:].view(dtype).view(self.ny, nstrips, 18, 32)}
        dtype = torch.float64 if self.precision == "fp64" else torch.float32
        pops = raw.view(dtype).view(self.ny, nstrips, 18, 32)
        return {"f": pops[:, :, 9:]} if self.shear else {"pops": pops}

    def __del__(self):
        try:
            lbm.lbm_destroy(self.ctx)
        except Exception:
            pass


class _Session:
    def __init__(self, case, seed):
        self.steps = case["steps"]
        self.problem, fields = _problem(case, seed)
        self.fields = [f.cpu().numpy() for f in fields]
        self.sim = lbm.Simulation(self.problem, precision=case["precision"])


class _Sweep:
    """A batch and the host arrays its fields are read into: the first EXACT_CASES cases one by
    one, the others end to end in one array per field."""

    def __init__(self, case, seed):
        self.steps = case["steps"]
        self.cases = _drops(case, seed)
        self.batch = lbm.Batch(self.cases, precision=case["precision"]).init_all()
        sizes = [c["nx"] * c["ny"] for c in self.cases]
        rest = {k: np.empty(sum(sizes[EXACT_CASES:])) for k in FIELDS}
        self.out = {"first": [{k: np.empty((c["ny"], c["nx"])) for k in FIELDS}
                              for c in self.cases[:EXACT_CASES]], "rest": rest}
        self.into, at = list(self.out["first"]), 0
        for n in sizes[EXACT_CASES:]:
            self.into.append({k: rest[k][at:at + n] for k in FIELDS})
            at += n

    def fields(self):
        for i, into in enumerate(self.into):
            lbm.lbm_batch_get_fields(self.batch.b, i, *(into[k] for k in FIELDS))
        return self.out


def prepare(case, seed):
    return {"run": _Run, "session": _Session, "batch": _Sweep}[case["kind"]](case, seed)


def run(state):
    if isinstance(state, _Run):
        lbm.lbm_init_fields_device(state.ctx, *(f.data_ptr() for f in state.fields))
        lbm.lbm_step(state.ctx, state.steps)
        return state.state()
    if isinstance(state, _Session):
        sim = state.sim
        sim.init(*state.fields).step(state.steps)
        return {"diagnostics": sim.diagnostics(), "fields": sim.fields()}
    state.batch.step(state.steps)
    return state.fields()


def work(case):
    per_node = BYTES_PER_NODE[case["precision"]]
    if case["kind"] == "batch":
        nodes = sum(c[0] * c[1] for c in _batch_grids(case))
        # the state read and written once, and five fields per node written for the host
        return {"bytes": nodes * (2 * per_node + 40),
                "flops": nodes * case["steps"] * FLOPS_PER_NODE}
    nodes = case["nx"] * case["ny"]
    flops = FLOPS_PER_NODE
    if case["setup"] == "shear":
        per_node, flops = per_node // 2, FLOPS_PER_NODE_SHEAR
    # four fields read and the state written (and, in a session, five fields read from it)
    extra = 40 + per_node if case["kind"] == "session" else 0
    return {"bytes": nodes * (32 + per_node + extra), "flops": nodes * case["steps"] * flops}


def _batch_grids(case):
    for i in range(case["ncases"]):
        g = np.random.default_rng(1000 + i)
        yield (int(g.integers(case["side_min"], case["side_max"] + 1)),
               int(g.integers(case["side_min"], case["side_max"] + 1)))


# ---- the scheme in float64 torch -------------------------------------------------------------------

class _Exact:
    """Both lattices of one grid in float64: populations [9, ny, nx]."""

    def __init__(self, problem, device="cuda"):
        P = self.P = dict(wall_x=0, wall_y=0, sigma0=0.0, dsigma_dT=0.0, gradT_x=0.0, gradT_y=0.0,
                          gx=0.0, gy=0.0, rho_ref=0.0, sigma_model=0, beta=0.0, psi0=0.0,
                          gradpsi_x=0.0, gradpsi_y=0.0, flow=0, u0=0.0, reverse_step=0)
        P.update(problem)
        nx, ny = P["nx"], P["ny"]
        self.t = 0
        opt = dict(dtype=torch.float64, device=device)
        self.x = torch.arange(nx, **opt)[None, :].expand(ny, nx)
        self.y = torch.arange(ny, **opt)[:, None].expand(ny, nx)
        # neighbour rows and columns of the stencils: mirror ghosts at walls, else periodic

        def around(n, wall):
            i = torch.arange(-1, n + 1, device=device)
            return i.clamp(0, n - 1) if wall else i % n

        self.ix, self.iy = around(nx, P["wall_x"]), around(ny, P["wall_y"])
        # destination of every population, inverted into one gather map
        xi = torch.arange(nx, device=device)[None, :].expand(ny, nx)
        yi = torch.arange(ny, device=device)[:, None].expand(ny, nx)
        dest = torch.empty(9, ny, nx, dtype=torch.int64, device=device)
        opposite = {(ex, ey): a for a, (ex, ey) in enumerate(zip(E_X, E_Y))}
        for a, (ex, ey) in enumerate(zip(E_X, E_Y)):
            cx = ((xi + ex < 0) | (xi + ex >= nx)) & bool(P["wall_x"])
            cy = ((yi + ey < 0) | (yi + ey >= ny)) & bool(P["wall_y"])
            back = (cx & (P["wall_x"] == 1)) | (cy & (P["wall_y"] == 1))
            sx = torch.where(back | cx, 0, ex)    # the step taken along x, along y
            sy = torch.where(back | cy, 0, ey)
            tx, ty = (xi + sx) % nx, (yi + sy) % ny
            plane = torch.full_like(xi, a)
            for rx, ry, mask in ((-ex, ey, cx & ~cy & ~back), (ex, -ey, cy & ~cx & ~back),
                                 (-ex, -ey, back | (cx & cy))):
                plane = torch.where(mask, opposite[(rx, ry)], plane)
            dest[a] = (plane * ny + ty) * nx + tx
        self.gather = torch.empty(9 * nx * ny, dtype=torch.int64, device=device)
        self.gather[dest.reshape(-1)] = torch.arange(9 * nx * ny, device=device)
        ex, ey = torch.tensor(E_X, **opt), torch.tensor(E_Y, **opt)
        # raw moments 00 10 01 20 02 11 21 12 22 and the inverse
        self.M = torch.stack([ex ** i * ey ** j for i, j in
                              ((0, 0), (1, 0), (0, 1), (2, 0), (0, 2), (1, 1), (2, 1), (1, 2),
                               (2, 2))])
        self.Minv = torch.linalg.inv(self.M.cpu()).to(device)

    def pops(self, raw):
        return torch.tensordot(self.Minv, torch.stack(raw), 1)

    def raw(self, q):
        return list(torch.tensordot(self.M, q, 1))

    @staticmethod
    def shifted(r, ux, uy):
        """Moments about (ux, uy) from moments about 0 (the reverse shift takes -u)."""
        m00, m10, m01, m20, m02, m11, m21, m12, m22 = r
        ux2, uy2, uxy = ux * ux, uy * uy, ux * uy
        return [m00, m10 - ux * m00, m01 - uy * m00,
                m20 - 2 * ux * m10 + ux2 * m00, m02 - 2 * uy * m01 + uy2 * m00,
                m11 - ux * m01 - uy * m10 + uxy * m00,
                m21 - 2 * ux * m11 - uy * m20 + 2 * uxy * m10 + ux2 * m01 - ux2 * uy * m00,
                m12 - 2 * uy * m11 - ux * m02 + 2 * uxy * m01 + uy2 * m10 - ux * uy2 * m00,
                m22 - 2 * ux * m12 - 2 * uy * m21 + ux2 * m02 + uy2 * m20 + 4 * uxy * m11
                - 2 * ux * uy2 * m10 - 2 * ux2 * uy * m01 + ux2 * uy2 * m00]

    def init(self, phi, p, ux, uy):
        P = self.P
        rho = P["rho_b"] + phi * (P["rho_a"] - P["rho_b"])
        zero = torch.zeros_like(phi)
        c = self._fluid_eq(p, p - rho / 3, ux, uy)
        c[1], c[2] = -(p - rho / 3) * ux, -(p - rho / 3) * uy
        self.g = self.pops(self.shifted(c, -ux, -uy))
        c = [phi, zero, zero, phi / 3, phi / 3, zero, zero, zero, phi / 9]
        self.f = self.pops(self.shifted(c, -ux, -uy))
        return self

    @staticmethod
    def _fluid_eq(p, psi, ux, uy):
        ux2, uy2 = ux * ux, uy * uy
        return [p, None, None, p / 3 + psi * ux2, p / 3 + psi * uy2, psi * ux * uy,
                -psi * uy * (1 / 3 + ux2), -psi * ux * (1 / 3 + uy2),
                p / 9 + psi * ((ux2 + uy2) / 3 + ux2 * uy2)]

    def _window(self, a):
        w = a[self.iy][:, self.ix]
        ny, nx = a.shape
        return {(i, j): w[1 + j:1 + j + ny, 1 + i:1 + i + nx] for i in (-1, 0, 1)
                for j in (-1, 0, 1)}

    @staticmethod
    def _grad(w):
        gx = ((w[1, 0] - w[-1, 0]) * 4 + (w[1, 1] + w[1, -1] - w[-1, 1] - w[-1, -1])) / 12
        gy = ((w[0, 1] - w[0, -1]) * 4 + (w[1, 1] + w[-1, 1] - w[1, -1] - w[-1, -1])) / 12
        return gx, gy

    def imposed(self):
        P = self.P
        s = -1.0 if P["reverse_step"] > 0 and self.t >= P["reverse_step"] else 1.0
        a = s * P["u0"] * math.pi
        xa, ya = math.pi * (self.x / P["nx"] - 0.5), math.pi * (self.y / P["ny"] - 0.5)
        return -a * torch.cos(xa) * torch.sin(ya), a * torch.sin(xa) * torch.cos(ya)

    def macro(self):
        P, g = self.P, self.g
        phi, ps = self.f.sum(0), g.sum(0)
        w = self._window(phi)
        dx, dy = self._grad(w)
        g2 = dx * dx + dy * dy
        gm = g2.sqrt()
        nx, ny = dx / (gm + 1e-6), dy / (gm + 1e-6)
        theta = 4.0 / P["width"] * phi * (1 - phi)
        m = dict(phi=phi, ps=ps, jx=P["mobility"] * theta * nx, jy=P["mobility"] * theta * ny)
        if P["flow"]:
            m["ux"], m["uy"] = self.imposed()
            return m
        rho = P["rho_b"] + phi * (P["rho_a"] - P["rho_b"])
        mu = P["mu_b"] + phi * (P["mu_a"] - P["mu_b"])
        px, py = self._grad(self._window(ps))
        corners = w[1, 1] + w[-1, 1] + w[1, -1] + w[-1, -1]
        axes = w[1, 0] + w[-1, 0] + w[0, 1] + w[0, -1]
        lap = (4 * axes + corners - 20 * phi) / 6
        hxx = sum(k * (w[1, j] - 2 * w[0, j] + w[-1, j]) for j, k in ((-1, 1), (0, 10), (1, 1)))
        hyy = sum(k * (w[i, 1] - 2 * w[i, 0] + w[i, -1]) for i, k in ((-1, 1), (0, 10), (1, 1)))
        hxx, hyy = hxx / 12, hyy / 12
        hxy = (w[1, 1] - w[-1, 1] - w[1, -1] + w[-1, -1]) / 4
        nhn = nx * nx * hxx + 2 * nx * ny * hxy + ny * ny * hyy
        k0 = 1.5 * P["width"]
        if P["sigma_model"]:
            om = 1 - (P["psi0"] + P["gradpsi_x"] * self.x + P["gradpsi_y"] * self.y)
            kt = k0 * P["sigma0"] * (1 + P["beta"] * torch.log(om))
            s = -k0 * P["sigma0"] * P["beta"] / om
            kx, ky = s * P["gradpsi_x"], s * P["gradpsi_y"]
        else:
            kx, ky = k0 * P["dsigma_dT"] * P["gradT_x"], k0 * P["dsigma_dT"] * P["gradT_y"]
            kt = k0 * P["sigma0"] + kx * self.x + ky * self.y
        cap = kt * gm * (nhn - lap)
        nk = nx * kx + ny * ky
        ftx = cap * nx + g2 * (kx - nx * nk) + (rho - P["rho_ref"]) * P["gx"]
        fty = cap * ny + g2 * (ky - ny * nk) + (rho - P["rho_ref"]) * P["gy"]
        third = (P["rho_a"] - P["rho_b"]) / 3
        fpx, fpy = third * dx - px, third * dy - py
        r = self.raw(g)
        ux, uy = 3 * (r[1] + ftx / 6) / rho, 3 * (r[2] + fty / 6) / rho
        m.update(rho=rho, omega=1 / (3 * mu / rho + 0.5), ux=ux, uy=uy, ftx=ftx, fty=fty,
                 fpx=fpx, fpy=fpy, p=ps + 0.5 * (fpx * ux + fpy * uy), r=r)
        return m

    def step(self):
        m = self.macro()
        ux, uy, phi = m["ux"], m["uy"], m["phi"]
        if not self.P["flow"]:
            om, p, rc2 = m["omega"], m["p"], m["rho"] / 3
            psi = p - rc2
            r = m["r"]
            c = self.shifted([p, rc2 * ux, rc2 * uy] + r[3:], ux, uy)
            eq = self._fluid_eq(p, psi, ux, uy)
            trace, dev = eq[3] + eq[4], (1 - om) * (c[3] - c[4]) + om * (eq[3] - eq[4])
            post = [p, c[1], c[2], (trace + dev) / 2, (trace - dev) / 2,
                    (1 - om) * c[5] + om * eq[5], eq[6], eq[7], eq[8]]
            b = self.shifted(post, -ux, -uy)
            ftx, fty, fpx, fpy = m["ftx"], m["fty"], m["fpx"], m["fpy"]
            g00 = fpx * ux + fpy * uy
            sx, sy = ftx + fpx, fty + fpy
            s20, s02 = 2 / 3 * sx * ux + g00 / 3, 2 / 3 * sy * uy + g00 / 3
            s11 = (sx * uy + sy * ux) / 3
            kq = 0.25 * (1 - om) * (s20 - s02)
            new = [m["ps"] + g00, rc2 * ux + ftx / 6, rc2 * uy + fty / 6,
                   b[3] + s20 / 2 + g00 / 3 + kq, b[4] + s02 / 2 + g00 / 3 - kq,
                   b[5] + (1 - om / 2) * s11, b[6] + fty / 9, b[7] + ftx / 9,
                   b[8] + 2 / 9 * g00]
            self.g = self.pops(new).reshape(-1)[self.gather].view_as(self.g)
        om = 1 / (3 * self.P["mobility"] + 0.5)
        c = self.shifted(self.raw(self.f), ux, uy)
        zero = torch.zeros_like(phi)
        post = [phi, c[1] + om * (m["jx"] - c[1]), c[2] + om * (m["jy"] - c[2]), phi / 3, phi / 3,
                zero, zero, zero, phi / 9]
        self.f = (self.pops(self.shifted(post, -ux, -uy)).reshape(-1)[self.gather]
                  .view_as(self.f))
        self.t += 1
        return m

    def fields(self):
        m = self.macro()
        rho = self.P["rho_b"] + m["phi"] * (self.P["rho_a"] - self.P["rho_b"])
        return {"phi": m["phi"], "p": m["p"], "ux": m["ux"], "uy": m["uy"], "rho": rho}


def _tiles(a):
    """[k, ny, nx] as [ny, tiles, k, 32], padding columns 0."""
    k, ny, nx = a.shape
    nt = (nx + 31) // 32
    out = torch.zeros(k, ny, nt * 32, dtype=a.dtype, device=a.device)
    out[:, :, :nx] = a
    return out.view(k, ny, nt, 32).permute(1, 2, 0, 3).contiguous()


def exact(case, seed):
    if case["kind"] == "batch":
        out = {"first": [], "rest": None}
        for c in _drops(case, seed)[:EXACT_CASES]:
            sim = _Exact(c).init(*(torch.from_numpy(c["fields"][k]).cuda()
                                   for k in ("phi", "p", "ux", "uy")))
            for _ in range(case["steps"]):
                sim.step()
            out["first"].append(sim.fields())
        return out
    if case["nx"] * case["ny"] * case["steps"] > 4096 * 4096 * 100:
        return None
    problem, fields = _problem(case, seed)
    sim = _Exact(problem).init(*fields)
    last = None
    for _ in range(case["steps"]):
        last = sim.step()
    if case["kind"] == "session":
        fl = sim.fields()
        speed = torch.hypot(fl["ux"], fl["uy"]).max()
        return {"diagnostics": {"sum_phi": fl["phi"].sum().item(), "sum_p": fl["p"].sum().item(),
                                "max_speed": speed.item(), "dp_laplace": 0.0, "nonfinite": 0},
                "fields": fl}
    if case["precision"] in ("fp16", "bf16"):
        scale = (16384.0, 4096.0) if case["precision"] == "fp16" else (1.0, 1.0)
        w = torch.tensor(WEIGHTS, dtype=torch.float64, device="cuda")[:, None, None]
        d = torch.cat([(sim.g - w * last["ps"]) * scale[0], (sim.f - w * last["phi"]) * scale[1]])
        return {"z": _tiles(torch.stack([last["ps"], last["phi"]])), "d": _tiles(d)}
    if case["setup"] == "shear":
        return {"f": _tiles(sim.f)}
    return {"pops": _tiles(torch.cat([sim.g, sim.f]))}
