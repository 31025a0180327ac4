"""The work that users of this framework have it do, as a list of cases that a timing program can run: solver calls (initialise,
advance, read the fields back) over the range of grids, precisions and sides, a sweep of many cases in one batch, and inference
and gradients of the learned surrogate.

Fields come back as one tensor [4, ny, nx] (rho, u_x, u_y, theta), in float32 from the forms that compute in float32, as the
surrogate's training data are kept.  `exact` is a separate statement of the same time step and network in float64 torch.
"""
import math

import torch

from paper_2002_03644_gb300 import hlbm, surrogate

PER, ZG, DIR, WALL = hlbm.HLBM_BC_PERIODIC, hlbm.HLBM_BC_ZEROGRAD, hlbm.HLBM_BC_DIRICHLET, hlbm.HLBM_BC_WALL
PRECISION = {"fp64": hlbm.HLBM_FP64, "fp32": hlbm.HLBM_FP32, "f16pop": hlbm.HLBM_FP32_F16POP, "bf16pop": hlbm.HLBM_FP32_BF16POP,
             "moments": hlbm.HLBM_FP32_MOMENTS}
# bytes of one cell's state between two steps: 9 populations, s and three a1 components; 7 values in the moment form
CELL_BYTES = {"fp64": 104, "fp32": 52, "f16pop": 34, "bf16pop": 34, "moments": 28}
SIDES = {"periodic": (PER, PER, PER, PER), "open": (ZG, ZG, ZG, ZG), "tube": (ZG, ZG, PER, PER), "channel": (DIR, ZG, ZG, ZG),
         "plates": (PER, PER, WALL, WALL)}
# one cell-update of Algorithm 1 as it is written: moments, entropy update, closure terms, a1 and the collision
CELL_FLOPS = 330
THETA = 300.0 / 1478.75  # sound speed 4/13 at gamma = 1.4


def _case(name, flow, nx, ny, precision, steps, sides="periodic", sigma=0.0, mu=1.5e-6, phi=0):
    return {"name": name, "kind": "solve", "flow": flow, "nx": nx, "ny": ny, "precision": precision, "steps": steps,
            "sides": sides, "sigma": sigma, "mu": mu, "phi": phi}


def listed():
    return [
        # the Sod shock tube at its own resolution, in the precision it is validated in: the smallest calls
        _case("sod_400x4_fp64", "sod", 400, 4, "fp64", 100, sides="tube", mu=3e-6),
        # disturbed thermal Couette flow between plates, run for very many steps: a thin grid with wall sides
        _case("couette_2x100_fp32", "couette", 2, 100, "fp32", 200, sides="plates", sigma=0.9, mu=0.03),
        # one training pair of the surrogate: random smooth field, 16 steps
        _case("fourier_256_fp32", "fourier", 256, 256, "fp32", 16, mu=1e-4),
        # the convected vortex on the grid the method is quoted on, fields out every 100 steps, and its validation in FP64
        _case("vortex_1024_fp32", "vortex", 1024, 1024, "fp32", 100),
        _case("vortex_1024_fp64", "vortex", 1024, 1024, "fp64", 10),
        # the same flow on a grid far larger than the L2 cache
        _case("vortex_4096_fp32", "vortex", 4096, 4096, "fp32", 25),
        # inflow, outflow and free sides on an odd grid, with the blended a1 of flows that need damping
        _case("channel_1501x701_fp32", "fourier", 1501, 701, "fp32", 20, sides="channel", sigma=0.5, mu=1e-3),
        # 16-bit population storage on an open box with the finite-difference heating of discontinuous flows
        _case("open_2048_f16pop", "vortex", 2048, 2048, "f16pop", 20, sides="open", sigma=0.1, mu=1e-4, phi=1),
        # the moment state: the least memory per cell
        _case("vortex_2048_moments", "vortex", 2048, 2048, "moments", 20),
        # a parameter sweep: cases of uneven size, Mach number and gamma advanced together on the tuned work shape
        {"name": "sweep_16_cases", "kind": "sweep", "cases": 16, "steps": 64},
        # the surrogate in a rollout of 16 states, and one gradient step of its training
        {"name": "surrogate_predict_16x256", "kind": "predict", "batch": 16, "n": 256, "width": 64, "hidden": 5},
        {"name": "surrogate_gradient_8x256", "kind": "gradient", "batch": 8, "n": 256, "width": 64, "hidden": 5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve"] * 6 + ["sweep", "predict", "predict", "gradient"])
    if kind == "sweep":
        return {"kind": kind, "cases": rng.randint(3, 16), "steps": rng.randint(9, 64)}
    if kind in ("predict", "gradient"):
        n = rng.choice([64, 96, 128, 128, 192, 256, 256, 256])
        return {"kind": kind, "batch": rng.randint(1, 16 if kind == "predict" else 8), "n": n,
                "width": rng.choice([32, 48, 64, 64, 64]), "hidden": rng.randint(1, 5)}
    precision = rng.choice(["fp64", "fp32", "fp32", "fp32", "f16pop", "bf16pop", "moments"])
    sides = rng.choice(["periodic", "periodic", "periodic", "open", "tube", "channel", "plates"])
    if sides == "plates" and precision == "moments":
        sides = "periodic"  # the moment state has no wall sides
    big = 1024 if precision == "fp64" else 4096
    nx, ny = _log_int(rng, 16, big), _log_int(rng, 16, big)
    updates = (8 if precision == "fp64" else 300) * 1e6
    steps = max(1, min(rng.randint(8, 64), int(updates / (nx * ny))))
    sigma = rng.choice([0.0, 0.0, 0.5, 0.9])
    flow = rng.choice(["fourier", "vortex"]) if min(nx, ny) >= 128 and sides != "plates" else "fourier"
    c = _case("", flow, nx, ny, precision, steps, sides, sigma, rng.choice([1e-5, 1e-4, 1e-3]),
              rng.choice([0, 0, 1]))
    del c["name"]
    return c


# ---- inputs ---------------------------------------------------------------------------------------------------------

def _rand(seed, *shape):
    g = torch.Generator(device="cpu")
    g.manual_seed(int(seed))
    return torch.rand(*shape, generator=g, dtype=torch.float64)


def _vortex(nx, ny, seed, ma, beta, radius, gamma, theta):
    """Isentropic vortex on a mean flow along x, a seeded +-1e-6 perturbation of the density at fixed pressure."""
    x = torch.arange(nx, device="cuda", dtype=torch.float64) + 0.5
    y = (torch.arange(ny, device="cuda", dtype=torch.float64) + 0.5)[:, None]
    c = math.sqrt(gamma * theta / 3.0)
    at = _rand(seed, 2) - 0.5
    dx = (x - nx * (0.5 + 0.2 * float(at[0]))) / radius
    dy = (y - ny * (0.5 + 0.2 * float(at[1]))) / radius
    r2 = dx * dx + dy * dy
    amp = c * beta * ma * torch.exp(0.5 * (1.0 - r2))
    t = 1.0 - 0.5 * (gamma - 1.0) * (beta * ma) ** 2 * torch.exp(1.0 - r2)
    rho = t ** (1.0 / (gamma - 1.0))
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    noisy = rho + 1e-6 * (2.0 * torch.rand(rho.shape, generator=g, device="cuda", dtype=torch.float64) - 1.0)
    return torch.stack([noisy, ma * c - amp * dy, amp * dx, rho * theta * t / noisy])


def _fourier(nx, ny, seed, modes=8, amp=0.05, gamma=1.4):
    """Sums of the lowest Fourier modes on rho, u and theta around a mean flow of random Mach number and direction."""
    modes = max(1, min(modes, nx // 8, ny // 8))
    r = _rand(seed, 4, modes, modes, 2).cuda()
    k = torch.arange(modes, device="cuda", dtype=torch.float64)
    ex = torch.exp(2j * math.pi / nx * k[:, None] * (torch.arange(nx, device="cuda", dtype=torch.float64) + 0.5))
    ey = torch.exp(2j * math.pi / ny * (torch.arange(ny, device="cuda", dtype=torch.float64) + 0.5)[:, None] * k)
    a = (2.0 * r[..., 0] - 1.0) / (1.0 + k[:, None] ** 2 + k ** 2)
    a[:, 0, 0] = 0.0
    f = amp * (ey @ (a * torch.exp(2j * math.pi * r[..., 1])) @ ex).real
    ma, way = _rand(seed + 1, 2).tolist()
    c, way = math.sqrt(gamma * THETA / 3.0) * (0.3 + 0.9 * ma), math.pi * (0.1 + 0.3 * way)
    return torch.stack([1.0 + f[0], c * math.cos(way) + f[1], c * math.sin(way) + f[2], THETA * (1.0 + f[3])])


def _problem(case, seed):
    """(parameters of the solver, initial fields [4, ny, nx]) of a "solve" case."""
    nx, ny = case["nx"], case["ny"]
    r = _rand(seed + 77, 4).tolist()
    bc_state = torch.zeros(4, 4, dtype=torch.float64)
    if case["flow"] == "sod":
        # 1 / 0.125 in density and 1 / 0.1 in pressure, each varied by some per cent; lattice speed 3.875
        left = torch.arange(nx, device="cuda") < nx // 2
        f = torch.zeros(4, ny, nx, device="cuda", dtype=torch.float64)
        t_r = 3.875 ** 2 / 3.0
        f[0] = torch.where(left, 1.0 + 0.05 * r[0], 0.125 * (1.0 + 0.1 * r[1]))
        p = torch.where(left, 1.0 + 0.05 * r[2], 0.1 * (1.0 + 0.1 * r[3]))
        f[3] = p / f[0] / t_r
    elif case["flow"] == "couette":
        # plates at one temperature, the upper one moving at Ma 0.7 to 0.9, a standing wave between them
        th = 0.2 * (1.0 + 0.02 * r[0])
        wall = (0.7 + 0.2 * r[1]) * math.sqrt(1.4 * th / 3.0)
        y = ((torch.arange(ny, device="cuda", dtype=torch.float64) + 0.5) / ny)[:, None].expand(ny, nx)
        f = torch.stack([1.0 + 0.02 * torch.cos(math.pi * y), wall * y, 0.02 * (1.0 + r[2]) * torch.sin(math.pi * y), th + 0.0 * y])
        bc_state[2] = torch.tensor([1.0, 0.0, 0.0, th])
        bc_state[3] = torch.tensor([1.0, wall, 0.0, th])
    elif case["flow"] == "vortex":
        f = _vortex(nx, ny, seed, 1.2, 0.2, max(4.0, min(nx, ny) / 32.0), 1.4, THETA)
    else:
        f = _fourier(nx, ny, seed)
    if case["sides"] == "plates" and case["flow"] != "couette":
        f[2] -= f[2].mean()  # no flow through the plates
        bc_state[2] = torch.tensor([1.0, 0.02, 0.0, THETA])
        bc_state[3] = torch.tensor([1.0, 0.3, 0.0, THETA])
    if case["sides"] == "channel":
        bc_state[0] = f.mean(dim=(1, 2)).cpu()  # the mean state flows in
    p = {"gamma": 1.4, "Pr": 0.71, "mu": case["mu"], "sigma": case["sigma"], "phi_mode": case["phi"], "bc": SIDES[case["sides"]],
         "bc_state": bc_state.tolist()}
    return p, f.contiguous()


def _sweep(case, seed):
    """Vortices on grids of 128^2 to 1024^2, Mach 0.1 to 1.5, three gammas, every one at CFL number 0.7."""
    out = []
    sizes = (1024, 256, 512, 128)
    r = _rand(seed, case["cases"], 2).tolist()
    for k in range(case["cases"]):
        n, ma, gamma = sizes[(3 * k + k // 4) % 4], 0.1 + 1.4 * r[k][0], (1.4, 1.3, 1.67)[int(3 * r[k][1]) % 3]
        theta = 3.0 * (0.7 / (ma + 1.0)) ** 2 / gamma
        p = {"gamma": gamma, "Pr": 0.71, "mu": 1.5e-6, "sigma": 0.0, "phi_mode": 0, "bc": SIDES["periodic"],
             "bc_state": torch.zeros(4, 4).tolist()}
        out.append((p, _vortex(n, n, seed * 64 + k, ma, 0.2, n / 32.0, gamma, theta).contiguous()))
    return out


def _net(case, seed):
    """(channel counts, parameters, input, target): normalised smooth states and the same a few cells downstream."""
    widths = (4,) + (case["width"],) * case["hidden"] + (4,)
    b, n = case["batch"], case["n"]
    x = torch.stack([_fourier(n, n, 16 * seed + k).permute(1, 2, 0) for k in range(b)])
    x = (x - x.mean(dim=(0, 1, 2))) / x.std(dim=(0, 1, 2))
    x = x.float().contiguous()
    t = torch.roll(x, (2, 3), (1, 2)).contiguous()
    return widths, surrogate.init_params(widths, seed=seed), x, t


def prepare(case, seed):
    if case["kind"] == "solve":
        p, f = _problem(case, seed)
        s = hlbm.Solver(case["nx"], case["ny"], stream=hlbm.torch_stream_handle(), precision=PRECISION[case["precision"]], **p)
        return {"case": case, "solver": s, "in": f, "out": torch.empty_like(f)}
    if case["kind"] == "sweep":
        probs = _sweep(case, seed)
        stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        b = hlbm.Batch([dict(nx=f.shape[2], ny=f.shape[1], precision=hlbm.HLBM_FP32, **p) for p, f in probs], stream=stream.cuda_stream)
        for s, (_, f) in zip(b.cases, probs):
            s.init(*f)
        b.autotune()
        return {"case": case, "batch": b, "in": [f for _, f in probs], "out": [torch.empty_like(f) for _, f in probs], "stream": stream}
    widths, params, x, t = _net(case, seed)
    n = case["n"]
    net = surrogate.Surrogate(widths, n, n, batch_max=case["batch"])
    net.set_params(params)
    return {"case": case, "net": net, "x": x, "t": t, "grads": torch.empty(net.nparam, device="cuda")}


def run(state):
    case = state["case"]
    if case["kind"] == "solve":
        s, out = state["solver"], state["out"]
        s.init(*state["in"])
        s.step(case["steps"])
        hlbm.hlbm_get_macros(s.h, *out)
        return out if case["precision"] == "fp64" else out.float()
    if case["kind"] == "sweep":
        b = state["batch"]
        for s, f in zip(b.cases, state["in"]):
            s.init(*f)
        b.step(case["steps"])
        with torch.cuda.stream(state["stream"]):
            got = []
            for s, out in zip(b.cases, state["out"]):
                hlbm.hlbm_get_macros(s.h, *out)
                got.append(out.float())
        return got
    net = state["net"]
    if case["kind"] == "predict":
        return net.predict(state["x"])
    loss = net.rollout_grads(state["x"], [state["t"]])
    hlbm.hlbm_sur_get_params(net.s, grads=state["grads"])
    return {"loss": loss, "grads": state["grads"]}


def work(case):
    """Every step reads and writes the state once, the fields come in and go out once in float64; a network reads its input and
    weights and writes its output or gradients, with 16-bit activations between its layers."""
    if case["kind"] in ("predict", "gradient"):
        c = [4] + [case["width"]] * case["hidden"] + [4]
        pix = case["batch"] * case["n"] ** 2
        macs = sum(9 * a * b for a, b in zip(c, c[1:]))
        between = sum(c[1:-1])
        if case["kind"] == "predict":
            return {"bytes": pix * (32 + 4 * between), "flops": 2 * macs * pix}
        # forward, input gradient (not of the first layer) and weight gradient
        return {"bytes": pix * (48 + 16 * between), "flops": 2 * pix * (3 * macs - 9 * c[0] * c[1])}
    if case["kind"] == "sweep":
        sizes = (1024, 256, 512, 128)
        cells = sum(sizes[(3 * k + k // 4) % 4] ** 2 for k in range(case["cases"]))
        state = CELL_BYTES["fp32"]
    else:
        cells, state = case["nx"] * case["ny"], CELL_BYTES[case["precision"]]
    return {"bytes": cells * (64 + 2 * state * case["steps"]), "flops": cells * CELL_FLOPS * case["steps"]}


# ---- the same in float64 torch ----------------------------------------------------------------------------------------

CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)


def _moments(f):
    # mirror directions in pairs: a symmetric set has no momentum at all
    rho = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])) + f[8]
    jx = (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7])
    jy = (f[2] - f[4]) + (f[5] - f[8]) + (f[6] - f[7])
    return rho, jx / rho, jy / rho


class _Exact:
    """Algorithm 1 with hybrid recursive regularised collision, upwind closure correction, polyatomic correction and the
    entropy update, on float64 tensors [ny, nx]."""

    def __init__(self, p, fields):
        self.p = p
        self.ny, self.nx = fields.shape[1:]
        self.gm1 = p["gamma"] - 1.0
        self.cv = 1.0 / 3.0 / self.gm1
        self.lam = p["mu"] * p["gamma"] * self.cv / p["Pr"]
        rho, u, v, th = fields
        self.s = self.entropy(rho, th)
        n1 = [self.pad(q, 1, k) for k, q in zip(("rho", "u", "v", "th"), (rho, u, v, th))]
        if WALL in p["bc"]:
            n1 = self.wall_macros(n1, 1)
        self.finish(*n1, None)

    def entropy(self, rho, th):
        return self.cv * (torch.log(th) - self.gm1 * torch.log(rho))

    def theta(self, rho, s):
        return torch.exp(self.gm1 * torch.log(rho) + s / self.cv)

    def side(self, k, what):
        rho, u, v, th = (torch.tensor(x, dtype=torch.float64, device="cuda") for x in self.p["bc_state"][k])
        if what == "s":
            return self.entropy(rho, th)
        if what[0] == "F":
            z = torch.zeros_like(rho)
            return self.populations(rho, u, v, th, z, z, z, z, z, z)[int(what[1])]
        return {"rho": rho, "u": u, "v": v, "th": th}[what]

    def pad(self, q, h, what):
        """`q` with h more cells on every side: wrapped, the edge cell's, or the imposed state (a y side wins at a corner); wall
        sides get the edge cell here and their own values later."""
        def index(n, lo, hi):
            i = torch.arange(-h, n + h, device="cuda")
            return i % n if lo == PER else i.clamp(0, n - 1)
        bc = self.p["bc"]
        q = q[index(self.ny, bc[2], bc[3])][:, index(self.nx, bc[0], bc[1])]
        for k, cut in ((0, (slice(None), slice(0, h))), (1, (slice(None), slice(-h, None))), (2, slice(0, h)), (3, slice(-h, None))):
            if bc[k] == DIR:
                q[cut] = self.side(k, what)
        return q

    def ghosts(self, h):
        """(ghost row, mirrored row, wall) of the wall sides' first h layers, in rows of an array padded by h."""
        for k, first, step in ((2, h - 1, -1), (3, self.ny + h, 1)):
            if self.p["bc"][k] == WALL:
                for g in range(h):
                    yield first + step * g, first - step * (g + 1), k

    def wall_macros(self, n1, h):
        """Ghost layers of a wall: velocity and temperature mirrored about the wall's, at the mirrored cell's pressure."""
        rho, u, v, th = n1
        for at, of, k in self.ghosts(h):
            _, uw, vw, tw = self.p["bc_state"][k]
            th[at] = 2.0 * tw - th[of]
            rho[at] = rho[of] * th[of] / th[at]
            u[at], v[at] = 2.0 * uw - u[of], 2.0 * vw - v[of]
        return rho, u, v, th

    def populations(self, rho, u, v, th, axx, axy, ayy, ex, ey, om):
        """f^eq + om f1 + psi / 2 from raw moments, the lattice taken as the product of two three-velocity ones."""
        mx, my = u * u + th / 3.0, v * v + th / 3.0
        axxy, ayyx = v * axx + 2.0 * u * axy, u * ayy + 2.0 * v * axy
        d = (th - 1.0) / 3.0
        axxyy = 2.0 * (u * ayyx + v * axxy) + (d - u * u) * ayy + (d - v * v) * axx - 4.0 * u * v * axy
        r = {(0, 0): rho, (1, 0): rho * u, (0, 1): rho * v, (1, 1): rho * u * v + om * axy,
             (2, 0): rho * mx + om * axx + 0.5 * ex, (0, 2): rho * my + om * ayy + 0.5 * ey,
             (2, 1): rho * mx * v + om * axxy, (1, 2): rho * u * my + om * ayyx,
             (2, 2): rho * mx * my + om * (axxyy + (axx + ayy) / 3.0) + (ex + ey) / 6.0}
        along = {(c, b): r[0, b] - r[2, b] if c == 0 else 0.5 * (r[2, b] + c * r[1, b]) for c in (-1, 0, 1) for b in (0, 1, 2)}
        return [along[c, 0] - along[c, 2] if e == 0 else 0.5 * (along[c, 2] + e * along[c, 1]) for c, e in zip(CX, CY)]

    def finish(self, rho, u, v, th, second):
        """psi, a1 and the next collision from the level's macros, padded by one."""
        mu, g = self.p["mu"], self.p["gamma"]
        C, W, E = (slice(1, -1), slice(1, -1)), (slice(1, -1), slice(0, -2)), (slice(1, -1), slice(2, None))
        S, N = (slice(0, -2), slice(1, -1)), (slice(2, None), slice(1, -1))
        uc, vc = u[C], v[C]
        dxu, dyu, dxv, dyv = (0.5 * (q[b] - q[a]) for q, a, b in ((u, W, E), (u, S, N), (v, W, E), (v, S, N)))

        def upwind(vel, gam, a, b):
            back, fore = gam[C] - gam[a], gam[b] - gam[C]
            return torch.where(vel > 0, back, torch.where(vel < 0, fore, 0.5 * (gam[b] - gam[a])))

        p = rho[C] * th[C] / 3.0
        e2 = p * (2.0 - g) * (dxu + dyv)
        ex = upwind(uc, rho * u * (1.0 - th - u * u), W, E) + e2
        ey = upwind(vc, rho * v * (1.0 - th - v * v), S, N) + e2
        tau_p = mu + 0.5 * p
        axx, axy = -tau_p * (dxu - dyv), -tau_p * (dyu + dxv)
        ayy = -axx
        if second is not None and self.p["sigma"] > 0.0:
            w = self.p["sigma"]
            mxx, mxy, myy = second
            axx = w * (mxx - rho[C] * uc * uc - p + 0.5 * ex) + (1.0 - w) * axx
            ayy = w * (myy - rho[C] * vc * vc - p + 0.5 * ey) + (1.0 - w) * ayy
            axy = w * (mxy - rho[C] * uc * vc) + (1.0 - w) * axy
        om = (2.0 * mu - p) / (2.0 * mu + p)
        self.F = self.populations(rho[C], uc, vc, th[C], axx, axy, ayy, ex, ey, om)
        self.a = (axx, axy, ayy)

    def advect(self, vel, q, dim):
        """u ds/dx with Van Albada limited, upwinded face values; q is padded by two."""
        def at(k):
            return q[2 + k:self.ny + 2 + k, 2:-2] if dim == 0 else q[2:-2, 2 + k:self.nx + 2 + k]

        def slope(a, b):
            return torch.where(a * b > 0, a * b * (a + b) / torch.where(a * b > 0, a * a + b * b, torch.ones_like(a)), torch.zeros_like(a))

        d = [at(k + 1) - at(k) for k in (-2, -1, 0, 1)]
        s0 = slope(d[1], d[2])
        back = d[1] + 0.5 * (s0 - slope(d[0], d[1]))
        fore = d[2] + 0.5 * (s0 - slope(d[2], d[3]))
        return vel * torch.where(vel > 0, back, fore)

    def step(self):
        mu = self.p["mu"]
        rho, u, v = _moments(self.F)
        th = self.theta(rho, self.s)
        F = [self.pad(f, 1, "F%d" % i) for i, f in enumerate(self.F)]
        sp = self.pad(self.s, 2, "s")
        n0 = [self.pad(q, 2, k) for k, q in zip(("rho", "u", "v", "th"), (rho, u, v, th))]
        if WALL in self.p["bc"]:
            n0 = self.wall_macros(n0, 2)
            for at, of, k in self.ghosts(2):
                sp[at] = self.entropy(n0[0][at], n0[3][at])
            a = [self.pad(q, 1, "a") for q in self.a]
            z = torch.zeros_like(a[0][0])
            for at, of, k in self.ghosts(1):
                r, uu, vv, tt = (q[at + 1, 1:-1] for q in n0)
                p = r * tt / 3.0
                om = (2.0 * mu - p) / (2.0 * mu + p)
                for f, g in zip(F, self.populations(r, uu, vv, tt, a[0][of], a[1][of], a[2][of], z, z, om)):
                    f[at] = g
        up, vp, tp = (q[1:-1, 1:-1] for q in n0[1:])
        W, E, S, N = (slice(1, -1), slice(0, -2)), (slice(1, -1), slice(2, None)), (slice(0, -2), slice(1, -1)), (slice(2, None), slice(1, -1))
        dxu, dyu, dxv, dyv = (0.5 * (q[b] - q[a]) for q, a, b in ((up, W, E), (up, S, N), (vp, W, E), (vp, S, N)))
        lap = tp[W] + tp[E] + tp[S] + tp[N] - 4.0 * th
        if self.p["phi_mode"] == 0:
            axx, axy, ayy = self.a
            phi = -2.0 * mu / (2.0 * mu + rho * th / 3.0) * (axx * dxu + axy * (dyu + dxv) + ayy * dyv)
        else:
            phi = mu * ((dxu - dyv) ** 2 + (dyu + dxv) ** 2)
        self.s = self.s - self.advect(u, sp, 1) - self.advect(v, sp, 0) + (self.lam * lap + phi) / (rho * th)
        g = [F[i][1 - CY[i]:self.ny + 1 - CY[i], 1 - CX[i]:self.nx + 1 - CX[i]] for i in range(9)]
        rho, u, v = _moments(g)
        th = self.theta(rho, self.s)
        diag = (g[5] + g[6]) + (g[7] + g[8])
        second = (g[1] + g[3] + diag, (g[5] - g[6]) + (g[7] - g[8]), g[2] + g[4] + diag)
        n1 = [self.pad(q, 1, k) for k, q in zip(("rho", "u", "v", "th"), (rho, u, v, th))]
        if WALL in self.p["bc"]:
            n1 = self.wall_macros(n1, 1)
        self.finish(*n1, second)

    def fields(self):
        rho, u, v = _moments(self.F)
        return torch.stack([rho, u, v, self.theta(rho, self.s)])


def _exact_solve(p, fields, steps):
    e = _Exact(p, fields)
    for _ in range(steps):
        e.step()
    return e.fields()


def exact(case, seed):
    if case["kind"] == "solve":
        return _exact_solve(*_problem(case, seed), case["steps"])
    if case["kind"] == "sweep":
        return [_exact_solve(p, f, case["steps"]) for p, f in _sweep(case, seed)]
    widths, params, x, t = _net(case, seed)
    theta = torch.from_numpy(params).cuda().double().requires_grad_(case["kind"] == "gradient")
    x64, t64 = x.double().permute(0, 3, 1, 2), t.double().permute(0, 3, 1, 2)

    def net(x):
        h, at = x, 0
        for l, (a, b) in enumerate(zip(widths, widths[1:])):
            w = theta[at:at + a * b * 9].view(b, a, 3, 3)
            bias = theta[at + a * b * 9:at + a * b * 9 + b]
            at += a * b * 9 + b
            h = torch.nn.functional.pad(h, (1, 1, 1, 1), mode="circular")
            # nine products of matrices: the convolution without a convolution routine's choice of algorithm
            n, m = h.shape[2] - 2, h.shape[3] - 2
            h = sum(torch.einsum("oc,bcij->boij", w[:, :, i, j], h[:, :, i:i + n, j:j + m]) for i in range(3) for j in range(3))
            h = h + bias[:, None, None]
            if l < len(widths) - 2:
                h = 0.5 * h * (1.0 + torch.erf(h / math.sqrt(2.0)))
        return x + h

    if case["kind"] == "predict":
        with torch.no_grad():
            return torch.cat([net(x64[k:k + 1]) for k in range(case["batch"])]).permute(0, 2, 3, 1)
    total = 0.0
    for k in range(case["batch"]):
        loss = ((net(x64[k:k + 1]) - t64[k:k + 1]) ** 2).mean() / case["batch"]
        loss.backward()
        total += float(loss.detach())
    return {"loss": total, "grads": theta.grad}
