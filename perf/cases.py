"""Timed cases of the framework: what a two-phase flow program has it do, step after step.

A time step hands over a moved level set, and then either projects a face velocity
(`project`: set_geometry + project_step) or solves for the pressure of its own right-hand
side (`pressure`: set_geometry + solve).  The learned initial guess adds the 3x3x3
convolution layers of its network: the layer (`conv`) and the weight gradient that
training it takes (`wgrad`).  Everything goes through the package's public entry points.

A solve's stopping point moves with rounding, and its velocity with it, so the cases solve
to a relative residual of 1e-13, at which pressure and velocity are fixed by the inputs.
"""
import math
import random

import torch

import paper_2312_11740_gb300 as mp
from paper_2312_11740_gb300 import Net, Poisson, mp_conv3d_fwd, mp_conv3d_wgrad, mp_poisson_set_net

DEVICE = "cuda"
RHO_L, RHO_G = 1.0, 1e-3  # liquid and gas density (air and water)
EVAPORATION = 1e-3        # mass flux: gas leaves the interface about as fast as the flow moves

# boundary letters per axis: p periodic, w walls, t wall or inflow below and outflow above,
# d outflow on both sides
BC = {"p": mp.poisson.PERIODIC, "w": mp.poisson.NEUMANN, "t": mp.poisson.NEUMANN_DIRICHLET,
      "d": mp.poisson.DIRICHLET}


def _flow(name, kind, nx, ny, nz, bubbles, pool, bc, sigma, precision, guess, evaporate, tol):
    case = dict(kind=kind, nx=nx, ny=ny, nz=nz, bubbles=bubbles, pool=pool, bc=bc, sigma=sigma,
                precision=precision, guess=guess, evaporate=evaporate, tol=tol)
    return dict(case, name=name) if name else case


def _layer(name, kind, nx, ny, nz, ca, cb, cout, up):
    case = dict(kind=kind, nx=nx, ny=ny, nz=nz, ca=ca, cb=cb, cout=cout, up=up)
    return dict(case, name=name) if name else case


def listed():
    return [
        # one bubble on a small grid, a quick look or one block of a parameter study: launches
        # and host round trips count
        _flow("project 32^3 bubble", "project", 32, 32, 32, 1, False, "ppw", 0.01, "mixed", "zero",
              False, 1e-13),
        # small ragged box in full FP64
        _flow("project 40x24x56 fp64", "project", 40, 24, 56, 2, False, "ppw", 0.01, "fp64", "zero",
              False, 1e-13),
        # time stepping at a middle size: the previous step's pressure is the start
        _flow("project 128^3 previous", "project", 128, 128, 128, 16, True, "ppw", 0.01, "mixed",
              "previous", False, 1e-13),
        # the benchmark's pool with 32 bubbles, one whole projection step; the paper's example
        # surface tension
        _flow("project 256^3 pool", "project", 256, 256, 256, 32, True, "ppw", 0.004, "mixed",
              "zero", False, 1e-13),
        # one bubble, FP64 throughout
        _flow("pressure 256^3 fp64", "pressure", 256, 256, 256, 1, False, "ppw", 0.07, "fp64",
              "zero", False, 1e-13),
        # the largest production grid of the benchmark's configurations
        _flow("pressure 512^3 bubbles", "pressure", 512, 512, 512, 64, False, "ppw", 0.07, "mixed",
              "zero", False, 1e-13),
        # evaporating bubbles under an outflow top, a box that halves to 10 x 5 x 6 cells
        _flow("pressure 160x80x96 outflow", "pressure", 160, 80, 96, 4, True, "pwt", 0.05, "mixed",
              "zero", True, 1e-13),
        # channel with outflow at both ends, FP64
        _flow("pressure 96x64x48 channel fp64", "pressure", 96, 64, 48, 3, False, "dwp", 0.05,
              "fp64", "zero", False, 1e-13),
        # the benchmark's learned form: the packaged network's guess on the half-resolution grid
        _flow("pressure 256^3 learned", "pressure", 256, 256, 256, 32, True, "ppw", 0.07, "mixed",
              "learned", False, 1e-13),
        # the network's finest encoder layer, its most frequent shape
        _layer("conv 16-16 128^3", "conv", 128, 128, 128, 16, 0, 16, False),
        # a decoder layer: upsampled coarse features beside the encoder's
        _layer("conv up 64+32-32 64^3", "conv", 64, 64, 64, 64, 32, 32, True),
        # the weight gradient of a middle layer
        _layer("wgrad 32-32 64^3", "wgrad", 64, 64, 64, 32, 0, 32, False),
    ]


def draw(rng):
    kind = rng.choice(["project", "project", "pressure", "pressure", "pressure", "learned", "conv",
                       "wgrad"])
    if kind in ("conv", "wgrad"):
        up = rng.random() < 0.4
        while True:  # grids from the coarsest level of a small network to its finest
            s = 2 ** rng.uniform(0, 3.6)
            nx, ny, nz = (max(16, 8 * round(rng.uniform(1, 3) * s)) for _ in range(3))
            ny, nz = max(8, ny - rng.choice([0, 4, 0])), max(8, nz - rng.choice([0, 4, 0]))
            if up:  # the half grid has the layer's own tile sizes
                nx, ny, nz = -(-nx // 16) * 16, -(-ny // 8) * 8, -(-nz // 8) * 8
            if nx * ny * nz <= 2 ** 21:
                break
        ca = rng.choice([32, 64]) if up else rng.choice([16, 32, 64])
        cb = rng.choice([16, 32, 64]) if up else 0
        return _layer(None, kind, nx, ny, nz, ca, cb, rng.choice([16, 32, 64]), up)
    if kind == "learned":
        while True:
            f = rng.choice([32, 64])
            nx, ny, nz = (f * rng.randint(1, 256 // f) for _ in range(3))
            if nx * ny * nz <= 2 ** 23:
                break
        return _flow(None, "pressure", nx, ny, nz, rng.randint(1, 24), rng.random() < 0.5, "ppw",
                     round(rng.uniform(0.02, 0.08), 3), "mixed", "learned", False, 1e-13)
    precision = rng.choice(["mixed", "mixed", "fp64"])
    cap = 4e7 if precision == "mixed" else 6e6
    while True:  # 2^f times a small odd or even box
        f = 2 ** rng.randint(2, 6)
        nx, ny, nz = (f * rng.randint(3, 8) for _ in range(3))
        if nx * ny * nz <= cap:
            break
    bubbles = round(2 ** rng.uniform(0, 5.3))
    if kind == "project":
        return _flow(None, kind, nx, ny, nz, bubbles, rng.random() < 0.5,
                     rng.choice(["ppw", "ppp", "pww", "www"]), round(rng.uniform(0.002, 0.012), 4),
                     precision,
                     rng.choice(["zero", "previous"]), False, 1e-13)
    bc = rng.choice(["ppw", "ppw", "pww", "pwt", "ppt", "dwp"])
    evaporate = rng.random() < 0.4
    return _flow(None, kind, nx, ny, nz, bubbles, rng.random() < 0.5 and bc != "dwp", bc,
                 round(rng.uniform(0.01, 0.08), 3), precision, "zero", evaporate, 1e-13)


# ------------------------------------------------------------------ inputs
def _place(rng, case):
    """Non-overlapping spheres in the box (lengths in units of its longest side), below the
    pool's surface where there is one; smaller ones after many misses."""
    n = (case["nx"], case["ny"], case["nz"])
    h = 1.0 / max(n)
    box = [h * m for m in n]
    top = box[2] * (0.6 if case["pool"] else 1.0)
    small = min(box[0], box[1], top)
    r_hi, out, misses = 0.25 * small, [], 0
    if case["bubbles"] > 1:
        r_hi = min(r_hi, max(0.02, 0.6 * (box[0] * box[1] * top / case["bubbles"]) ** (1 / 3) / 2))
    r_lo = max(0.4 * r_hi, min(r_hi, 3 * h))
    while len(out) < case["bubbles"] and misses < 2000:
        r = rng.uniform(r_lo, r_hi)
        c = []
        for a in range(3):
            lo, hi = (0.0, box[a]) if case["bc"][a] == "p" else (r + 2 * h, box[a] - r - 2 * h)
            if a == 2 and case["pool"]:
                lo, hi = r + 2 * h, top - r - 3 * h
            c.append(rng.uniform(lo, max(lo, hi)))
        clear = True
        for other, q in out:
            d = [abs(x - y) for x, y in zip(c, other)]
            d = [min(x, box[a] - x) if case["bc"][a] == "p" else x for a, x in enumerate(d)]
            clear = clear and math.dist(d, (0, 0, 0)) > r + q + 4 * h
        if clear:
            out.append((c, r))
        else:
            misses += 1
            r_lo, r_hi = max(3 * h, 0.999 * r_lo), max(3 * h, 0.999 * r_hi)
    return out, (top if case["pool"] else None), h, box


def _axes(case, h, at=(0.5, 0.5, 0.5)):
    """x, y, z coordinates as broadcastable tensors; `at`: offsets in cells."""
    return [((torch.arange(n, dtype=torch.float64, device=DEVICE) + o) * h).view(s)
            for n, o, s in zip((case["nx"], case["ny"], case["nz"]), at,
                               ((1, 1, -1), (1, -1, 1), (-1, 1, 1)))]


def _level_set(case, spheres, top, h, box):
    """Gas-positive signed distance of the spheres and the gas above the pool."""
    xyz = _axes(case, h)
    phi = torch.full((case["nz"], case["ny"], case["nx"]), -math.inf, dtype=torch.float64,
                     device=DEVICE)
    if top is not None:
        phi = torch.maximum(phi, xyz[2] - top)
    for c, r in spheres:
        d2 = 0.0
        for a in range(3):
            d = xyz[a] - c[a]
            if case["bc"][a] == "p":
                d = d - box[a] * torch.round(d / box[a])
            d2 = d2 + d * d
        phi = torch.maximum(phi, r - torch.sqrt(d2))
    return phi.contiguous()


def _smooth(rng, case, h, box, at, modes=16):
    """Sum of 16 Fourier modes of up to four waves per axis, at most 1 in size."""
    xyz = _axes(case, h, at)
    u = 0.0
    for _ in range(modes):
        k = [rng.randint(-4, 4) for _ in range(3)]
        ph = [2 * math.pi * k[a] / box[a] * xyz[a] for a in range(3)]
        ph[2] = ph[2] + rng.uniform(0, 2 * math.pi)
        yz = ph[1] + ph[2]
        u = u + rng.gauss(0, 1) * (torch.cos(yz) * torch.cos(ph[0]) -
                                   torch.sin(yz) * torch.sin(ph[0]))
    return (u / u.abs().max()).contiguous()


def _velocity(rng, case, h, box):
    """Face velocity (low-face owned), zero on the wall faces."""
    u = [_smooth(rng, case, h, box, at)
         for at in ((0.0, 0.5, 0.5), (0.5, 0.0, 0.5), (0.5, 0.5, 0.0))]
    for a in range(3):
        if case["bc"][a] != "p":
            u[a].select(2 - a, 0).zero_()
    return u


def _flow_inputs(case, seed):
    rng = random.Random(seed * 7919 + 17)
    spheres, top, h, box = _place(rng, case)
    d = dict(case=case, h=h, bc=tuple(BC[c] for c in case["bc"]),
             phi=_level_set(case, spheres, top, h, box), mdot=None)
    if case["evaporate"]:
        x, y, z = _axes(case, h)
        d["mdot"] = (EVAPORATION * (1.0 + x + 0.5 * y * z)).contiguous()
    if case["kind"] == "project":
        d["u"] = _velocity(rng, case, h, box)
        if case["guess"] == "previous":  # last step's velocity differed by 5 %
            d["u_before"] = [a - 0.05 * b for a, b in zip(d["u"], _velocity(rng, case, h, box))]
    else:
        d["rhs"] = 20.0 * _smooth(rng, case, h, box, (0.5, 0.5, 0.5))
    return d


def _layer_inputs(case, seed):
    """Activations after a ReLU, weights at their usual initial scale, BF16."""
    g = torch.Generator(device=DEVICE).manual_seed(seed)
    rand = lambda *s: torch.randn(s, generator=g, device=DEVICE)  # noqa: E731
    shape = (case["nz"], case["ny"], case["nx"])
    half = tuple(n // 2 for n in shape) if case["up"] else shape
    cin = case["ca"] + case["cb"]
    d = dict(case=case, xa=rand(*half, case["ca"]).relu().bfloat16(), xb=None)
    if case["cb"]:
        d["xb"] = rand(*shape, case["cb"]).relu().bfloat16()
    if case["kind"] == "conv":
        d["w"] = (rand(case["cout"], 27, cin) * math.sqrt(2.0 / (27 * cin))).bfloat16()
        d["bias"] = 0.1 * rand(case["cout"])
    else:
        d["g"] = (1e-2 * rand(*shape, case["cout"])).bfloat16()
    return d


def prepare(case, seed):
    if case["kind"] in ("conv", "wgrad"):
        return _layer_inputs(case, seed)
    d = _flow_inputs(case, seed)
    guess = {"zero": 0, "previous": 1, "learned": 2}[case["guess"]]
    d["solver"] = Poisson(d["phi"], d["h"], d["bc"], RHO_L, RHO_G, case["sigma"],
                          precision=1 if case["precision"] == "mixed" else 0)
    if d["mdot"] is not None:
        d["solver"].set_mass_flux(d["mdot"])
    if guess == 1:
        d["p"] = torch.zeros_like(d["phi"])
        d["solver"].project_step(*[c.clone() for c in d["u_before"]], d["p"], tol=case["tol"])
    if guess == 2:
        n = (case["nx"], case["ny"], case["nz"])
        f = 2 if max(n) > 128 and all(m % 64 == 0 for m in n) else 1
        d["net"] = Net(*[m // f for m in n])
        d["net"].load()
        mp_poisson_set_net(d["solver"].handle, d["net"])
    d["solver"].set_opts(initial_guess=guess)
    return d


def run(state):
    case = state["case"]
    if case["kind"] == "conv":
        return mp_conv3d_fwd(state["xa"], state["w"], case["cout"], xb=state["xb"],
                             bias=state["bias"], up_a=case["up"], relu=True)
    if case["kind"] == "wgrad":
        return mp_conv3d_wgrad(state["xa"], state["g"], xb=state["xb"], up_a=case["up"])
    solver = state["solver"]
    solver.set_geometry(state["phi"], RHO_L, RHO_G, case["sigma"])
    p = state["p"].clone() if "p" in state else torch.zeros_like(state["phi"])
    if case["kind"] == "pressure":
        return solver.solve(state["rhs"], p=p, tol=case["tol"])[0]
    u = [c.clone() for c in state["u"]]
    solver.project_step(*u, p, tol=case["tol"])
    return dict(ux=u[0], uy=u[1], uz=u[2], p=p)


def work(case):
    n = case["nx"] * case["ny"] * case["nz"]
    if case["kind"] in ("conv", "wgrad"):
        cin = case["ca"] + case["cb"]
        inputs = 2 * (n * case["ca"] / (8 if case["up"] else 1) + n * case["cb"])
        weights = 27 * cin * case["cout"] * (2 if case["kind"] == "conv" else 4)
        return {"bytes": inputs + 2 * n * case["cout"] + weights,
                "flops": 2.0 * 27 * cin * case["cout"] * n}
    # level set and velocity (or right-hand side) in, velocity and pressure (or pressure) out
    arrays = (8 if case["kind"] == "project" else 3) + (1 if case["evaporate"] else 0)
    return {"bytes": 8.0 * arrays * n, "flops": 0.0}


# ------------------------------------------- the same in plain torch, 64 bits
def _lo(a, axis):
    return torch.roll(a, 1, 2 - axis)


def _hi(a, axis):
    return torch.roll(a, -1, 2 - axis)


def _ghost(a, axis, step, periodic):
    """The neighbour along an axis; at a wall the cell itself."""
    out = torch.roll(a, -step, 2 - axis)
    if not periodic:
        edge = -1 if step > 0 else 0
        out.select(2 - axis, edge).copy_(a.select(2 - axis, edge))
    return out


def _curvature(phi, h, per):
    def nb(a, axis, step):
        return _ghost(a, axis, step, per[axis])
    lo, hi = [nb(phi, a, -1) for a in range(3)], [nb(phi, a, 1) for a in range(3)]
    g = [(hi[a] - lo[a]) / (2 * h) for a in range(3)]
    gg = [(hi[a] - 2 * phi + lo[a]) / (h * h) for a in range(3)]

    def mixed(a, b):
        return (nb(hi[a], b, 1) - nb(hi[a], b, -1) - nb(lo[a], b, 1) + nb(lo[a], b, -1)) / (4 * h * h)
    size = torch.sqrt(g[0] ** 2 + g[1] ** 2 + g[2] ** 2).clamp(min=1e-12)
    num = (g[0] ** 2 * (gg[1] + gg[2]) + g[1] ** 2 * (gg[0] + gg[2]) + g[2] ** 2 * (gg[0] + gg[1]) -
           2 * (g[0] * g[1] * mixed(0, 1) + g[0] * g[2] * mixed(0, 2) + g[1] * g[2] * mixed(1, 2)))
    return (-num / size ** 3).clamp(-1 / h, 1 / h)


def _system(d):
    """Ghost-fluid faces, pressure jumps and source of the case's level set."""
    case, phi, h = d["case"], d["phi"], d["h"]
    per = [c == "p" for c in case["bc"]]
    gas = phi > 0
    rho = torch.where(gas, RHO_G, RHO_L).to(torch.float64)
    kap = _curvature(phi, h, per)
    beta, jump, source = [], [], torch.zeros_like(phi)
    dd = torch.zeros_like(phi)  # outflow faces
    share = torch.zeros_like(phi)
    for a in range(3):
        pl, gl, kl, rl = _lo(phi, a), _lo(gas, a), _lo(kap, a), _lo(rho, a)
        cross = gl != gas
        wl = pl.abs() / (pl.abs() + phi.abs())  # fraction of the segment in the low cell's fluid
        b = torch.where(cross, 1 / (wl * rl + (1 - wl) * rho), 1 / rho)
        if not per[a]:
            b.select(2 - a, 0).zero_()
            letter = case["bc"][a]
            for side, there in ((0, letter == "d"), (-1, letter in "dt")):
                if there:
                    dd.select(2 - a, side).add_(2 / rho.select(2 - a, side))
        kg = (1 - wl) * kl + wl * kap
        j = torch.where(cross, case["sigma"] * torch.where(gas, kg, -kg), 0.0)
        t = b * j / (h * h)
        source += _hi(t, a) - t
        if d["mdot"] is not None:
            m = d["mdot"]
            flux = torch.where(cross, -((1 - wl) * _lo(m, a) + wl * m) * (1 / RHO_G - 1 / RHO_L), 0.0)
            share += b * wl * rl * flux / h + _hi(b * (1 - wl) * rho * flux / h, a)
        beta.append(b)
        jump.append(j)
    return beta, jump, source + share, dd


def _solve(beta, dd, b, h, singular):
    """Jacobi-preconditioned conjugate gradients, restarted on the true residual."""
    bh = [_hi(c, a) for a, c in enumerate(beta)]
    diag = (sum(beta) + sum(bh) + dd) / (h * h)

    def minus_a(x):
        y = dd * x
        for a in range(3):
            f = beta[a] * (x - _lo(x, a))
            y = y + f - _hi(f, a)
        return y / (h * h)
    if singular:
        b = b - b.mean()
    size = float(torch.linalg.norm(b))
    x, best, least = torch.zeros_like(b), None, math.inf
    for _ in range(10):
        r = -b - minus_a(x)
        if singular:
            r = r - r.mean()
        now = float(torch.linalg.norm(r))
        if not now < 0.7 * least:  # the true residual no longer falls: 64 bits are used up
            break
        best, least = x, now
        d, rz = torch.zeros_like(b), torch.ones((), dtype=b.dtype, device=b.device)
        for it in range(20000):
            z = r / diag
            new = (r * z).sum()
            d = z + (new / rz if it else 0.0) * d
            q = minus_a(d)
            alpha = new / (d * q).sum()
            x = x + alpha * d
            r = r - alpha * q
            rz = new
            if it % 16 == 15 and float(torch.linalg.norm(r)) <= max(1e-6 * now, 1e-15 * size):
                break
    x = best
    return x - x.mean() if singular else x


def exact(case, seed):
    n = case["nx"] * case["ny"] * case["nz"]
    if case["kind"] in ("conv", "wgrad"):
        d = _layer_inputs(case, seed)
        x = d["xa"].double()
        if case["up"]:
            for axis in range(3):
                x = x.repeat_interleave(2, axis)
        if d["xb"] is not None:
            x = torch.cat([x, d["xb"].double()], 3)
        x = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
        taps = [x[t // 9:t // 9 + case["nz"], t // 3 % 3:t // 3 % 3 + case["ny"],
                  t % 3:t % 3 + case["nx"]] for t in range(27)]
        if case["kind"] == "conv":
            w, y = d["w"].double(), d["bias"].double()
            for t in range(27):
                y = y + taps[t] @ w[:, t].T
            return y.relu()
        g = d["g"].double().reshape(n, -1)
        return torch.stack([g.T @ taps[t].reshape(n, -1) for t in range(27)], 1)
    if n > 3e6:
        return None  # the plain iteration takes too long
    d = _flow_inputs(case, seed)
    h = d["h"]
    beta, jump, source, dd = _system(d)
    rhs = (sum(_hi(c, a) - c for a, c in enumerate(d["u"])) / h if case["kind"] == "project"
           else d["rhs"])
    p = _solve(beta, dd, rhs + source, h, not any(c in "td" for c in case["bc"]))
    if case["kind"] == "pressure":
        return p
    u = [c - b * (p - _lo(p, a) - j) / h
         for a, (c, b, j) in enumerate(zip(d["u"], beta, jump))]
    return dict(ux=u[0], uy=u[1], uz=u[2], p=p)
