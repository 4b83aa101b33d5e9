"""What a user of this package has it do, as measurable cases: the density map, the coupled time
step, the lattice-Boltzmann step and the predictor network, through the Python binding.

A case is a plain dict; "kind" says which call it is:
  density   phi[U] of one system (Context.densities)
  step      restore a state (compositions, potentials, populations), advance it, read it back
            (Context.set / step / get), one system or several replicas in one context
  lb        restore populations, advance the lattice-Boltzmann part alone under a given force
  forward   the predictor network on a batch of potentials (Net.forward)
  gradient  loss and parameter gradient of the network on a batch of pairs (Net.gradient)
`exact` restates each of them in 64 bits with plain torch operations.
"""
import math

import torch

from paper_1204_2088_gb300 import dscf, inputs

DEV = "cuda"


# -- the cases --------------------------------------------------------------------------------

def _system(name, kind, grid, N, f, chiN, fp=32, ns=2, phi_p=1.0, iters=4, hydro=1, steps=1, tau_s=1.0, tau_b=0.8):
    return {"name": name, "kind": kind, "nx": grid[0], "ny": grid[1], "nz": grid[2], "N": N, "f": f, "chiN": chiN,
            "fp": fp, "ns": ns, "phi_p": phi_p, "iters": iters, "hydro": hydro, "steps": steps, "tau_s": tau_s,
            "tau_b": tau_b, "replicas": ""}


def listed():
    cases = [
        # the symmetric 32^3 melt of the plain method in double precision: small, launch-bound
        _system("density_melt32_fp64", "density", (32, 32, 32), 32, 0.5, 20.0, fp=64),
        # the 128^3 melt with 64 beads, the package's headline system: one density evaluation
        _system("density_melt128", "density", (128, 128, 128), 64, 0.3, 25.0),
        # a box whose sides fit no tile, as when the box is matched to a domain spacing
        _system("density_ragged", "density", (100, 90, 75), 48, 0.4, 20.0),
        # the 256^3 melt (the workload the predictor was meant for): the largest single system
        _system("density_melt256", "density", (256, 256, 256), 64, 0.5, 20.0),
        # ordering runs: the 48^3 box of short chains, many cheap steps between two readings
        _system("step_quench48", "step", (48, 48, 48), 16, 0.5, 16.0, iters=6, steps=2, tau_b=1.0),
        # the headline: coupled steps of the 128^3 melt between two checkpoints
        _system("step_melt128", "step", (128, 128, 128), 64, 0.3, 25.0, steps=2),
        # the same system in double precision, the form the 32-bit one is judged against
        _system("step_melt128_fp64", "step", (128, 128, 128), 64, 0.3, 25.0, fp=64),
        # amphiphile in solvent, three species
        _system("step_solution128", "step", (128, 128, 128), 48, 0.3, 30.0, ns=3, phi_p=0.12, steps=2, tau_s=0.8, tau_b=1.2),
        # the batch of 48 melts of three sizes and mixed chain lengths in one context
        dict(_system("step_batch48", "step", (0, 0, 0), 0, 0.0, 0.0), replicas="batch48"),
        # flow alone: relaxation of a velocity field at 128^3 under a given force
        _system("lb_melt128", "lb", (128, 128, 128), 64, 0.3, 25.0, steps=16),
        # predictor inference on the headline grid
        {"name": "net_forward128", "kind": "forward", "nx": 128, "ny": 128, "nz": 128, "batch": 1},
        # predictor training: batches of eight 32^3 boxes
        {"name": "net_gradient32", "kind": "gradient", "nx": 32, "ny": 32, "nz": 32, "batch": 8},
    ]
    return cases


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _side(rng, hi):
    """A box side from 16 to hi: half of them the usual ones, the others any number."""
    if rng.random() < 0.5:
        return rng.choice([s for s in (16, 32, 48, 64, 96, 128, 256) if s <= hi])
    return _log(rng, 16, hi)


def draw(rng):
    kind = rng.choice(["density", "density", "density", "step", "step", "step", "batch", "lb", "forward", "gradient"])
    if kind in ("forward", "gradient"):
        while True:
            nx = 16 * rng.randint(1, 8)
            ny, nz, batch = _log(rng, 8, 128), _log(rng, 8, 128), rng.randint(1, 8)
            if nx * ny * nz * batch <= (1 << 21 if kind == "forward" else 1 << 18):
                return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "batch": batch}
    if kind == "batch":
        reps = []
        for _ in range(rng.randint(2, 12)):
            L = rng.choice([32, 48, 48, 64, 64, 96, _log(rng, 16, 96)])
            reps.append("%dx%dx%d:%d:%.2f:%.1f" % (L, L, L, rng.choice([32, 48, 64]), rng.choice([0.3, 0.4, 0.5]),
                                                    rng.choice([15.0, 20.0, 30.0])))
        c = dict(_system("", "step", (0, 0, 0), 0, 0.0, 0.0, steps=rng.randint(1, 2)), replicas=";".join(reps))
        del c["name"]
        return c
    fp = 64 if rng.random() < 0.3 else 32
    most = {"density": (1 << 24) // (4 if fp == 64 else 1), "step": (1 << 21) // (2 if fp == 64 else 1), "lb": 1 << 21}[kind]
    while True:
        grid = [_side(rng, 256 if kind == "density" else 128) for _ in range(3)]
        if grid[0] * grid[1] * grid[2] <= most:
            break
    ns = 3 if rng.random() < 0.3 else 2
    c = _system("", kind, grid, _log(rng, 8, 64), round(rng.uniform(0.2, 0.8), 2), round(rng.uniform(12.0, 30.0), 1),
                fp=fp, ns=ns, phi_p=round(rng.uniform(0.1, 0.4), 2) if ns == 3 else 1.0, iters=rng.randint(1, 6),
                hydro=rng.randint(0, 1) if kind == "step" else 1,
                steps=1 if fp == 64 else rng.randint(1, 16 if kind == "lb" else 2),
                tau_s=rng.choice([0.6, 1.0, 2.0]), tau_b=rng.choice([0.8, 1.0, 1.5]))
    del c["name"]
    return c


# -- systems ----------------------------------------------------------------------------------

def _configs(case):
    """The parameter dicts of the case's replicas (the binding's own input)."""
    it = {"ncg_iters": case["iters"], "hydro": case["hydro"]}
    if case["replicas"] == "batch48":
        return inputs.batch48(**it)
    if case["replicas"]:
        out = []
        for k, r in enumerate(case["replicas"].split(";")):
            g, N, f, chiN = r.split(":")
            out.append(dict(inputs.melt([int(v) for v in g.split("x")], int(N), float(f), float(chiN),
                                        (0.6, 1.0, 2.0)[k % 3], (0.8, 1.5)[k % 2], dt=inputs.WORKLOAD_DT), **it))
        return out
    g, N, chiN = (case["nx"], case["ny"], case["nz"]), case["N"], case["chiN"]
    if case["ns"] == 3:
        c = inputs.solution(g, N, case["f"], case["phi_p"], chiN, 1.15 * chiN, 0.0, case["tau_s"], case["tau_b"], dt=inputs.WORKLOAD_DT)
    else:
        c = inputs.melt(g, N, case["f"], chiN, case["tau_s"], case["tau_b"], dt=inputs.WORKLOAD_DT)
    c["nA"] = min(max(c["nA"], 1), N - 1)
    return [dict(c, **it)]


def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) & 0x7FFFFFFFFFFF)


def _pattern(gen, shape, modes=6, period=(10.0, 16.0)):
    """A smooth periodic field of unit variance: a few plane waves of the box in random directions
    with periods of some lattice spacings, as a microphase pattern part-way through its ordering."""
    nz, ny, nx = shape
    ax = [2 * math.pi * torch.arange(n, dtype=torch.float64, device=DEV) / n for n in (nz, ny, nx)]
    n = torch.tensor(shape, dtype=torch.float64, device=DEV)
    f = torch.zeros(shape, dtype=torch.float64, device=DEV)
    for _ in range(modes):
        k = _noise(gen, (3,))
        r = torch.rand(2, generator=gen, dtype=torch.float64, device=DEV)
        k = torch.round(n * k / k.norm() / (period[0] + (period[1] - period[0]) * r[0]))
        k[0] = torch.where((k == 0).all(), torch.ones_like(k[0]), k[0])
        f += torch.cos(k[0] * ax[0][:, None, None] + k[1] * ax[1][None, :, None] + k[2] * ax[2][None, None, :] + 2 * math.pi * r[1])
    return f / math.sqrt(modes / 2)


def _noise(gen, shape):
    return torch.randn(shape, generator=gen, dtype=torch.float64, device=DEV)


def _potentials(gen, cfg):
    """Potentials of a part-way ordered state: opposite patterns on the two blocks, balanced along
    the chain as incompressibility wants it, and the roughness that the composition noise leaves."""
    nx, ny, nz = cfg["grid"]
    shape = (nz, ny, nx)
    N, nA = cfg["N"], cfg["nA"]
    amp = 1.0 / N
    h, p = _pattern(gen, shape), _pattern(gen, shape)
    U = torch.stack([2 * amp * (N - nA) / N * h, -2 * amp * nA / N * h] + ([0.5 * amp * h] if cfg["ns"] == 3 else []))
    return U + 0.02 * amp * p + 0.02 * amp * _noise(gen, (cfg["ns"],) + shape)


C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
     (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1),
     (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12


def _populations(gen, cfg):
    """Population deviations of a smooth flow of Courant numbers of some thousandths."""
    nx, ny, nz = cfg["grid"]
    u = torch.stack([4e-3 * _pattern(gen, (nz, ny, nx), 3, (24.0, 64.0)) for _ in range(3)])
    rho = 1e-4 * _pattern(gen, (nz, ny, nx), 3, (24.0, 64.0))
    return torch.stack([w * (rho + 3 * (c[0] * u[0] + c[1] * u[1] + c[2] * u[2])) for c, w in zip(C, W)])


def _inputs(case, seed):
    """What the user holds, as a dict of lists over replicas (in the precision of the call)."""
    gen = _generator(seed)
    dt = torch.float64 if case["fp"] == 64 else torch.float32
    cfgs = _configs(case)
    d = {"cfgs": cfgs, "dt": dt}
    if case["kind"] == "lb":
        d["pop"] = [_populations(gen, c).to(dt) for c in cfgs]
        d["force"] = [torch.stack([1e-5 * _pattern(gen, c["grid"][::-1], 3) for _ in range(3)]).to(dt) for c in cfgs]
        return d
    d["U"] = [_potentials(gen, c).to(dt) for c in cfgs]
    if case["kind"] == "step":
        # compositions that these potentials nearly reproduce: one time step has moved them since
        d["phi"] = []
        for c, U in zip(cfgs, d["U"]):
            phi = _exact_densities(c, U.double())
            g = 1e-3 * _noise(gen, phi.shape[1:])
            g = g - g.mean()
            phi[0] += 0.3 * g * phi[0]
            phi[1] -= 0.3 * g * phi[1]
            d["phi"].append(phi.to(dt))
        d["pop"] = [_populations(gen, c).to(dt) for c in cfgs]
    return d


def _net_inputs(case, seed):
    gen = _generator(seed)
    shape = (case["nz"], case["ny"], case["nx"])
    U = []
    for _ in range(case["batch"]):
        h = 0.2 * _pattern(gen, shape)
        U.append(torch.stack([h, -h]) + 0.02 * _noise(gen, (2,) + shape))
    U = torch.stack(U).float()
    target = 0.5 - 0.8 * (U - U.mean(dim=(2, 3, 4), keepdim=True))
    return U, target.contiguous()


def _net_params(seed):
    """Weights of the size that an untrained or lightly trained network has, small biases."""
    gen = _generator(int(seed) + 7)
    p = []
    for cin, cout in ((2, 32), (32, 32), (32, 2)):
        p.append(math.sqrt(2.0 / ((cin + cout) * 125)) * _noise(gen, (cout * cin * 125,)))
        p.append(0.02 * _noise(gen, (cout,)))
    return torch.cat(p).float()


# -- the calls --------------------------------------------------------------------------------

PHIBAR = (0.5, 0.5)


def prepare(case, seed):
    if case["kind"] in ("forward", "gradient"):
        U, target = _net_inputs(case, seed)
        net = dscf.Net((case["nx"], case["ny"], case["nz"]), case["batch"])
        net.set_params(_net_params(seed))
        return {"case": case, "net": net, "U": U, "target": target}
    d = _inputs(case, seed)
    cfgs = d["cfgs"]
    ctx = dscf.Context(cfgs[0] if len(cfgs) == 1 else cfgs, dscf.FP64 if case["fp"] == 64 else dscf.FP32)
    s = {"case": case, "ctx": ctx}
    for k in ("U", "phi", "pop", "force"):
        if k in d:
            s[k] = d[k][0] if len(cfgs) == 1 else torch.cat([v.reshape(-1) for v in d[k]])
    return s


def run(state):
    case = state["case"]
    if case["kind"] == "forward":
        return state["net"].forward(state["U"], PHIBAR)
    if case["kind"] == "gradient":
        loss, g = state["net"].gradient(state["U"], state["target"], PHIBAR)
        return {"loss": loss, "gradient": g}
    ctx = state["ctx"]
    if case["kind"] == "density":
        return ctx.densities(state["U"])
    if case["kind"] == "lb":
        ctx.set(dscf.POP, state["pop"])
        ctx.lb_step(state["force"], case["steps"])
        return {"populations": ctx.get(dscf.POP), "velocity": ctx.get(dscf.VEL)}
    ctx.set(dscf.PHI, state["phi"])
    ctx.set(dscf.U, state["U"])
    if case["hydro"]:
        ctx.set(dscf.POP, state["pop"])
    ctx.step(case["steps"])
    out = {"phi": ctx.get(dscf.PHI), "U": ctx.get(dscf.U)}
    if case["hydro"]:
        out["populations"], out["velocity"] = ctx.get(dscf.POP), ctx.get(dscf.VEL)
    return out


# -- what a pass cannot do without ------------------------------------------------------------

def work(case):
    if case["kind"] in ("forward", "gradient"):
        S = case["nx"] * case["ny"] * case["nz"] * case["batch"]
        conv = 2 * 125 * (2 * 32 + 32 * 32 + 32 * 2) * S      # multiply-adds of the three layers
        params = 4 * 144418
        if case["kind"] == "forward":
            return {"bytes": 16 * S + params, "flops": conv}
        # the input gradient of the first layer is not needed
        return {"bytes": 16 * S + 2 * params, "flops": 3 * conv - 2 * 125 * 2 * 32 * S}
    es = case["fp"] // 8
    b = fl = 0
    for c in _configs(case):
        V, ns, N = c["grid"][0] * c["grid"][1] * c["grid"][2], c["ns"], c["N"]
        # one density evaluation: U in, phi out, and the propagators of one chain direction written
        # once and read once (the other direction can meet them on the way); 15 operations for each
        # bead of either direction (three three-point passes and the factor), two for the quadrature
        ev_b, ev_f = V * es * (2 * ns + 2 * N), V * (2 * N * 15 + 2 * N)
        if case["kind"] == "density":
            b, fl = b + ev_b, fl + ev_f
            continue
        lb_b, lb_f = V * es * (2 * 19 + 3 + 3), V * 250
        if case["kind"] == "lb":
            b, fl = b + case["steps"] * lb_b, fl + case["steps"] * lb_f
            continue
        evals = 2 * case["iters"] * case["steps"] + 1          # the first for phi at the potentials given
        # phi, U in and out, mu out and in, one pass of the Crank-Nicolson update
        rest_b = V * es * (6 * ns + 4 * ns) + (lb_b if case["hydro"] else 0)
        rest_f = V * ns * (60 + 25 * c["cn_sweeps"]) + (lb_f if case["hydro"] else 0)
        b += evals * ev_b + case["steps"] * rest_b
        fl += evals * ev_f + case["steps"] * rest_f
    return {"bytes": b, "flops": fl}


# -- the same in 64 bits, with plain torch ------------------------------------------------------

def _sigma(f, alpha):
    """The 27-point linkage stencil (its three passes) on the last three axes."""
    for ax in (-1, -2, -3):
        f = (1 - 2 * alpha) * f + alpha * (torch.roll(f, 1, ax) + torch.roll(f, -1, ax))
    return f


def _exact_densities(c, U):
    N, nA, ns, a = c["N"], c["nA"], c["ns"], c["a"] ** 2 / 6
    E = torch.exp(-U)
    g = torch.ones_like(U[0])
    G = []
    for s in range(1, N + 1):
        g = E[0 if s <= nA else 1] * _sigma(g, a)
        G.append(g)
    Q = G[-1].mean()
    q = torch.zeros_like(U[:2])
    g = torch.ones_like(U[0])
    for s in range(N, 0, -1):
        I = 0 if s <= nA else 1
        sg = _sigma(g, a)
        q[I] += G[s - 1] * sg
        g = E[I] * sg
    del G
    phi = torch.empty_like(U)
    phi[:2] = c["phi_p"] / (N * Q) * q
    if ns == 3:
        phi[2] = (1 - c["phi_p"]) * E[2] / E[2].mean()
    return phi


def _exact_invert(c, phi, U, pm):
    """Fletcher-Reeves with one trial point per line search."""
    g = phi - pm
    d = -g
    gg = (g * g).sum()
    for k in range(c["ncg_iters"]):
        h0, cd = (g * d).sum(), (d * pm * d).sum()
        a1 = -h0 / cd if cd > 0 else torch.zeros_like(h0)
        h1 = ((phi - _exact_densities(c, U + a1 * d)) * d).sum()
        a = a1 * (-h0) / (h1 - h0) if h1 - h0 > 0 else a1
        U = U + a * d
        pm = _exact_densities(c, U)
        g = phi - pm
        new = (g * g).sum()
        d = -g + (new / gg if gg > 0 else 0.0) * d
        gg = new
    return U, pm


def _exact_lb(c, pop, f):
    """One collision under the lattice force f and the streaming after it; the velocity of the
    collision beside the new populations."""
    gs, gb = 1 - 1 / c["tau_s"], 1 - 1 / c["tau_b"]
    w = torch.tensor(W, dtype=torch.float64, device=DEV)
    ci = torch.tensor(C, dtype=torch.float64, device=DEV)
    rho_d = pop.sum(0)
    rho = c["rho0"] + rho_d
    u = (torch.einsum("ia,i...->a...", ci, pop) + 0.5 * f) / rho
    ident = torch.eye(3, dtype=torch.float64, device=DEV)[:, :, None, None, None]
    neq = torch.einsum("ia,ib,i...->ab...", ci, ci, pop) - rho * u[:, None] * u[None, :] - ident * rho_d / 3
    tr = (neq[0, 0] + neq[1, 1] + neq[2, 2]) / 3
    uf = (u * f).sum(0)
    sym = u[:, None] * f[None, :] + u[None, :] * f[:, None]
    S = 0.5 * (1 + gs) * (sym - ident * 2 * uf / 3) + (1 + gb) / 3 * ident * uf
    # second-order part of the post-collision state, contracted with c c - 1/3
    Q2 = rho * u[:, None] * u[None, :] + gs * (neq - ident * tr) + gb * ident * tr + S
    q_tr = (Q2[0, 0] + Q2[1, 1] + Q2[2, 2]) / 3
    lin = 3 * rho * u + 1.5 * f
    out = []
    for i, (x, y, z) in enumerate(C):
        quad = sum(C[i][a] * C[i][b] * Q2[a, b] for a in range(3) for b in range(3) if C[i][a] and C[i][b])
        n = w[i] * (rho_d + x * lin[0] + y * lin[1] + z * lin[2] + 4.5 * (quad - q_tr))
        out.append(torch.roll(n, (z, y, x), (0, 1, 2)))
    return torch.stack(out), u


def _exact_diffuse(c, phi, mu, u, mass):
    """Convection by u, Crank-Nicolson diffusion by Jacobi sweeps, totals put back."""
    ns, kap, cc = c["ns"], c["kappa"], 0.5 * c["dt"] * c["M"]
    ax = (-1, -2, -3)
    rhs = torch.zeros_like(phi)
    for k in range(3):
        up = lambda f: torch.roll(f, -1, ax[k])        # noqa: E731
        down = lambda f: torch.roll(f, 1, ax[k])       # noqa: E731
        face = 0.5 * (phi + up(phi))
        half = face - 0.5 * (up(u[k] * phi) - u[k] * phi)
        flux = 0.5 * (u[k] + up(u[k])) * half - c["dt"] * c["M"] * face * (up(mu) - mu)
        rhs -= flux - down(flux)
    inv = 1 / torch.clamp(phi, min=c["phi_floor"])
    wsum = sum(0.5 * (phi + torch.roll(phi, s, a)) for a in ax for s in (1, -1))
    D, A = 1 + cc * wsum * inv, cc * kap * wsum
    den = 1 + (A / D).sum(0)
    x = torch.zeros_like(phi)
    for _ in range(c["cn_sweeps"]):
        psi = x * inv + kap * x.sum(0)
        r = rhs + cc * sum(0.5 * (phi + torch.roll(phi, s, a)) * torch.roll(psi, s, a) for a in ax for s in (1, -1))
        x = (r - A * ((r / D).sum(0) / den)) / D
    new = phi + x
    return new + (mass - new.sum(dim=(1, 2, 3)))[:, None, None, None] / phi[0].numel()


def _exact_steps(c, phi, U, pop, steps):
    chi = torch.zeros(3, 3, dtype=torch.float64, device=DEV)
    for (i, j), v in c["chi"].items():
        chi[i, j] = chi[j, i] = v
    chi = chi[:c["ns"], :c["ns"]]
    mass = phi.sum(dim=(1, 2, 3))
    pm = _exact_densities(c, U)
    u = torch.zeros((3,) + phi.shape[1:], dtype=torch.float64, device=DEV)
    for _ in range(steps):
        U, pm = _exact_invert(c, phi, U, pm)
        mu = -U + torch.einsum("ij,j...->i...", chi, _sigma(phi, c["a"] ** 2 / 6)) + c["kappa"] * (phi.sum(0) - 1)
        if pop is not None:
            f = -c["dt"] ** 2 * torch.stack([(phi * 0.5 * (torch.roll(mu, -1, a) - torch.roll(mu, 1, a))).sum(0) for a in (-1, -2, -3)])
            pop, u = _exact_lb(c, pop, f)
        phi = _exact_diffuse(c, phi, mu, u, mass)
    return phi, U, pop, u


def _split(params):
    out, at = [], 0
    for cin, cout in ((2, 32), (32, 32), (32, 2)):
        n = cout * cin * 125
        out.append((params[at:at + n].reshape(cout, cin, 5, 5, 5), params[at + n:at + n + cout]))
        at += n + cout
    return out


class _Conv(torch.autograd.Function):
    """A circular 5^3 convolution in 64 bits, offset by offset: [Cin, z, y, x] -> [Cout, z, y, x]."""

    @staticmethod
    def forward(ctx, x, w):
        ctx.save_for_backward(x, w)
        out = torch.zeros((w.shape[0],) + x.shape[1:], dtype=x.dtype, device=x.device)
        flat = out.view(w.shape[0], -1)
        for o in range(125):
            z, y, k = o // 25, o // 5 % 5, o % 5
            flat.addmm_(w[:, :, z, y, k], torch.roll(x, (2 - z, 2 - y, 2 - k), (1, 2, 3)).view(x.shape[0], -1))
        return out

    @staticmethod
    def backward(ctx, g):
        x, w = ctx.saved_tensors
        gw, gx = torch.zeros_like(w), torch.zeros_like(x)
        gf = g.reshape(g.shape[0], -1)
        for o in range(125):
            z, y, k = o // 25, o // 5 % 5, o % 5
            gw[:, :, z, y, k] = gf @ torch.roll(x, (2 - z, 2 - y, 2 - k), (1, 2, 3)).reshape(x.shape[0], -1).T
            gx += torch.roll((w[:, :, z, y, k].T @ gf).view(x.shape), (z - 2, y - 2, k - 2), (1, 2, 3))
        return gx, gw


def _exact_net(U, params):
    """phi_hat of every sample of U [B, 2, z, y, x]."""
    out = []
    for s in range(U.shape[0]):
        x = U[s] - U[s].mean(dim=(1, 2, 3), keepdim=True)
        for k, (w, b) in enumerate(_split(params)):
            x = _Conv.apply(x, w) + b[:, None, None, None]
            if k < 2:
                x = torch.tanh(x)
        out.append(torch.tensor(PHIBAR, dtype=torch.float64, device=DEV)[:, None, None, None] + x - x.mean(dim=(1, 2, 3), keepdim=True))
    return torch.stack(out)


def exact(case, seed):
    if case["kind"] in ("forward", "gradient"):
        U, target = _net_inputs(case, seed)
        params = _net_params(seed).double()
        if case["kind"] == "forward":
            with torch.no_grad():
                return _exact_net(U.double(), params)
        params.requires_grad_(True)
        total = 0.0
        for s in range(case["batch"]):              # sample by sample: the graph of one at a time
            loss = 0.5 * ((_exact_net(U[s:s + 1].double(), params) - target[s:s + 1].double()) ** 2).sum() / target.numel()
            loss.backward()
            total += float(loss.detach())
        return {"loss": total, "gradient": params.grad}
    d = _inputs(case, seed)
    cfgs = d["cfgs"]
    if case["kind"] == "density":
        return _exact_densities(cfgs[0], d["U"][0].double())
    whole = (lambda v: v[0]) if len(cfgs) == 1 else (lambda v: torch.cat([t.reshape(-1) for t in v]))
    if case["kind"] == "lb":
        pops, us = [], []
        for c, pop, f in zip(cfgs, d["pop"], d["force"]):
            pop, f = pop.double(), f.double()
            for _ in range(case["steps"]):
                pop, u = _exact_lb(c, pop, f)
            pops.append(pop)
            us.append(u)
        return {"populations": whole(pops), "velocity": whole(us)}
    got = [_exact_steps(c, phi.double(), U.double(), pop.double() if case["hydro"] else None, case["steps"])
           for c, phi, U, pop in zip(cfgs, d["phi"], d["U"], d["pop"])]
    out = {"phi": whole([g[0] for g in got]), "U": whole([g[1] for g in got])}
    if case["hydro"]:
        out["populations"], out["velocity"] = whole([g[2] for g in got]), whole([g[3] for g in got])
    return out
