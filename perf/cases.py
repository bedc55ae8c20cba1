"""The work that users of this framework have it do, as cases that can be timed.

A case is a dict of plain values. `prepare` builds what a program holds before the call (the
solver and its state on the GPU), `run` is one pass through the public entry points, `exact`
recomputes a pass in plain 64-bit torch operations from the definition of the scheme (Porth
et al. 2014, Sec. 2 and 4, App. C), without the framework.

Kinds of pass ("do"):
  run       `steps` time steps of one domain from its initial state; "path" is the entry
            point: "cfl" (step_cfl), "plain" (dt, then step), "graph" (dt, then step_batched)
  batch     one step of many independent 3D blocks of uneven size, some of them passive, each
            with its own time step
  dt        the time step alone of many blocks, without a handle (dt_noalloc)
  grad      one differentiable step: the new state and the gradient of its input
  rollout   `steps` differentiable steps with a checkpoint every `every`: state and gradient
  activate  the steady-state criterion, the safety belt and one step of the active blocks
"""
import math

import torch

from paper_1407_2052_gb300 import amrfd, autodiff
from paper_1407_2052_gb300.workloads import Domain

EULER, MHD = amrfd.EULER, amrfd.MHD_GLM
RK3, RK54, RK43 = amrfd.SSPRK3, amrfd.SSPRK54, amrfd.SSPRK43
MP5, LIMO3 = amrfd.MP5, amrfd.LIMO3
STAGES = {RK3: 3, RK54: 5, RK43: 4}
GLM_CR = 0.18
GAMMA = {EULER: 1.4, MHD: 5.0 / 3.0}
BATCH_EDGES = (8, 12, 16, 24, 32)


def box(do, phys, n, nb, bc, ic, integ=RK3, recon=MP5, path="cfl", steps=1, tune=False, every=0, cfl=0.4):
    """A case of one domain. n: cells, nb: blocks, bc: one letter per dimension (p periodic,
    o outflow, w reflecting wall) for both faces."""
    n, nb = tuple(n) + (1,) * (3 - len(n)), tuple(nb) + (1,) * (3 - len(nb))
    return {"do": do, "phys": phys, "ndim": len(bc), "nx": n[0], "ny": n[1], "nz": n[2], "bx": nb[0], "by": nb[1],
            "bz": nb[2], "bc": bc, "ic": ic, "integ": integ, "recon": recon, "path": path, "steps": steps,
            "tune": tune, "every": every, "cfl": cfl}


def listed():
    return [
        # the smallest work: a shock tube of 512 cells; 16 dependent steps, launches and latency
        {"name": "sod_512", **box("run", EULER, (512,), (1,), "o", "tube", steps=16)},
        # a 1D MHD tube with the five-stage integrator, dt and step as separate calls
        {"name": "briowu_512", **box("run", MHD, (512,), (1,), "o", "tube", RK54, path="plain", steps=8)},
        # a small 2D MHD run between reflecting walls, several blocks
        {"name": "wall_blast_128", **box("run", MHD, (128, 128), (4, 4), "pw", "blast", steps=4, cfl=0.3)},
        # an ordinary 2D MHD run: the smooth vortex at its own size, graph replay, five stages
        {"name": "vortex_1024", **box("run", MHD, (1024, 1024), (1, 1), "pp", "vortex", RK54, path="graph")},
        # Euler in 3D at odd sizes with all three kinds of face, SSPRK(4,3), dt and step separate
        {"name": "euler_ragged", **box("run", EULER, (123, 95, 78), (3, 5, 2), "owp", "blast", RK43, path="plain")},
        # the paper's cheap scheme: RK3 with LIMO3, 3D MHD blast
        {"name": "limo3_blast_128", **box("run", MHD, (128,) * 3, (8,) * 3, "ppp", "blast", recon=LIMO3, cfl=0.3)},
        # the largest work, the benchmark's: 3D MHD blast, 256^3 cells in 16^3 blocks, tuned tile
        {"name": "blast_256", **box("run", MHD, (256,) * 3, (16,) * 3, "ppp", "blast", tune=True, cfl=0.3)},
        # many uneven blocks, 30 % of them passive, each with its own time step
        {"name": "batch_1500", "do": "batch", "blocks": 1500, "passive": 0.3},
        # time step of many small blocks, no allocation
        {"name": "dt_900", "do": "dt", "blocks": 900, "passive": 0.1, "edge": 16},
        # training through one step: the adjoint workload at its own size
        {"name": "grad_512", **box("grad", MHD, (512, 512), (1, 1), "pp", "waves")},
        # the gradient through several steps, checkpointed
        {"name": "rollout_192", **box("rollout", MHD, (192, 192), (1, 1), "pp", "waves", steps=10, every=5)},
        # dynamic activation: a blast into a steady background, few blocks active
        {"name": "quiet_blast_128", **box("activate", MHD, (128,) * 3, (8,) * 3, "ppp", "quiet", cfl=0.3)},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _edges(rng, lo, hi, most_blocks):
    """(cells, blocks) along one dimension: a block edge and a number of blocks."""
    nb = rng.randint(1, most_blocks)
    return max(6, _log_int(rng, lo, hi) // nb) * nb, nb


def draw(rng):
    do = rng.choice(("tube", "tube", "plane", "plane", "box", "box", "box", "batch", "dt", "grad", "rollout", "activate"))
    phys = rng.choice((EULER, MHD, MHD))
    integ, recon = rng.choice((RK3, RK3, RK54, RK43)), rng.choice((MP5, MP5, LIMO3))
    path = rng.choice(("cfl", "plain", "graph"))
    if do == "tube":
        n, nb = _edges(rng, 48, 30000, 4)
        return box("run", phys, (n,), (nb,), rng.choice("opw"), "tube", integ, recon, path, rng.randint(1, 16))
    if do == "plane":
        x, y = _edges(rng, 24, 1300, 8), _edges(rng, 24, 1300, 8)
        return box("run", phys, (x[0], y[0]), (x[1], y[1]), rng.choice("pow") + rng.choice("pow"),
                   rng.choice(("blast", "waves")), integ, recon, path, rng.randint(1, 3), cfl=0.3)
    if do == "box":
        x, y, z = (_edges(rng, 16, 190, 8) for _ in range(3))
        return box("run", phys, (x[0], y[0], z[0]), (x[1], y[1], z[1]), "".join(rng.choice("ppow") for _ in range(3)),
                   rng.choice(("blast", "waves")), rng.choice((RK3, RK43)), recon, path, 1, cfl=0.3)
    if do == "batch":
        return {"do": "batch", "blocks": _log_int(rng, 20, 1400), "passive": rng.choice((0.0, 0.3, 0.6))}
    if do == "dt":
        return {"do": "dt", "blocks": _log_int(rng, 10, 1000), "passive": rng.choice((0.0, 0.1, 0.5)),
                "edge": rng.choice((6, 9, 16, 21, 32))}
    if do == "grad":
        n = _log_int(rng, 24, 500)
        return box("grad", phys, (n, _log_int(rng, 24, 500)), (1, 1), "pp", "waves", integ, recon)
    if do == "rollout":
        n, steps = _log_int(rng, 24, 190), rng.randint(2, 10)
        return box("rollout", phys, (n, n), (1, 1), "pp", "waves", RK3, MP5, steps=steps, every=rng.randint(1, steps))
    e = [(rng.randint(6, 18), rng.randint(3, 7)) for _ in range(3)]
    return box("activate", phys, [a * b for a, b in e], [b for _, b in e], "ppp", "quiet", recon=recon, cfl=0.3)


# ------------------------------------------------------------------- inputs
def _nv(c):
    return 9 if c["do"] in ("batch", "dt") or c["phys"] == MHD else 2 + c["ndim"]


def _conserved(phys, ndim, rho, vel, p, B=None):
    """Conserved variables stacked in dimension -4 from fields of shape (..., nz, ny, nx)."""
    g = GAMMA[phys]
    if phys == EULER:
        e = p / (g - 1.0) + 0.5 * rho * sum(v * v for v in vel[:ndim])
        return torch.stack([rho] + [rho * v for v in vel[:ndim]] + [e], dim=-4)
    e = p / (g - 1.0) + 0.5 * rho * sum(v * v for v in vel) + 0.5 * sum(b * b for b in B)
    return torch.stack([rho] + [rho * v for v in vel] + [e] + list(B) + [torch.zeros_like(rho)], dim=-4)


def _length(c):
    return 2.0 * math.pi if c["ic"] in ("vortex", "waves") else 1.0


def _spacing(c):
    n = (c["nx"], c["ny"], c["nz"])
    return tuple(_length(c) / n[d] if d < c["ndim"] else 1.0 for d in range(3))


def _rand(gen, *shape):
    return torch.rand(*shape, generator=gen, device="cuda", dtype=torch.float64)


def _initial(c, seed):
    """(state, steady background or None) of a one-domain case, shape (nv, nz, ny, nx)."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    n, dx, nd = (c["nx"], c["ny"], c["nz"]), _spacing(c), c["ndim"]
    ax = [(torch.arange(m, device="cuda", dtype=torch.float64) + 0.5) * h for m, h in zip(n, dx)]
    X, Y, Z = ax[0].view(1, 1, -1), ax[1].view(1, -1, 1), ax[2].view(-1, 1, 1)
    zero = torch.zeros(n[2], n[1], n[0], device="cuda", dtype=torch.float64)
    rho, p, vel, B, back = zero + 1.0, zero + 1.0, [zero, zero, zero], [zero, zero, zero], None
    if c["ic"] == "tube":  # Sod's and Brio and Wu's states, the diaphragm and the levels varied
        u = _rand(gen, 4).tolist()
        left = X + zero < 0.4 + 0.2 * u[0]
        rho = torch.where(left, zero + 1.0 + 0.1 * u[1], zero + 0.125)
        p = torch.where(left, zero + 1.0 + 0.1 * u[2], zero + 0.1)
        B = [zero + 0.75, torch.where(left, zero + 1.0, zero - 1.0), zero]
    elif c["ic"] in ("blast", "quiet"):  # high pressure in the middle of a uniform field, density noise
        u = (_rand(gen, 3) * 0.1 + 0.45).tolist()
        r2 = sum((q - a) ** 2 for q, a in zip((X, Y, Z)[:nd], u)) + zero
        if c["ic"] == "blast":
            rho = 1.0 + 1e-3 * (2.0 * _rand(gen, *zero.shape) - 1.0)
        b = 1.0 / math.sqrt(2.0)
        B = [zero + b, zero + b, zero]
        if c["ic"] == "quiet":
            back = _conserved(c["phys"], nd, rho, vel, zero + 0.1, B)
        p = torch.where(r2 < 0.01, zero + 10.0, zero + 0.1)
    elif c["ic"] == "vortex":  # the smooth vortex, its phases varied
        a, b = (_rand(gen, 2) * 2.0 * math.pi).tolist()
        rho, p = zero + 25.0 / 9.0, zero + 5.0 / 3.0
        vel = [zero - torch.sin(Y + a), zero + torch.sin(X + b), zero]
        B = [zero - torch.sin(Y + a), zero + torch.sin(2.0 * (X + b)), zero]
    else:  # smooth Fourier modes about a uniform state
        def modes(amp, m=12):
            ks = (torch.floor(_rand(gen, m, 3) * 9.0) - 4.0).tolist()
            co = ((2.0 * _rand(gen, m) - 1.0) * amp / m).tolist()
            ph = (_rand(gen, m) * 2.0 * math.pi).tolist()
            xs = [q * (2.0 * math.pi / _length(c)) for q in (X, Y, Z)]
            return sum(a * torch.sin(k[0] * xs[0] + (k[1] * xs[1] if nd > 1 else 0.0) + (k[2] * xs[2] if nd > 2 else 0.0)
                                     + f) for a, k, f in zip(co, ks, ph)) + zero
        rho, p, vel = 1.0 + modes(0.02), 1.0 + modes(0.02), [modes(0.02) for _ in range(3)]
        B = [0.5 + modes(0.02), modes(0.02), modes(0.02)]
    return _conserved(c["phys"], nd, rho, vel, p, B).contiguous(), back


def _walls(c, d):
    """Variables odd across a reflecting wall normal to d (B a pseudovector)."""
    if c["phys"] == EULER:
        return 1 << (1 + d)
    return (1 << (1 + d)) | (1 << 8) | sum(1 << (5 + k) for k in range(3) if k != d)


def _domain(c):
    kind = {"p": amrfd.PERIODIC, "o": amrfd.OUTFLOW, "w": amrfd.SYMMETRIC}
    bc = tuple((kind[c["bc"][d]],) * 2 if d < c["ndim"] else (0, 0) for d in range(3))
    asym = tuple((_walls(c, d),) * 2 if d < c["ndim"] and c["bc"][d] == "w" else (0, 0) for d in range(3))
    return Domain((c["nx"], c["ny"], c["nz"]), _spacing(c), bc=bc, nb=(c["bx"], c["by"], c["bz"]), asym=asym)


def _batch_sizes(c):
    """Edges, spacings and active flags of a batch (the case's, whatever the seed)."""
    nb = c["blocks"]
    g = torch.Generator().manual_seed(nb)
    if c["do"] == "dt":  # uneven blocks about the edge
        edges = (c["edge"] + torch.randint(-2, 3, (nb,), generator=g)).tolist()
    else:
        edges = [BATCH_EDGES[i] for i in torch.randint(len(BATCH_EDGES), (nb,), generator=g).tolist()]
    dxs = torch.exp(math.log(1e-3) + torch.rand(nb, generator=g, dtype=torch.float64) * math.log(100.0)).tolist()
    active = (torch.rand(nb, generator=g) >= c["passive"]).to(torch.uint8)
    return edges, dxs, active


def _batch(c, seed):
    """Blocks of a batch: (edges, spacings, offsets, active flags, flat state), all periodic 3D
    MHD with smooth perturbations; the sizes are the case's, the fields the seed's."""
    nb = c["blocks"]
    edges, dxs, active = _batch_sizes(c)
    offs, total = [], 0
    for m in edges:
        offs.append(total)
        total += 9 * m ** 3
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    amp, ph = 0.05 * (2.0 * _rand(gen, nb, 5, 3) - 1.0), _rand(gen, nb, 5, 3) * 2.0 * math.pi
    U = torch.empty(total, device="cuda", dtype=torch.float64)
    for m in sorted(set(edges)):
        sel = [i for i, e in enumerate(edges) if e == m]
        t = (torch.arange(m, device="cuda", dtype=torch.float64) + 0.5) * (2.0 * math.pi / m)
        xs = (t.view(1, 1, -1), t.view(1, -1, 1), t.view(-1, 1, 1))
        for lo in range(0, len(sel), 256):
            at = sel[lo:lo + 256]
            ix = torch.tensor(at, device="cuda")
            a, f = amp[ix].view(-1, 5, 3, 1, 1, 1), ph[ix].view(-1, 5, 3, 1, 1, 1)
            w = sum(a[:, :, k] * torch.sin(xs[k] + xs[(k + 1) % 3] + f[:, :, k]) for k in range(3))
            zero = torch.zeros_like(w[:, 0])
            blk = _conserved(MHD, 3, 1.0 + w[:, 0], [w[:, 2], w[:, 3], w[:, 4]], 1.0 + w[:, 1], [zero + 0.5, zero, zero])
            where = torch.tensor([offs[i] for i in at], device="cuda").view(-1, 1) + torch.arange(9 * m ** 3, device="cuda")
            U[where.reshape(-1)] = blk.reshape(-1)
    return edges, dxs, offs, active, U


def prepare(case, seed):
    c = dict(case)
    if c["do"] in ("batch", "dt"):
        edges, dxs, offs, active, U = _batch(c, seed)
        doms = [Domain((m, m, m), (h,) * 3, offset=o) for m, h, o in zip(edges, dxs, offs)]
        st = {"case": c, "U0": U, "dt": torch.empty(len(doms), device="cuda", dtype=torch.float64)}
        if c["do"] == "dt":
            st.update(domains=doms, active=active.cuda())
        else:
            st.update(solver=amrfd.Solver(MHD, 3, RK3, GAMMA[MHD], 0.4, doms, active=active.numpy(), glm_cr=GLM_CR),
                      U=torch.empty_like(U))
        return st
    U0, back = _initial(c, seed)
    s = amrfd.Solver(c["phys"], c["ndim"], c["integ"], GAMMA[c["phys"]], c["cfl"], [_domain(c)], glm_cr=GLM_CR,
                     recon=c["recon"])
    st = {"case": c, "solver": s, "U0": U0, "dt": s.dt(U0), "U": torch.empty_like(U0), "back": back}
    if c["tune"]:
        s.autotune(U0, st["dt"])
    if c["do"] in ("grad", "rollout"):  # the gradient that a loss sends back
        gen = torch.Generator(device="cuda").manual_seed(int(seed) + 1)
        st["g"] = torch.randn(U0.shape, generator=gen, device="cuda", dtype=torch.float64)
    return st


def run(st):
    c = st["case"]
    if c["do"] == "dt":
        return amrfd.dt_noalloc(MHD, 3, GAMMA[MHD], 0.4, st["domains"], st["U0"], st["dt"], active=st["active"])
    s = st["solver"]
    if c["do"] in ("grad", "rollout"):
        U = st["U0"].detach().requires_grad_()
        if c["do"] == "grad":
            new = autodiff.step(s, U, st["dt"])
        else:
            new = autodiff.rollout(s, U, st["dt"], c["steps"], c["every"])
        (g,) = torch.autograd.grad(new, U, st["g"])
        return {"U": new.detach(), "g": g}
    # a run starts from its initial state and keeps it
    U, dt = st["U"], st["dt"]
    U.copy_(st["U0"])
    if c["do"] == "activate":
        s.activate(s.flag_steady(U, st["back"], 1e-12), belt=2)
    if c["do"] != "run" or c["path"] == "graph":
        for _ in range(c.get("steps", 1)):
            s.dt(U, out=dt)
            s.step_batched(U, dt)
    elif c["path"] == "cfl":
        for _ in range(c["steps"]):
            s.step_cfl(U, out=dt)
    else:
        for _ in range(c["steps"]):
            s.step(U, s.dt(U, out=dt))
    return {"U": U, "dt": dt}


# -------------------------------------------------------------------- work
def _step_work(cells, nv, ndim, stages):
    """One step: the state in and out once, and the arithmetic of the scheme: per cell and
    direction the flux and its split, per face, variable and bias one reconstruction of
    eleven operations, per stage the combination."""
    flops = stages * cells * (ndim * (nv * (2 * 11 + 4) + 21) + 2 * nv * (ndim + 1))
    return {"bytes": 2 * 8 * nv * cells, "flops": flops}


def work(case):
    c = case
    if c["do"] in ("batch", "dt"):
        edges, _, active = _batch_sizes(c)
        cells = sum(m ** 3 for m, a in zip(edges, active.tolist()) if a)
        if c["do"] == "dt":
            return {"bytes": 72 * cells, "flops": 60 * cells}
        return _step_work(cells, 9, 3, 3)
    cells, nv = c["nx"] * c["ny"] * c["nz"], _nv(c)
    one = _step_work(cells, nv, c["ndim"], STAGES[c["integ"]])
    if c["do"] == "run":
        return {"bytes": c["steps"] * one["bytes"], "flops": c["steps"] * one["flops"]}
    if c["do"] == "activate":  # the state and the background once; about a sixth of the blocks advances
        return {"bytes": one["bytes"], "flops": one["flops"] // 6}
    # forward, and a reverse sweep of about twice its arithmetic; gradient in and out
    return {"bytes": 2 * one["bytes"] * c["steps"], "flops": 3 * one["flops"] * c["steps"]}


# ------------------------------------------------------------- the definition
def _minmod(a, b):
    return 0.5 * (torch.sign(a) + torch.sign(b)) * torch.minimum(a.abs(), b.abs())


def _mp5(a, b, c, d, e):
    """Suresh and Huynh's limited face value right of the centre cell c."""
    v = (2.0 * a - 13.0 * b + 47.0 * c + 27.0 * d - 3.0 * e) / 60.0
    ok = (v - c) * (v - c - _minmod(d - c, 4.0 * (c - b))) <= 1e-10
    km, k0, kp = a - 2.0 * b + c, b - 2.0 * c + d, c - 2.0 * d + e

    def m4(p, q):
        return _minmod(_minmod(4.0 * p - q, 4.0 * q - p), _minmod(p, q))
    ul, lc = c + 4.0 * (c - b), c + 0.5 * (c - b) + 4.0 / 3.0 * m4(km, k0)
    md = 0.5 * (c + d) - 0.5 * m4(k0, kp)
    lo = torch.maximum(torch.minimum(torch.minimum(c, d), md), torch.minimum(torch.minimum(c, ul), lc))
    hi = torch.minimum(torch.maximum(torch.maximum(c, d), md), torch.maximum(torch.maximum(c, ul), lc))
    med = torch.maximum(torch.minimum(v, lo), torch.minimum(torch.maximum(v, lo), hi))
    return torch.where(ok, v, med)


def _limo3(b, c, d, dx):
    """Cada and Torrilhon's limited face value right of the centre cell c (r = 1)."""
    dm, dp = c - b, d - c
    theta = dm / torch.where(dp == 0.0, torch.ones_like(dp), dp)
    p3 = (2.0 + theta) / 3.0
    lim = torch.clamp(torch.minimum(p3, torch.maximum(-0.5 * theta, torch.minimum(torch.minimum(2.0 * theta, p3),
                                                                                  torch.full_like(p3, 1.6)))), min=0.0)
    y3, yl = (2.0 * dp + dm) / 3.0, torch.where(dp == 0.0, torch.zeros_like(dp), dp * lim)
    eta = (dm * dm + dp * dp) / (dx * dx)
    z = (eta - 1.0) / 1e-12
    y = torch.where(z <= -1.0, y3, torch.where(z >= 1.0, yl, 0.5 * ((1.0 - z) * y3 + (1.0 + z) * yl)))
    return c + 0.5 * y


def _pad(U, dim, kind, odd):
    """Three ghost layers on both sides of `dim`."""
    n = U.shape[dim]
    if kind == "p":
        return torch.cat([U.narrow(dim, n - 3, 3), U, U.narrow(dim, 0, 3)], dim)
    if kind == "o":
        return torch.cat([U.narrow(dim, 0, 1)] * 3 + [U] + [U.narrow(dim, n - 1, 1)] * 3, dim)
    sg = torch.tensor([-1.0 if (odd >> v) & 1 else 1.0 for v in range(U.shape[1])], device=U.device,
                      dtype=U.dtype).view(1, -1, 1, 1, 1)
    return torch.cat([U.narrow(dim, 0, 3).flip(dim) * sg, U, U.narrow(dim, n - 3, 3).flip(dim) * sg], dim)


def _speeds(U, c):
    """|v_d| + fast (or sound) speed per direction, of states (D, nv, nz, ny, nx)."""
    g, nd = GAMMA[c["phys"]], c["ndim"]
    rho = U[:, 0]
    if c["phys"] == EULER:
        v = [U[:, 1 + k] / rho for k in range(nd)]
        p = (g - 1.0) * (U[:, -1] - 0.5 * rho * sum(q * q for q in v))
        return [q.abs() + torch.sqrt(g * p / rho) for q in v]
    v, B = [U[:, 1 + k] / rho for k in range(3)], [U[:, 5 + k] for k in range(3)]
    b2 = sum(q * q for q in B)
    a2 = g * (g - 1.0) * (U[:, 4] - 0.5 * rho * sum(q * q for q in v) - 0.5 * b2) / rho
    s = a2 + b2 / rho
    return [v[d].abs() + torch.sqrt(0.5 * (s + torch.sqrt(torch.clamp(s * s - 4.0 * a2 * B[d] * B[d] / rho, min=0.0))))
            for d in range(nd)]


def _flux(U, c, d, ch2):
    g, rho = GAMMA[c["phys"]], U[:, 0]
    if c["phys"] == EULER:
        m = [U[:, 1 + k] for k in range(c["ndim"])]
        v = m[d] / rho
        p = (g - 1.0) * (U[:, -1] - 0.5 * sum(q * q for q in m) / rho)
        return torch.stack([m[d]] + [v * q + (p if k == d else 0.0) for k, q in enumerate(m)] + [v * (U[:, -1] + p)], 1)
    v, B = [U[:, 1 + k] / rho for k in range(3)], [U[:, 5 + k] for k in range(3)]
    b2 = sum(q * q for q in B)
    pt = (g - 1.0) * (U[:, 4] - 0.5 * rho * sum(q * q for q in v) - 0.5 * b2) + 0.5 * b2
    vb = sum(p * q for p, q in zip(v, B))
    return torch.stack([U[:, 1 + d]] + [v[d] * U[:, 1 + k] - B[d] * B[k] + (pt if k == d else 0.0) for k in range(3)]
                       + [v[d] * (U[:, 4] + pt) - B[d] * vb]
                       + [U[:, 8] if k == d else v[d] * B[k] - B[d] * v[k] for k in range(3)]
                       + [ch2.view(-1, 1, 1, 1) * B[d]], 1)


def _residual(U, c, dx, alpha, ch2):
    """L(U) of states (D, nv, nz, ny, nx); dx, alpha: per domain and direction."""
    L = torch.zeros_like(U)
    for d in range(c["ndim"]):
        dim, n = 4 - d, U.shape[4 - d]
        P = _pad(U, dim, c["bc"][d], _walls(c, d))
        F, a = _flux(P, c, d, ch2), alpha[:, d].view(-1, 1, 1, 1, 1)
        G, h = 0.5 * (F + a * P), 0.5 * (F - a * P)
        h_ = dx[:, d].view(-1, 1, 1, 1, 1)

        def at(q, j):
            return q.narrow(dim, j, n + 1)
        if c["recon"] == MP5:
            f = _mp5(*(at(G, j) for j in range(5))) + _mp5(*(at(h, j) for j in (5, 4, 3, 2, 1)))
        else:
            f = _limo3(at(G, 1), at(G, 2), at(G, 3), h_) + _limo3(at(h, 4), at(h, 3), at(h, 2), h_)
        L = L - (f.narrow(dim, 1, n) - f.narrow(dim, 0, n)) / h_
    return L


TABLES = {  # per stage: ({state: weight}, {residual: weight}), residual k = L of state k
    RK3: [({0: 1.0}, {0: 1.0}), ({0: 0.75, 1: 0.25}, {1: 0.25}), ({0: 1.0 / 3.0, 2: 2.0 / 3.0}, {2: 2.0 / 3.0})],
    RK43: [({0: 1.0}, {0: 0.5}), ({1: 1.0}, {1: 0.5}), ({0: 2.0 / 3.0, 2: 1.0 / 3.0}, {2: 1.0 / 6.0}), ({3: 1.0}, {3: 0.5})],
    RK54: [({0: 1.0}, {0: 0.39175222700392}), ({0: 0.44437049406734, 1: 0.55562950593266}, {1: 0.36841059262959}),
           ({0: 0.62010185138540, 2: 0.37989814861460}, {2: 0.25189177424738}),
           ({0: 0.17807995410773, 3: 0.82192004589227}, {3: 0.54497475021237}),
           ({0: 0.00683325884039, 2: 0.51723167208978, 3: 0.12759831133288, 4: 0.34833675773694},
            {3: 0.08460416338212, 4: 0.22600748319395})],
}


def _maxima(U, c, live):
    """Largest speeds per domain and direction over the active cells, (D, ndim)."""
    with torch.no_grad():
        return torch.stack([torch.where(live, s, torch.zeros_like(s)).flatten(1).amax(1) for s in _speeds(U, c)], 1)


def _time_step(U, c, dx, live, cfl):
    if c["phys"] == MHD:
        return cfl / (_maxima(U, c, live).amax(1) * (1.0 / dx[:, :c["ndim"]]).sum(1))
    rate = sum(s / dx[:, d].view(-1, 1, 1, 1) for d, s in enumerate(_speeds(U, c)))
    return cfl / torch.where(live, rate, torch.zeros_like(rate)).flatten(1).amax(1)


def _step(U, c, dx, dt, live):
    """One SSPRK step; live: (D, nz, ny, nx), the cells of active blocks."""
    S, Ls = [U], []
    w, act = dt.view(-1, 1, 1, 1, 1), live.unsqueeze(1)
    every = bool(live.all())
    ch = None
    for a, b in TABLES[c["integ"]]:
        alpha = _maxima(S[-1], c, live)
        if c["phys"] == MHD:
            ch = alpha.amax(1) if ch is None else ch
            alpha = torch.maximum(alpha, ch.view(-1, 1))
        Ls.append(_residual(S[-1], c, dx, alpha, ch * ch if ch is not None else None))
        new = sum(x * S[k] for k, x in a.items()) + w * sum(x * Ls[k] for k, x in b.items())
        Ls[:3] = [None] * len(Ls[:3])  # no later stage needs them
        if len(S) == STAGES[c["integ"]] and c["phys"] == MHD:
            damp = torch.exp(-dt * ch / GLM_CR).view(-1, 1, 1, 1, 1)
            new = torch.cat([new[:, :8], new[:, 8:] * damp], 1)
        S.append(new if every else torch.where(act, new, U))
    return S[-1]


def _blocks_to_cells(c, flags):
    n = (c["nx"], c["ny"], c["nz"])
    f = flags.view(c["bz"], c["by"], c["bx"])
    for d, nb in enumerate((c["bx"], c["by"], c["bz"])):
        f = f.repeat_interleave(n[d] // nb, dim=2 - d)
    return f


def _belt(c, U, back):
    """Active blocks: those with a cell off the background, and two layers around them."""
    off = ((U - back).abs() > 1e-12).any(0).view(c["bz"], c["nz"] // c["bz"], c["by"], c["ny"] // c["by"], c["bx"],
                                                   c["nx"] // c["bx"])
    a = off.any(5).any(3).any(1)
    for _ in range(2):
        for d in range(3):
            a = a | a.roll(1, d) | a.roll(-1, d)
    return a


def exact(case, seed):
    c = dict(case)
    if c["do"] in ("batch", "dt"):
        edges, dxs, offs, active, U = _batch(c, seed)
        spec = {"phys": MHD, "ndim": 3, "bc": "ppp", "recon": MP5, "integ": RK3}
        dt = torch.full((len(edges),), math.inf, device="cuda", dtype=torch.float64)
        for m in sorted(set(edges)):
            sel = [i for i, e in enumerate(edges) if e == m and active[i]]
            for lo in range(0, len(sel), 128):
                at = sel[lo:lo + 128]
                ix = torch.tensor(at, device="cuda")
                where = torch.tensor([offs[i] for i in at], device="cuda").view(-1, 1) + torch.arange(9 * m ** 3, device="cuda")
                V = U[where].view(-1, 9, m, m, m)
                dx = torch.tensor([[dxs[i]] * 3 for i in at], device="cuda", dtype=torch.float64)
                live = torch.ones_like(V[:, 0], dtype=torch.bool)
                dt[ix] = _time_step(V, spec, dx, live, 0.4)
                if c["do"] == "batch":
                    U[where.reshape(-1)] = _step(V, spec, dx, dt[ix], live).reshape(-1)
        return dt if c["do"] == "dt" else {"U": U, "dt": dt}
    U0, back = _initial(c, seed)
    dx = torch.tensor([_spacing(c)], device="cuda", dtype=torch.float64)
    U = U0.unsqueeze(0)
    live = torch.ones_like(U[:, 0], dtype=torch.bool)
    if c["do"] in ("grad", "rollout"):
        gen = torch.Generator(device="cuda").manual_seed(int(seed) + 1)
        g = torch.randn(U0.shape, generator=gen, device="cuda", dtype=torch.float64)
        dt = _time_step(U, c, dx, live, c["cfl"])
        states = [U]
        with torch.no_grad():
            for _ in range(c["steps"]):
                states.append(_step(states[-1], c, dx, dt, live))
        back_g = g.unsqueeze(0)
        for s in reversed(states[:-1]):
            s = s.detach().requires_grad_()
            (back_g,) = torch.autograd.grad(_step(s, c, dx, dt, live), s, back_g)
        return {"U": states[-1][0], "g": back_g[0]}
    if c["do"] == "activate":
        live = _blocks_to_cells(c, _belt(c, U0, back)).unsqueeze(0)
    dt = None
    with torch.no_grad():
        for _ in range(c["steps"]):
            dt = _time_step(U, c, dx, live, c["cfl"])
            U = _step(U, c, dx, dt, live)
    return {"U": U[0], "dt": dt}
