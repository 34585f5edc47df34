"""The work that users of the library have it do, as measurable cases: single-point forces, stretches of
velocity-Verlet dynamics, batches of replicas, differentiable trajectories and Hessian-vector products,
each through the public entry points of the binding and the C ABI.

Starting states are synthetic liquids: an FCC lattice of at least density 0.8 thinned at random to the
wanted density (so the cells' occupation fluctuates as a liquid's does), every site displaced at random as far
as a closest approach of 0.98 sigma allows, ids in lattice order, Gaussian velocities.

The mixed form computes its forces in FP32, so its outputs are returned as float32 (the accuracy that its user
has); the FP64 form's are returned as float64.  Positions are returned unwrapped (x + img L), or as the
displacement from the start where the entry point gives no image counts.
"""
import ctypes
import math
import random

import torch

from paper_1012_2677_gb300 import ljmd
from paper_1012_2677_gb300.autograd import trajectory_loss

DEV = "cuda"
RC = 2.5
FORMS = {"auto": ljmd.LJ_LIST_AUTO, "full": ljmd.LJ_LIST_FULL, "half": ljmd.LJ_LIST_HALF}
PREC = {"mixed": ljmd.LJ_MIXED, "fp64": ljmd.LJ_FP64}


def _md(name, n, steps, precision="mixed", rho=0.5, T=1.0, margin=0.5, dt=0.005, form="auto", every=1, speed=0.0):
    return dict(name=name, kind="md", n=n, steps=steps, precision=precision, rho=rho, T=T, margin=margin, dt=dt,
                form=form, every=every, speed=speed)


def listed():
    return [
        # the smallest call: one force evaluation of a few hundred particles (a Monte Carlo or
        # minimiser move, a unit cell); launches and host round trips are all of it
        dict(name="forces_500_mixed", kind="forces", n=500, precision="mixed", rho=0.5, margin=0.5, form="full"),
        # the small configuration of the benchmark (4,000 particles, 100 steps, energies every
        # step), in both forms: studies of many short runs of one small box
        _md("md_4k_mixed", 4000, 100),
        _md("md_4k_fp64", 4000, 100, "fp64"),
        # a mid-size box with an odd number of particles, as experiments with tens of thousands
        # of particles have
        _md("md_32k_mixed", 32003, 50, rho=0.6, T=1.2),
        # the paper's benchmark: 500,000 particles, r_s = 2.8, dt = 0.001, |v| = 0.9 in random
        # directions, no energies inside the run
        _md("md_500k_paper", 500000, 100, margin=0.3, dt=0.001, every=0, speed=0.9),
        # the 1M configuration in the FP64 form: reference trajectories
        _md("md_1m_fp64", 1048576, 10, "fp64"),
        # a dense liquid (rho 0.8, T 0.9), where the automatic list form takes the half list
        _md("md_2m_dense", 2000003, 20, rho=0.8, T=0.9),
        # the headline configuration: 16.4M particles, 20 steps
        _md("md_16m_mixed", 16384000, 20),
        # many independent replicas of uneven size, density and temperature (500 to 50,000 particles),
        # as parameter scans run them: 40 steps of 10-step graphs
        dict(name="batch_256", kind="batch", replicas=256, n_min=500, n_max=50000, steps=40, graph=10, margin=0.3,
             dt=0.004),
        # training through a trajectory: loss and gradients of 32,000 particles, 50 steps
        dict(name="grad_32k_mixed", kind="grad", n=32000, steps=50, n_pe=10, ckpt=10, precision="mixed", rho=0.6, T=1.2),
        # the same in the FP64 form at a tenth of the size, where gradients are being checked
        dict(name="grad_3k_fp64", kind="grad", n=3200, steps=50, n_pe=10, ckpt=10, precision="fp64", rho=0.6, T=1.2),
        # a Hessian-vector product at fixed positions (normal modes, implicit differentiation)
        dict(name="hvp_1m_mixed", kind="hvp", n=1048576, precision="mixed", rho=0.5, margin=0.5),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["md", "md", "md", "md", "forces", "batch", "grad", "hvp"])
    precision = rng.choice(["mixed", "mixed", "fp64"])
    rho = round(rng.uniform(0.3, 0.9), 3)
    T = round(rng.uniform(0.7, 1.5), 3)
    margin = rng.choice([0.3, 0.4, 0.5])
    if kind == "md":
        n = _log(rng, 500, 4000000 if precision == "mixed" else 1000000)
        top = max(10, min(100, (40000000 if precision == "mixed" else 8000000) // n))
        return dict(kind="md", n=n, steps=_log(rng, 5, top), precision=precision, rho=rho, T=T, margin=margin,
                    dt=rng.choice([0.002, 0.004, 0.005]), form=rng.choice(["auto", "auto", "full", "half"]),
                    every=rng.choice([0, 1, 1, 5]), speed=0.0)
    if kind == "forces":
        return dict(kind="forces", n=_log(rng, 500, 4000000), precision=precision, rho=rho, margin=margin,
                    form=rng.choice(["auto", "full", "half"]))
    if kind == "batch":
        lo = _log(rng, 500, 5000)
        return dict(kind="batch", replicas=_log(rng, 3, 256), n_min=lo, n_max=_log(rng, lo + 1, 50000),
                    steps=rng.randint(5, 40), graph=rng.choice([0, 5, 10]), margin=0.3, dt=0.004)
    if kind == "grad":
        n = _log(rng, 500, 50000 if precision == "mixed" else 5000)
        steps = rng.randint(5, 50)
        return dict(kind="grad", n=n, steps=steps, n_pe=rng.randint(1, steps), ckpt=rng.randint(2, 12),
                    precision=precision, rho=round(min(rho, 0.7), 3), T=T)
    return dict(kind="hvp", n=_log(rng, 500, 2000000 if precision == "mixed" else 300000), precision=precision, rho=rho,
                margin=margin)


# ---- inputs -----------------------------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) & ((1 << 62) - 1))
    return g


def _positions(n, rho, g):
    """(x[n, 3], L): the thinned and displaced FCC lattice."""
    L = (n / rho) ** (1.0 / 3.0)
    M = math.ceil((max(0.8, rho / 0.9) * L ** 3 / 4.0) ** (1.0 / 3.0))
    a = L / M
    k = torch.randperm(4 * M ** 3, generator=g, device=DEV)[:n].sort().values
    c, b = k // 4, k % 4
    cell = torch.stack([c // (M * M), (c // M) % M, c % M], 1).to(torch.float64)
    basis = torch.tensor([[0.0, 0.0, 0.0], [0.0, 0.5, 0.5], [0.5, 0.0, 0.5], [0.5, 0.5, 0.0]], dtype=torch.float64,
                         device=DEV)
    j = max(0.0, (a / math.sqrt(2.0) - 0.98) / (2.0 * math.sqrt(2.0)))
    u = torch.rand((n, 3), generator=g, dtype=torch.float64, device=DEV) * 2.0 - 1.0
    return torch.remainder((cell + basis[b] + 0.25) * a + j * u, L).contiguous(), L


def _velocities(n, T, g, speed=0.0):
    v = torch.randn((n, 3), generator=g, dtype=torch.float64, device=DEV)
    if speed > 0.0:
        return speed * v / v.norm(dim=1, keepdim=True)
    v = v - v.mean(0)
    return v * torch.sqrt(3.0 * max(n - 1, 1) * T / v.square().sum())


def _replicas(case, seed):
    """(n, box) lists and x, v of the replicas, concatenated.  The table of their sizes, densities and
    temperatures belongs to the case; the states come from the seed."""
    r = random.Random("%d %d %d" % (case["replicas"], case["n_min"], case["n_max"]))
    u = [(r.random(), r.random(), r.random()) for _ in range(case["replicas"])]
    g = _generator(seed)
    n = [case["n_min"] + int(a * (case["n_max"] - case["n_min"] + 1)) for a, _, _ in u]
    xs, vs, box = [], [], []
    for k, (_, b, c) in zip(n, u):
        x, L = _positions(k, 0.3 + 0.6 * b, g)
        xs.append(x)
        vs.append(_velocities(k, 0.7 + 0.8 * c, g))
        box.append(L)
    return n, box, torch.cat(xs), torch.cat(vs)


def _inputs(case, seed):
    g = _generator(seed)
    x, L = _positions(case["n"], case["rho"], g)
    if case["kind"] == "hvp":
        return x, torch.randn((case["n"], 3), generator=g, dtype=torch.float64, device=DEV), L
    if case["kind"] == "forces":
        return x, None, L
    return x, _velocities(case["n"], case["T"], g, case.get("speed", 0.0)), L


# ---- the measured pass --------------------------------------------------------------------------

def _system(case):
    return ljmd.System(cutoff=RC, margin=case["margin"], precision=PREC[case["precision"]],
                       list_form=FORMS[case.get("form", "full")], energy_every=case.get("every", 1),
                       stream=torch.cuda.current_stream())


def prepare(case, seed):
    if case["kind"] == "batch":
        n, box, x, v = _replicas(case, seed)
        b = ljmd.Batch(n, box, cutoff=RC, margin=case["margin"], stream=torch.cuda.current_stream())
        L = torch.repeat_interleave(torch.tensor(box, dtype=torch.float64, device=DEV),
                                    torch.tensor(n, device=DEV)).unsqueeze(1)
        return dict(case=case, b=b, x=x, v=v, L=L)
    x, v, L = _inputs(case, seed)
    if case["kind"] == "grad":
        eps, sigma = (torch.tensor(1.0, dtype=torch.float64, device=DEV, requires_grad=True) for _ in range(2))
        return dict(case=case, x=x.requires_grad_(), v=v.requires_grad_(), eps=eps, sigma=sigma, L=L)
    s = _system(case)
    if case["kind"] == "hvp":  # the positions are fixed; the products are taken at them
        s.set_state(x, None, L)
        s.build_pairlist()
    return dict(case=case, s=s, x=x, v=v, L=L)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        return _run_batch(state)
    x, v, L = state["x"], state["v"], state["L"]
    out = torch.float32 if case["precision"] == "mixed" else torch.float64
    if kind == "grad":
        loss = trajectory_loss(x, v, state["eps"], state["sigma"], L, dt=0.005, nsteps=case["steps"], n_pe=case["n_pe"],
                               ckpt_every=case["ckpt"], precision=PREC[case["precision"]])
        grads = torch.autograd.grad(loss, [x, v, state["eps"], state["sigma"]])
        return [t.to(out) for t in (loss.detach(), *grads)]
    s = state["s"]
    if kind == "hvp":
        hw = torch.empty_like(v)
        dtheta = ljmd.ljmd_hvp(s.h, v, hw)
        return dict(hw=hw.to(out), dtheta=[float(t) for t in dtheta])
    s.set_state(x, v, L)
    if kind == "forces":
        s.compute_forces()
        f = torch.empty_like(x)
        ljmd.ljmd_get_state(s.h, None, None, f, None, 1)
        pe, _, virial = s.energies()
        return dict(f=f.to(out), energy=[pe, virial])
    s.step(case["dt"], case["steps"])
    xo, vo, f = torch.empty_like(x), torch.empty_like(x), torch.empty_like(x)
    img = torch.empty(x.shape, dtype=torch.int32, device=DEV)
    ljmd.ljmd_get_state(s.h, xo, vo, f, img, 1)
    energy = list(s.energies())
    return dict(x=torch.add(xo, img, alpha=L).to(out), v=vo.to(out), f=f.to(out), energy=energy)


def _run_batch(state):
    case, b, x, v, L = state["case"], state["b"], state["x"], state["v"], state["L"]
    b.set_state(x, v)
    b.step(case["dt"], case["steps"], graph_steps=case["graph"])
    xo, vo, f = torch.empty_like(x), torch.empty_like(x), torch.empty_like(x)
    p = [ctypes.c_void_p(t.data_ptr()) for t in (xo, vo, f)]
    code = ljmd.load().ljmd_batch_get_state(b.h, *p, 1)
    if code != ljmd.LJ_OK:
        raise ljmd.LjmdError(code, "ljmd_batch_get_state")
    pe, ke, virial = b.energies()
    d = xo - x
    d = d - L * torch.round(d / L)
    e = torch.tensor([list(pe), list(ke), list(virial)], dtype=torch.float32)
    return dict(d=d.float(), v=vo.float(), f=f.float(), energy=e)


def work(case):
    """Inputs read once, outputs written once; the arithmetic of the pairs inside r_c (each once, 33
    operations with its energy and virial; 95 for an adjoint pair), per step where there are steps."""
    if case["kind"] == "batch":
        n, rho = case["replicas"] * (case["n_min"] + case["n_max"]) / 2.0, 0.6
    else:
        n, rho = case["n"], case["rho"]
    pairs = n * 2.0 * math.pi / 3.0 * RC ** 3 * rho
    if case["kind"] == "forces":
        return dict(bytes=48.0 * n, flops=33.0 * pairs)
    if case["kind"] == "hvp":
        return dict(bytes=72.0 * n, flops=95.0 * pairs)
    if case["kind"] == "grad":
        return dict(bytes=96.0 * n, flops=case["steps"] * pairs * (33.0 + 95.0))
    return dict(bytes=(48.0 + 72.0 + 12.0) * n, flops=case["steps"] * (33.0 * pairs + 30.0 * n))


# ---- the same in plain torch, 64 bits -----------------------------------------------------------

def _pairs(x, L, r):
    """Index pairs (i, j), each once, with minimum-image distance below r."""
    n = x.shape[0]
    m = int(L // r)
    if m < 3:
        i, j = torch.triu_indices(n, n, 1, device=DEV)
        d = x[j] - x[i]
        d = d - L * torch.round(d / L)
        keep = d.square().sum(1) < r * r
        return i[keep], j[keep]
    c = (torch.remainder(x, L) * (m / L)).long().clamp_(0, m - 1)
    cell = (c[:, 0] * m + c[:, 1]) * m + c[:, 2]
    order = cell.argsort()
    counts = torch.bincount(cell, minlength=m ** 3)
    start = counts.cumsum(0) - counts
    occ = int(counts.max())
    slot = torch.arange(n, device=DEV) - start[cell[order]]
    table = torch.full((m ** 3, occ), -1, dtype=torch.int64, device=DEV)
    table[cell[order], slot] = order
    forward = [(a, b, e) for a in (-1, 0, 1) for b in (-1, 0, 1) for e in (-1, 0, 1) if (a, b, e) >= (0, 0, 0)]
    out_i, out_j = [], []
    step = max(1, 40000000 // (occ * occ))
    for lo in range(0, m ** 3, step):
        k = torch.arange(lo, min(lo + step, m ** 3), device=DEV)
        cx, cy, cz = k // (m * m), (k // m) % m, k % m
        own = table[k]
        xi = x[own.clamp(min=0)]
        for a, b, e in forward:
            other = table[((cx + a) % m * m + (cy + b) % m) * m + (cz + e) % m]
            d = x[other.clamp(min=0)].unsqueeze(1) - xi.unsqueeze(2)
            d = d - L * torch.round(d / L)
            ok = (d.square().sum(3) < r * r) & (own >= 0).unsqueeze(2) & (other >= 0).unsqueeze(1)
            if (a, b, e) == (0, 0, 0):
                ok &= own.unsqueeze(2) < other.unsqueeze(1)
            q, p1, p2 = ok.nonzero(as_tuple=True)
            out_i.append(own[q, p1])
            out_j.append(other[q, p2])
    return torch.cat(out_i), torch.cat(out_j)


# Eq. 2's truncation constants at r_c / sigma = 2.5
C2 = 6.0 * RC ** -14 - 3.0 * RC ** -8
C0 = 4.0 * RC ** -6 - 7.0 * RC ** -12


def _pair_terms(x, i, j, L, eps=1.0, sigma=1.0):
    """(d, f, u) of the pairs inside r_c = 2.5 sigma: the force on i is f d (d = x_j - x_i), u the pair energy."""
    d = x[j] - x[i]
    d = d - L * torch.round(d / L).detach()
    r2 = d.square().sum(1)
    keep = (r2 < float(RC * sigma) ** 2).nonzero().squeeze(1)
    i, j, d, r2 = i[keep], j[keep], d[keep], r2[keep]
    s2 = sigma * sigma
    a3 = (s2 / r2) ** 3
    f = eps * ((24.0 * a3 - 48.0 * a3 * a3) / r2 + 8.0 * C2 / s2)
    u = 4.0 * eps * (a3 * a3 - a3 + C2 * r2 / s2 + C0)
    return i, j, d, r2, f, u


def _forces(x, i, j, L, chunk=50000000):
    F = torch.zeros_like(x)
    pe, vir = 0.0, 0.0
    for lo in range(0, i.shape[0], chunk):
        a, b, d, r2, f, u = _pair_terms(x, i[lo:lo + chunk], j[lo:lo + chunk], L)
        fd = f.unsqueeze(1) * d
        F.index_add_(0, a, fd)
        F.index_add_(0, b, -fd)
        pe += float(u.sum())
        vir -= float((f * r2).sum())
    return F, pe, vir


def _dynamics(x, v, L, dt, steps, skin=0.5):
    x, v = x.clone(), v.clone()
    ref, (i, j) = x.clone(), _pairs(x, L, RC + skin)
    F, pe, vir = _forces(x, i, j, L)
    for _ in range(steps):
        v += 0.5 * dt * F
        x += dt * v
        if float((x - ref).square().sum(1).max()) > (0.5 * skin) ** 2:
            ref, (i, j) = x.clone(), _pairs(x, L, RC + skin)
        F, pe, vir = _forces(x, i, j, L)
        v += 0.5 * dt * F
    return x, v, F, [pe, 0.5 * float(v.square().sum()), vir]


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        n, box, x, v = _replicas(case, seed)
        parts, at = [], 0
        for k, L in zip(n, box):
            xr, vr = x[at:at + k], v[at:at + k]
            xo, vo, F, e = _dynamics(xr, vr, L, case["dt"], case["steps"])
            parts.append((xo - xr, vo, F, e))
            at += k
        return dict(d=torch.cat([p[0] for p in parts]), v=torch.cat([p[1] for p in parts]),
                    f=torch.cat([p[2] for p in parts]),
                    energy=torch.tensor([p[3] for p in parts], dtype=torch.float64).T.contiguous())
    x, v, L = _inputs(case, seed)
    if kind == "md":
        xo, vo, F, e = _dynamics(x, v, L, case["dt"], case["steps"])
        return dict(x=xo, v=vo, f=F, energy=e)
    if kind == "forces":
        F, pe, vir = _forces(x, *_pairs(x, L, RC), L)
        return dict(f=F, energy=[pe, vir])
    one = lambda: torch.tensor(1.0, dtype=torch.float64, device=DEV, requires_grad=True)  # noqa: E731
    eps, sigma = one(), one()
    if kind == "hvp":
        x.requires_grad_()
        i, j, d, _, f, u = _pair_terms(x, *_pairs(x.detach(), L, RC), L, eps, sigma)
        wF = ((v[i] - v[j]) * d).sum(1).mul(f).sum()  # w . F
        gx, ge, gs = torch.autograd.grad(wF, [x, eps, sigma], retain_graph=True)
        pe, ps = torch.autograd.grad(u.sum(), [eps, sigma])
        return dict(hw=-gx, dtheta=[float(ge), float(gs), float(pe), float(ps)])
    x0, v0 = x.requires_grad_(), v.requires_grad_()
    n, dt, steps = case["n"], 0.005, case["steps"]
    x, v, loss = x0, v0, 0.0

    def force(x, ref):
        if float((x.detach() - ref[0]).square().sum(1).max()) > 0.25 ** 2:
            ref[0], ref[1] = x.detach().clone(), _pairs(x.detach(), L, RC + 0.5)
        i, j, d, _, f, u = _pair_terms(x, *ref[1], L, eps, sigma)
        fd = f.unsqueeze(1) * d
        return torch.zeros_like(x).index_add(0, i, fd).index_add(0, j, -fd), u.sum()

    ref = [x.detach().clone(), _pairs(x.detach(), L, RC + 0.5)]
    F, _ = force(x, ref)
    for t in range(1, steps + 1):
        v = v + 0.5 * dt * F
        x = x + dt * v
        F, u = force(x, ref)
        v = v + 0.5 * dt * F
        if t > steps - case["n_pe"]:
            loss = loss + u / (case["n_pe"] * n)
    loss = loss + (x - x0).square().sum() / n
    return [loss.detach(), *torch.autograd.grad(loss, [x0, v0, eps, sigma])]
