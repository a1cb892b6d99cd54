"""Performance cases: what programs that use this framework have it do.

Each case is one pass through the public Python entry points (``Lattice``,
``Batch``, ``AdjointProblem``, ``BatchAdjointProblem``), over the range of
lattice sizes, storage types, boundary rules and directions that the
repository's tests and benchmark use: from a lattice that one launch hardly
fills to the 384^3 benchmark lattice, ragged sizes among them.

``exact`` restates every pass in plain FP64 torch (halfway and on-site walls,
Guo force, the discrete adjoint by automatic differentiation of the step).
"""

from __future__ import annotations

import math

import numpy as np
import torch

DEV = "cuda"

E = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
     (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (0, 1, 1), (0, -1, -1), (0, 1, -1),
     (0, -1, 1), (1, 0, 1), (-1, 0, -1), (-1, 0, 1), (1, 0, -1)]
W = [1.0 / 3.0] + [1.0 / 18.0] * 6 + [1.0 / 36.0] * 12
OPP = [E.index((-e[0], -e[1], -e[2])) for e in E]

WALLS = {"periodic": (False, False, False), "channel": (False, False, True),
         "duct": (False, True, True), "cavity": (True, True, True)}
DTYPE = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
ELEM = {"f32": 4, "f16": 2, "bf16": 2}

# Floating-point operations of one node update, of one reverse node update.
STEP_FLOPS, REVERSE_FLOPS = 230, 350

# A drawn case updates at most this many nodes (the largest listed one:
# 384^3, 20 steps), times its kind's cost.
MOST_UPDATES = 1.1e9


def listed():
    return [
        # the smallest calls: a program that looks at the flow after every
        # step of a small lattice
        dict(name="monitor 24x20x16 f32", kind="monitor", nx=24, ny=20, nz=16, storage="f32",
             geometry="cavity", onsite=False, force=False, tau=0.6, steps=1),
        # a small cavity (the tests' size) in chunks of many steps
        dict(name="cavity 32 f32", kind="steps", nx=32, ny=32, nz=32, storage="f32",
             geometry="cavity", onsite=False, force=False, tau=0.6, steps=200),
        # a lattice that fits the L2 cache (the benchmark sweep's smallest)
        dict(name="periodic 64 f32", kind="steps", nx=64, ny=64, nz=64, storage="f32",
             geometry="periodic", onsite=False, force=False, tau=0.8, steps=100),
        # ragged sizes: a forced channel with odd rows
        dict(name="channel 101x67x45 f32 force", kind="steps", nx=101, ny=67, nz=45,
             storage="f32", geometry="channel", onsite=False, force=True, tau=0.7, steps=50),
        # an ordinary cavity just above the L2 cache
        dict(name="cavity 128 f32", kind="steps", nx=128, ny=128, nz=128, storage="f32",
             geometry="cavity", onsite=False, force=False, tau=0.55, steps=100),
        # the benchmark's lattice and storage
        dict(name="periodic 384 f32", kind="steps", nx=384, ny=384, nz=384, storage="f32",
             geometry="periodic", onsite=False, force=False, tau=0.8, steps=20),
        # the same size, walled, with half the bytes per value
        dict(name="cavity 384 f16", kind="steps", nx=384, ny=384, nz=384, storage="f16",
             geometry="cavity", onsite=False, force=False, tau=0.55, steps=20),
        # the paper's own boundary rule, odd rows, BF16
        dict(name="onsite 193x160x129 bf16", kind="steps", nx=193, ny=160, nz=129,
             storage="bf16", geometry="cavity", onsite=True, force=False, tau=0.65, steps=20),
        # host buffers in and out, one step (the benchmark's end-to-end call)
        dict(name="host 256 f32", kind="host", nx=256, ny=256, nz=256, storage="f32",
             geometry="periodic", onsite=False, force=False, tau=0.8, steps=1),
        # many uneven cavities advanced together (the benchmark's batch)
        dict(name="batch 64 cavities", kind="batch", domains=64, low=16, high=96, steps=60),
        # optimisation over an initial velocity and a force: the benchmark's
        # adjoint lattice with a shorter horizon
        dict(name="adjoint 128 T60", kind="adjoint", nx=128, ny=128, nz=128,
             geometry="periodic", tau=0.7, steps=60, every=20),
        # the same for a batch of cavities
        dict(name="batch adjoint 32 T40", kind="batch_adjoint", domains=32, low=16, high=96,
             steps=40, every=20),
    ]


def _edge(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def draw(rng):
    kind = rng.choice(["steps", "steps", "steps", "steps", "monitor", "host", "batch",
                       "adjoint", "batch_adjoint"])
    if kind in ("batch", "batch_adjoint"):
        high = _edge(rng, 24, 96)
        steps = _edge(rng, 4, 60)
        domains = _edge(rng, 2, 64 if kind == "batch" else 32)
        c = dict(kind=kind, domains=domains, low=16, high=high, steps=steps)
        if kind == "batch_adjoint":
            c["steps"] = max(4, min(steps, 40))
            c["every"] = rng.randint(3, 20)
        return c
    if kind == "adjoint":
        n = [_edge(rng, 16, 128) for _ in range(3)]
        return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2],
                    geometry=rng.choice(["periodic", "channel", "cavity"]),
                    tau=round(rng.uniform(0.6, 1.0), 3), steps=_edge(rng, 6, 60),
                    every=rng.randint(3, 20))
    top = 256 if kind == "host" else 384
    n = [_edge(rng, 12, top) for _ in range(3)]
    storage = rng.choice(["f32", "f32", "f16", "bf16"])
    onsite = kind != "host" and rng.random() < 0.15
    geometry = "cavity" if onsite else rng.choice(["periodic", "channel", "duct", "cavity"])
    steps = 1 if kind == "monitor" else _edge(rng, 1, 200 if kind == "steps" else 8)
    steps = max(1, min(steps, int(MOST_UPDATES / (n[0] * n[1] * n[2]))))
    return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], storage=storage, geometry=geometry,
                onsite=onsite, force=rng.random() < 0.25,
                tau=round(rng.uniform(0.62 if onsite else 0.55, 1.0), 3), steps=steps)


# ------------------------------------------------------------------ inputs

def _modes(shape, gen, amp, terms=3):
    """A smooth random field of max |value| <= amp: products of sines with
    wave numbers 1..3 and random phases (FP32, on the GPU)."""
    nz, ny, nx = shape
    out = torch.zeros(shape, dtype=torch.float64, device=DEV)
    for _ in range(terms):
        k = gen.integers(1, 4, size=3)
        ph = gen.random(3)
        axes = [torch.sin(2 * math.pi * (int(k[a]) * torch.arange(n, dtype=torch.float64, device=DEV)
                                         / n + float(ph[a])))
                for a, n in enumerate((nz, ny, nx))]
        out += (amp / terms) * axes[0][:, None, None] * axes[1][None, :, None] * axes[2]
    return out.float()


def _vector(shape, gen, amp):
    return torch.stack([_modes(shape, gen, amp) for _ in range(3)])


def _lattice_inputs(case, seed):
    """Initial density and velocity, force and lid of a lattice case: a smooth
    flow as a program would start from or restart with."""
    gen = np.random.default_rng(seed)
    shape = (case["nz"], case["ny"], case["nx"])
    d = {"rho": 1.0 + _modes(shape, gen, 0.01), "u": _vector(shape, gen, 0.02), "force": None,
         "lid": None}
    if case.get("force"):
        d["force"] = _vector(shape, gen, 2e-6)
    if case["geometry"] in ("cavity", "duct"):
        d["lid"] = (float(np.float32(gen.uniform(0.03, 0.06))), 0.0, 0.0)
    return d


def _adjoint_inputs(case, seed):
    gen = np.random.default_rng(seed)
    shape = (case["nz"], case["ny"], case["nx"])
    return {"u0": _vector(shape, gen, 0.02), "F": _vector(shape, gen, 2e-6),
            "target": _vector(shape, gen, 0.02),
            "lid": (0.05, 0.0, 0.0) if case["geometry"] == "cavity" else None}


def _batch_geometry(case):
    """Uneven cavities: sizes belong to the case, not to the seed."""
    gen = np.random.default_rng(3)
    dims = gen.integers(case["low"], case["high"] + 1, size=(case["domains"], 3))
    tau = gen.uniform(0.55, 1.0, size=case["domains"]).astype(np.float32)
    lid = gen.uniform(0.02, 0.08, size=case["domains"]).astype(np.float32)
    return [tuple(int(v) for v in d) for d in dims], tau, lid


def _batch_fields(case, dims, seed, amp=0.02):
    """One velocity field per domain and their packed form."""
    gen = np.random.default_rng(seed)
    fields = [_vector((nz, ny, nx), gen, amp) for nx, ny, nz in dims]
    return fields, torch.cat([f.reshape(-1) for f in fields])


# ------------------------------------------------------------------ passes

def prepare(case, seed):
    kind = case["kind"]
    if kind in ("batch", "batch_adjoint"):
        from paper_1309_1983_gb300.adjoint import BatchAdjointProblem
        from paper_1309_1983_gb300.batch import Batch

        dims, tau, lid = _batch_geometry(case)
        b = Batch(np.array(dims), tau, lid)
        b.f_a.zero_()  # the gaps between domains, so that whole buffers compare
        b.f_b.zero_()
        _, u0 = _batch_fields(case, dims, seed)
        if kind == "batch":
            b.init_equilibrium(u0)
            return {"kind": kind, "batch": b, "steps": case["steps"]}
        _, target = _batch_fields(case, dims, seed + 1_000_003)
        return {"kind": kind, "problem": BatchAdjointProblem(b, case["steps"], K=case["every"]),
                "u0": u0, "F": torch.zeros_like(u0), "target": target}
    if kind == "adjoint":
        from paper_1309_1983_gb300.adjoint import AdjointProblem

        d = _adjoint_inputs(case, seed)
        p = AdjointProblem(case["nx"], case["ny"], case["nz"], case["tau"], case["steps"],
                           K=case["every"], walls=WALLS[case["geometry"]], lid=d["lid"])
        return {"kind": kind, "problem": p, "u0": d["u0"], "F": d["F"], "target": d["target"]}
    from paper_1309_1983_gb300.lattice import Lattice

    d = _lattice_inputs(case, seed)
    lat = Lattice(case["nx"], case["ny"], case["nz"], case["tau"], walls=WALLS[case["geometry"]],
                  lid=d["lid"], storage=case["storage"], force=bool(case["force"]),
                  onsite=bool(case["onsite"]))
    if d["force"] is not None:
        lat.force.copy_(d["force"])
    state = {"kind": kind, "lat": lat, "steps": case["steps"], "dtype": DTYPE[case["storage"]]}
    if kind == "host":
        state["u0"] = d["u"].cpu().pin_memory()
        state["rho"] = torch.empty(lat.shape, dtype=torch.float32).pin_memory()
        state["u"] = torch.empty((3,) + lat.shape, dtype=torch.float32).pin_memory()
    else:
        lat.init_equilibrium(rho=d["rho"], u=d["u"])
    return state


def _f(lat, dtype):
    """The current state, without the row padding (a view)."""
    lay = lat.layout
    buf, _ = lat.current_buffers()
    return buf.view(dtype)[: 19 * lay.plane].view(19, lat.nz, lat.ny, lay.pitch)[..., : lat.nx]


def run(state):
    kind = state["kind"]
    if kind == "batch":
        b = state["batch"]
        b.step(state["steps"])
        rho, u = b.moments()
        return {"f": b.current_buffers()[0].view(torch.float32), "rho": rho, "u": u}
    if kind in ("adjoint", "batch_adjoint"):
        loss, gu0, gF = state["problem"].loss_and_grad(state["u0"], state["F"], state["target"])
        return {"loss": loss, "grad_u0": gu0, "grad_F": gF}
    lat = state["lat"]
    if kind == "host":
        lat.run_host(state["u0"], state["steps"], state["rho"], state["u"])
        return {"rho": state["rho"], "u": state["u"]}
    if kind == "monitor":
        rho, u = lat.step_moments(state["steps"])
    else:
        lat.step(state["steps"])
        rho, u = lat.moments()
    return {"f": _f(lat, state["dtype"]), "rho": rho, "u": u}


# ------------------------------------------------------------------ figures

def work(case):
    kind, n = case["kind"], case["steps"]
    if kind in ("batch", "batch_adjoint"):
        cells = sum(nx * ny * nz for nx, ny, nz in _batch_geometry(case)[0])
    else:
        cells = case["nx"] * case["ny"] * case["nz"]
    if kind in ("adjoint", "batch_adjoint"):
        # u0, F (single lattice) and target in, both gradients out
        fields = 5 if kind == "adjoint" else 4
        return {"bytes": 12 * fields * cells, "flops": (STEP_FLOPS + REVERSE_FLOPS) * cells * n}
    if kind == "host":
        return {"bytes": 28 * cells, "flops": STEP_FLOPS * cells * n}
    elem = 4 if kind == "batch" else ELEM[case["storage"]]
    force = 12 if case.get("force") else 0
    # the state in, the state and the moments out
    return {"bytes": (2 * 19 * elem + 16 + force) * cells, "flops": STEP_FLOPS * cells * n}


def tolerance(case):
    # From the distances to FP64 seen over listed and drawn cases (2-norms):
    # up to 1.1e-6 for FP32 states after 100 steps and 8.2e-7 for gradients
    # after 60, sums of 32-bit values that another order rounds differently
    # over up to 200 steps; 4.0e-4 with FP16 and 2.4e-3 with BF16 storage,
    # which round the state at every step.
    storage = case.get("storage", "f32")
    return {"rel": {"f32": 1e-5, "f16": 2e-3, "bf16": 1.2e-2}[storage]}


# ------------------------------------------------------------------ FP64 restatement

def _equilibrium(rho, u):
    """Shifted equilibrium f^eq - w (19, nz, ny, nx)."""
    usq = 1.5 * (u * u).sum(0)
    out = []
    for e, w in zip(E, W):
        eu = sum(c * u[a] for a, c in enumerate(e) if c)
        if any(e):
            out.append(w * (rho - 1 + rho * (3 * eu + 4.5 * eu * eu - usq)))
        else:
            out.append(w * (rho - 1 - rho * usq))
    return torch.stack(out)


def _stream(f, walls, lid):
    """Pull with halfway bounce-back; the moving face is z = nz."""
    g = []
    for i, e in enumerate(E):
        v = torch.roll(f[i], shifts=(e[2], e[1], e[0]), dims=(0, 1, 2)) if any(e) else f[i]
        for a in range(3):  # x, y, then z: its lid term holds on the top edges too
            if walls[a] and e[a]:
                dim = 2 - a
                at = [slice(None)] * 3
                at[dim] = 0 if e[a] == 1 else v.shape[dim] - 1
                at = tuple(at)
                moved = 6 * W[i] * sum(e[b] * lid[b] for b in range(3)) \
                    if a == 2 and e[2] == -1 and lid is not None else 0.0
                v = v.clone() if v.requires_grad else v
                v[at] = f[OPP[i]][at] + moved
        g.append(v)
    return g


def _onsite(f, g, walls, lid, force):
    """On-site velocity walls (Hecht & Harting) on the pulled shifted values g,
    in place; f is the state that was pulled."""
    n = f.shape[:0:-1]  # nx, ny, nz
    options = [((0, 1, -1) if walls[a] else (0,)) for a in range(3)]
    for sx in options[0]:
        for sy in options[1]:
            for sz in options[2]:
                s = (sx, sy, sz)
                faces = sum(1 for v in s if v)
                if not faces:
                    continue
                at = []
                for a in (2, 1, 0):
                    at.append({1: slice(0, 1), -1: slice(n[a] - 1, n[a])}.get(s[a]) if s[a]
                              else (slice(1, n[a] - 1) if walls[a] else slice(None)))
                at = tuple(at)
                d = [v[at].clone() for v in g]
                F = [force[a][at] if force is not None else 0.0 for a in range(3)]
                unknown = [any(s[a] and e[a] == s[a] for a in range(3)) for e in E]
                if faces == 1:
                    a = [k for k in range(3) if s[k]][0]
                    u = lid if lid is not None and s == (0, 0, -1) else (0.0, 0.0, 0.0)
                    s0 = sum(d[i] for i, e in enumerate(E) if e[a] == 0)
                    sm = sum(d[i] for i, e in enumerate(E) if e[a] * s[a] < 0)
                    un = s[a] * u[a]
                    rho = 1.0 + (s0 + 2 * sm - 0.5 * s[a] * F[a] + un) / (1 - un)
                    j = [rho * u[k] - 0.5 * F[k] for k in range(3)]
                    N = [0.0 if k == a else
                         0.5 * sum(e[k] * d[i] for i, e in enumerate(E) if e[a] == 0 and e[k])
                         - j[k] / 3 for k in range(3)]
                    buried = []
                else:
                    at_in = []
                    for dim, a in enumerate((2, 1, 0)):
                        w = at[dim]
                        at_in.append(slice(w.start + s[a], w.stop + s[a]) if s[a] else w)
                    dr = sum(f[i][tuple(at_in)] for i in range(19))
                    j = [-0.5 * F[k] for k in range(3)]
                    p = [s[k] * j[k] for k in range(3)]
                    if faces == 3:
                        N = [s[k] * (sum(p) - 3 * p[k]) / 12 for k in range(3)]
                    else:
                        c = [k for k in range(3) if not s[k]][0]
                        a, b = [k for k in range(3) if s[k]]
                        N = [0.0] * 3
                        N[a] = s[a] * (p[b] - p[a]) / 18
                        N[b] = -s[b] * (p[b] - p[a]) / 18
                        plus = E.index(tuple(1 if k == c else 0 for k in range(3)))
                        N[c] = (d[plus] - d[OPP[plus]]) / 4 - j[c] / 12
                    buried = [i for i in range(19) if unknown[i] and unknown[OPP[i]]]
                for i, e in enumerate(E):
                    if unknown[i] and i not in buried:
                        ej = sum(e[k] * j[k] for k in range(3))
                        eN = sum(e[k] * N[k] for k in range(3))
                        d[i] = d[OPP[i]] + 6 * W[i] * ej - eN
                if buried:
                    rest = sum(d[i] for i in range(19) if i not in buried)
                    for i in buried:
                        d[i] = (dr - rest) / len(buried)
                for i in range(19):
                    if unknown[i]:
                        g[i][at] = d[i]


def _collide(g, omega, force):
    """BGK with the Guo force, on shifted values; a list of 19 fields."""
    dr = sum(g)
    rho = 1.0 + dr
    j = [sum(e[a] * v for e, v in zip(E, g) if e[a]) for a in range(3)]
    if force is not None:
        j = [j[a] + 0.5 * force[a] for a in range(3)]
    u = [c / rho for c in j]
    base = dr - 1.5 * sum(a * b for a, b in zip(j, u))
    k = 1.0 - 0.5 * omega
    uF = sum(u[a] * force[a] for a in range(3)) if force is not None else None
    out = []
    for e, w, v in zip(E, W, g):
        if any(e):
            ej = sum(c * j[a] for a, c in enumerate(e) if c)
            eq = w * (base + 3 * ej + 4.5 * ej * ej / rho)
        else:
            eq = w * base
        new = (1.0 - omega) * v + omega * eq
        if force is not None:
            s = -3 * uF
            if any(e):
                eF = sum(c * force[a] for a, c in enumerate(e) if c)
                s = s + 3 * eF + 9 * ej / rho * eF
            new = new + k * w * s
        out.append(new)
    return out


def _step(f, omega, walls, lid, force, onsite=False):
    if onsite:
        g = _stream(f, (False,) * 3, None)
        g[0] = g[0].clone()
        _onsite(f, g, walls, lid, force)
    else:
        g = _stream(f, walls, lid)
    return torch.stack(_collide(g, omega, force))


def _moments(f, force):
    rho = 1.0 + f.sum(0)
    j = torch.stack([sum(e[a] * f[i] for i, e in enumerate(E) if e[a]) for a in range(3)])
    if force is not None:
        j = j - 0.5 * force
    return rho, j / rho


def _loss_and_grad(u0, F, target, omega, walls, lid, steps):
    """Loss and gradients of one domain: states kept, one reverse step at a
    time by automatic differentiation."""
    u0 = u0.double().requires_grad_()
    F = F.double().requires_grad_()
    target = target.double()
    with torch.no_grad():
        states = [_equilibrium(torch.ones_like(u0[0]), u0)]
        for _ in range(steps):
            states.append(_step(states[-1], omega, walls, lid, F))
    f = states.pop().requires_grad_()
    _, u = _moments(f, F)
    loss = 0.5 * ((u - target) ** 2).sum()
    lam, gF = torch.autograd.grad(loss, (f, F))
    while len(states) > 0:
        f = states.pop().requires_grad_()
        lam, more = torch.autograd.grad(_step(f, omega, walls, lid, F), (f, F), lam)
        gF = gF + more
    f0 = _equilibrium(torch.ones_like(u0[0]), u0)
    (gu0,) = torch.autograd.grad(f0, u0, lam)
    return loss.detach(), gu0, gF


def exact(case, seed):
    kind, steps = case["kind"], case["steps"]
    if kind in ("batch", "batch_adjoint"):
        dims, tau, lid = _batch_geometry(case)
        fields, _ = _batch_fields(case, dims, seed)
        walls = (True, True, True)
        omegas = [1.0 / float(t) for t in tau]
        lids = [(float(v), 0.0, 0.0) for v in lid]
        if kind == "batch_adjoint":
            targets, _ = _batch_fields(case, dims, seed + 1_000_003)
            got = [_loss_and_grad(u, torch.zeros_like(u), t, om, walls, ld, steps)
                   for u, t, om, ld in zip(fields, targets, omegas, lids)]
            return {"loss": sum(g[0] for g in got),
                    "grad_u0": torch.cat([g[1].reshape(-1) for g in got]),
                    "grad_F": torch.cat([g[2].reshape(-1) for g in got])}
        fs, rhos, us = [], [], []
        for u, om, ld in zip(fields, omegas, lids):
            f = _equilibrium(torch.ones_like(u[0], dtype=torch.float64), u.double())
            for _ in range(steps):
                f = _step(f, om, walls, ld, None)
            rho, v = _moments(f, None)
            fs.append(torch.cat([f.reshape(-1), f.new_zeros(-f.numel() % 64)]))
            rhos.append(rho.reshape(-1))
            us.append(v.reshape(-1))
        return {"f": torch.cat(fs), "rho": torch.cat(rhos), "u": torch.cat(us)}
    omega = 1.0 / float(np.float32(case["tau"]))
    walls = WALLS[case["geometry"]]
    if kind == "adjoint":
        d = _adjoint_inputs(case, seed)
        loss, gu0, gF = _loss_and_grad(d["u0"], d["F"], d["target"], omega, walls, d["lid"], steps)
        return {"loss": loss, "grad_u0": gu0, "grad_F": gF}
    d = _lattice_inputs(case, seed)
    force = d["force"].double() if d["force"] is not None else None
    rho = torch.ones_like(d["rho"]) if kind == "host" else d["rho"]
    f = _equilibrium(rho.double(), d["u"].double())
    for _ in range(steps):
        f = _step(f, omega, walls, d["lid"], force, onsite=bool(case["onsite"]))
    rho, u = _moments(f, force)
    if kind == "host":
        return {"rho": rho.cpu(), "u": u.cpu()}
    return {"f": f, "rho": rho, "u": u}
