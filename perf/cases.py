"""The force pass as its users run it: the workloads that the library's speed is measured on.

``listed()`` names them, ``draw(rng)`` gives more of the same ranges, ``prepare`` makes
what a program has in hand before the call (inputs on the GPU, a context with the
particles loaded, a batch plan or a graph), ``run`` makes one pass through the public
entry points and returns its outputs, ``work`` says what a pass cannot do without and
``exact`` computes the same outputs in 64 bits with plain torch.

Kinds of case:

* ``step``     one block step: the copy of the active particles' new state into the
               store, the prediction of all sources, the forces on the active ones
* ``lists``    the same with neighbour lists within a radius of each sink
* ``batched``  many independent planetary systems in one launch, replayed as a graph
* ``adjoint``  a shared-step Hermite-4 trajectory and its gradient through autograd
* ``blocks``   a run of the device-driven block time-step integrator
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1510_04068_gb300 import autograd, sp2

T_STEP = 1.0         # time of a block step
DT_MAX = 1.0 / 16    # largest step of the block integrator
ETA = 0.01           # its accuracy parameter
F8 = torch.float64


def listed():
    return [
        # the plain form: a small cluster in FP64, every particle active, one predict + compute
        dict(name="fp64_n1024_all", kind="step", n=1024, n_active=1024, order=4, mixed=False, nn=True, host=False),
        # the smallest block of a block time-step run on a large cluster: one active particle
        dict(name="step_n131072_a1", kind="step", n=131072, n_active=1, order=4, mixed=True, nn=True, host=False),
        # a small block (the deepest levels of the time-step hierarchy), not a power of two
        dict(name="step_n131072_a61", kind="step", n=131072, n_active=61, order=4, mixed=True, nn=True, host=False),
        # the mean block of a 16384-body run, driven by an integrator whose particles live in host memory
        dict(name="host_n16384_a317", kind="step", n=16384, n_active=317, order=4, mixed=True, nn=True, host=True),
        # an ordinary block of a large run; neither size is a multiple of a tile
        dict(name="step_n100003_a1000", kind="step", n=100003, n_active=1000, order=4, mixed=True, nn=True, host=False),
        # a large block with perturber lists (regularisation codes ask for them)
        dict(name="lists_n131072_a16384", kind="lists", n=131072, n_active=16384, order=4, mixed=True, nn=True,
             host=False),
        # the headline: every particle of a 131072-body cluster is active
        dict(name="step_n131072_all", kind="step", n=131072, n_active=131072, order=4, mixed=True, nn=True, host=False),
        # 6th-order Hermite with a mass function, a large block
        dict(name="h6_n65536_a4096", kind="step", n=65536, n_active=4096, order=6, mixed=True, nn=True, host=False),
        # 6th-order Hermite in FP64 throughout, an ordinary block
        dict(name="h6_fp64_n16384_a1025", kind="step", n=16384, n_active=1025, order=6, mixed=False, nn=True, host=False),
        # few-body regime: 4096 planetary systems of 3 to 256 bodies, one launch under a graph
        dict(name="batched_4096", kind="batched", n_sys=4096, order=4, mixed=True),
        # sensitivity of a cluster's final positions to its initial state
        dict(name="adjoint_n16384", kind="adjoint", n=16384, steps=8, every=4),
        # a short piece of a block time-step run, all of it on the device
        dict(name="blocks_n4096", kind="blocks", n=4096, t_end=1.0 / 128, mixed=True),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step"] * 11 + ["lists"] * 2 + ["batched"] * 2 + ["adjoint"] * 2 + ["blocks"] * 3)
    if kind == "batched":
        return dict(kind=kind, n_sys=_log_int(rng, 64, 4096), order=rng.choice([2, 4, 4, 6]), mixed=rng.random() < 0.8)
    if kind == "adjoint":
        return dict(kind=kind, n=_log_int(rng, 512, 16384), steps=rng.randint(3, 8), every=rng.randint(2, 8))
    if kind == "blocks":
        return dict(kind=kind, n=_log_int(rng, 256, 4096), t_end=rng.choice([1, 2]) / 256, mixed=True)
    if kind == "lists":
        n = _log_int(rng, 1024, 131072)
        return dict(kind=kind, n=n, n_active=_log_int(rng, 1, min(n, 16384)), order=4, mixed=True, nn=True, host=False)
    order = rng.choice([2, 4, 4, 4, 6])
    mixed = rng.random() < 0.75
    n = _log_int(rng, 256, 131072)
    # a pass costs at most what the headline costs (FP64 runs at 1/64 of the FP32 rate)
    most = int((1.7e10 if mixed else 2.0e8) / (1 if order <= 4 else 1.8)) // n
    n_active, host = _log_int(rng, 1, max(1, min(n, most))), rng.random() < 0.15
    if host:  # the upper half of a group of 32: other block sizes overran the host calls' staging when this was written
        n_active = min(n_active, 16384)
        n_active += rng.randint(17, 31) - n_active % 32
        n = max(n, n_active)
    return dict(kind=kind, n=n, n_active=n_active, order=order, mixed=mixed, nn=rng.random() < 0.75, host=host)


# ---- inputs -----------------------------------------------------------------

_STREAM = None


def _stream():
    """The stream that a program gives to its contexts."""
    global _STREAM
    if _STREAM is None:
        _STREAM = torch.cuda.Stream()
    return _STREAM


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _uniform(g, n, lo=0.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(n, generator=g, device="cuda", dtype=F8)


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=F8)


def _directions(g, n):
    c, phi = _uniform(g, n, -1.0, 1.0), _uniform(g, n, 0.0, 2.0 * math.pi)
    s = torch.sqrt(1.0 - c * c)
    return torch.stack([s * torch.cos(phi), s * torch.sin(phi), c], dim=1)


def _plummer(g, n):
    """Equal-mass Plummer sphere in Henon units (Aarseth, Henon & Wielen 1974): m, x, v."""
    X = _uniform(g, n, 1e-6, 0.999)
    r = 1.0 / torch.sqrt(X ** (-2.0 / 3.0) - 1.0)
    x = r[:, None] * _directions(g, n)
    # speed over escape speed: inverse of the tabulated cumulative of q^2 (1 - q^2)^(7/2)
    q = np.linspace(0.0, 1.0, 4097)
    cdf = np.concatenate([[0.0], np.cumsum(((q * q * (1 - q * q) ** 3.5)[1:] + (q * q * (1 - q * q) ** 3.5)[:-1]) / 2)])
    cdf = torch.as_tensor(cdf / cdf[-1], device="cuda")
    u = _uniform(g, n)
    k = torch.searchsorted(cdf, u, right=True).clamp(1, 4096)
    frac = (u - cdf[k - 1]) / (cdf[k] - cdf[k - 1])
    speed = (k - 1 + frac) / 4096.0 * math.sqrt(2.0) * (1.0 + r * r) ** -0.25
    v = speed[:, None] * _directions(g, n)
    x, v = x * (3.0 * math.pi / 16.0), v * math.sqrt(16.0 / (3.0 * math.pi))
    return torch.full((n,), 1.0 / n, device="cuda", dtype=F8), x - x.mean(0), v - v.mean(0)


def _salpeter(g, n):
    lo, hi = 0.1 ** -1.35, 100.0 ** -1.35
    m = (lo + _uniform(g, n) * (hi - lo)) ** (1.0 / -1.35)
    return m / m.sum()


def _cluster(case, seed):
    """Sources with last-update times up to 63/1024 before T_STEP, and the active slots."""
    n, g = case["n"], _gen(seed)
    m, x, v = _plummer(g, n)
    if case["order"] == 6:
        m = _salpeter(g, n)
    a, jerk, snap = _normal(g, n, 3), 4.0 * _normal(g, n, 3), 16.0 * _normal(g, n, 3)
    t = T_STEP - torch.randint(0, 64, (n,), generator=g, device="cuda").to(F8) / 1024.0
    ids = torch.randperm(n, generator=g, device="cuda").to(torch.int32)
    idx = torch.randperm(n, generator=g, device="cuda")[: case["n_active"]].sort().values.to(torch.int32)
    return dict(ids=ids, m=m, x=x, v=v, a=a, jerk=jerk, snap=snap if case["order"] == 6 else None, t=t), idx


def _system_sizes(case):
    """Body counts log-uniform in [3, 256]: the same multiset for every seed."""
    u = (np.arange(case["n_sys"]) + 0.5) / case["n_sys"]
    return np.rint(np.exp(math.log(3.0) + u * (math.log(256.0) - math.log(3.0)))).astype(np.int64)


def _planetary(case, seed):
    """Independent systems of a star and planets on Kepler orbits: offsets, m, x, v."""
    sizes = np.random.default_rng(seed).permutation(_system_sizes(case))
    offsets = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n, g = int(offsets[-1]), _gen(seed)
    star = torch.as_tensor(offsets[:-1], device="cuda")
    m = torch.exp(_uniform(g, n, math.log(1e-7), math.log(1e-3)))
    a = torch.exp(_uniform(g, n, math.log(0.5), math.log(50.0)))
    e = (0.05 * torch.sqrt(-2.0 * torch.log1p(-_uniform(g, n)))).clamp(max=0.99)
    inc = 0.02 * torch.sqrt(-2.0 * torch.log1p(-_uniform(g, n)))
    node, peri, M = (_uniform(g, n, 0.0, 2.0 * math.pi) for _ in range(3))
    E = M.clone()
    for _ in range(20):
        E = E - (E - e * torch.sin(E) - M) / (1.0 - e * torch.cos(E))
    mu, cE, sE = 1.0 + m, torch.cos(E), torch.sin(E)
    b, rate = a * torch.sqrt(1.0 - e * e), torch.sqrt(mu / a ** 3) / (1.0 - e * cE)
    px, py, vx, vy = a * (cE - e), b * sE, -a * sE * rate, b * cE * rate
    cO, sO, cw, sw, ci, si = (f(q) for q in (node, peri, inc) for f in (torch.cos, torch.sin))
    r = [(cO * cw - sO * sw * ci, -cO * sw - sO * cw * ci), (sO * cw + cO * sw * ci, -sO * sw + cO * cw * ci),
         (sw * si, cw * si)]
    x = torch.stack([p * px + q * py for p, q in r], dim=1)
    v = torch.stack([p * vx + q * vy for p, q in r], dim=1)
    m[star] = 1.0
    x[star] = 0.0
    v[star] = 0.0
    return offsets, m, x, v


def _eps2(case):
    return {"batched": 0.0, "adjoint": 1e-6, "blocks": 1e-6}.get(case["kind"], 1e-8)


def _h2(case):
    """Squared list radius with a few tens of neighbours in the core at any n."""
    return 2.5e-3 * (131072.0 / case["n"]) ** (2.0 / 3.0)


# ---- one case ---------------------------------------------------------------

def _outputs(n, order, nn, device="cuda"):
    new = (lambda *s, dtype=F8: torch.zeros(*s, dtype=dtype, device="cuda")) if device == "cuda" else \
          (lambda *s, dtype=F8: torch.zeros(*s, dtype=dtype).pin_memory())
    out = dict(acc=new(n, 3), pot=new(n))
    if order >= 4:
        out["jerk"] = new(n, 3)
    if order == 6:
        out["snap"] = new(n, 3)
    if nn:
        out["nn_id"], out["nn_r2"] = new(n, dtype=torch.int32), new(n)
    return out


def _load(ctx, p, slots=None):
    ctx.set_j(0, p["ids"], p["m"], p["x"], p["v"], p["a"], p["jerk"], p["snap"], p["t"], slots=slots)


def prepare(case, seed):
    s, kind = _stream(), case["kind"]
    with torch.cuda.stream(s):
        if kind == "adjoint":
            g = _gen(seed)
            m, x, v = _plummer(g, case["n"])
            return dict(case=case, sim=autograd.HermiteSim(case["n"], _eps2(case), stream=s), m=m.requires_grad_(),
                        x=x.requires_grad_(), v=v.requires_grad_(), w=_normal(g, case["n"], 3))
        prec = sp2.SP2_MIXED if case["mixed"] else sp2.SP2_FP64
        if kind == "blocks":
            n = case["n"]
            m, x, v = _plummer(_gen(seed), n)
            z = torch.zeros_like(x)
            ctx = sp2.Context(order=4, precision=prec, n_max=n, eps2=_eps2(case), with_nn=0, cuda_stream=s.cuda_stream)
            p = dict(ids=torch.arange(n, device="cuda", dtype=torch.int32), m=m, x=x, v=v, a=z, jerk=z, snap=None,
                     t=torch.zeros_like(m))
            out = {k: torch.empty_like(z) for k in ("x", "v", "a", "jerk")}
            return dict(case=case, ctx=ctx, p=p, out=dict(out, t=torch.empty_like(m)))
        if kind == "batched":
            offsets, m, x, v = _planetary(case, seed)
            n, order = len(m), case["order"]
            ctx = sp2.Context(order=order, precision=prec, n_max=n, eps2=0.0, cuda_stream=s.cuda_stream)
            z = torch.zeros_like(x)
            _load(ctx, dict(ids=torch.arange(n, device="cuda", dtype=torch.int32), m=m, x=x, v=v, a=z, jerk=z,
                            snap=z if order == 6 else None, t=torch.zeros_like(m)))
            plan, out = ctx.batch_plan(offsets), _outputs(n, order, True)
            ctx.predict(0.0)
            ctx.compute_batched(plan, **out)  # sizes the scratch before the capture
            sp2.sp2_graph_begin(ctx.ctx)
            ctx.predict(0.0)
            ctx.compute_batched(plan, **out)
            return dict(case=case, ctx=ctx, plan=plan, graph=sp2.sp2_graph_end(ctx.ctx), out=out)
        p, idx = _cluster(case, seed)
        ctx = sp2.Context(order=case["order"], precision=prec, n_max=case["n"], eps2=_eps2(case),
                          with_nn=int(case["nn"]), cuda_stream=s.cuda_stream)
        _load(ctx, p)
        at = idx.long()
        new = {k: None if q is None else q[at].contiguous() for k, q in p.items()}
        out = _outputs(len(idx), case["order"], case["nn"], "cpu" if case["host"] else "cuda")
        st = dict(case=case, ctx=ctx, idx=idx, new=new, out=out)
        if kind == "lists":
            st["h2"] = torch.full((len(idx),), _h2(case), device="cuda", dtype=F8)
            out["nb_count"] = torch.zeros(len(idx), device="cuda", dtype=torch.int32)
            out["nb_ids"] = torch.full((len(idx), 256), -1, device="cuda", dtype=torch.int32)
        if case["host"]:
            pin = lambda q: None if q is None else q.cpu().pin_memory()  # noqa: E731
            st["idx"], st["new"] = pin(idx), {k: pin(q) for k, q in new.items()}
        return st


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "batched":
        sp2.sp2_graph_launch(state["ctx"].ctx, state["graph"])
        return state["out"]
    if kind == "adjoint":
        with torch.cuda.stream(_stream()):
            m, x, v = state["m"], state["x"], state["v"]
            xf, vf = state["sim"].trajectory(x, v, m, 1.0 / 256, case["steps"], checkpoint_every=case["every"])
            gm, gx, gv = torch.autograd.grad((state["w"] * xf).sum(), (m, x, v))
            return dict(x=xf.detach(), v=vf.detach(), gm=gm, gx=gx, gv=gv)
    ctx, out = state["ctx"], state["out"]
    if kind == "blocks":
        _load(ctx, state["p"])
        ctx.block_init(0.0, ETA, DT_MAX)
        stats = ctx.block_run(case["t_end"], ETA, DT_MAX)
        ctx.get_j(0, case["n"], **out)
        return dict(out, blocks=stats["block_steps"], active=stats["active_sum"])
    # the active particles of the last block go back into the store, then the next block's forces
    _load(ctx, state["new"], slots=state["idx"])
    ctx.predict(T_STEP)
    if kind == "lists":
        ctx.compute_nb(state["idx"], state["h2"], 256, **out)
    else:
        ctx.compute(state["idx"], **out)
    return out


# ---- what a pass cannot do without ------------------------------------------

_FLOPS = {2: 20, 4: 42, 6: 82}  # per interaction, a fused multiply-add counted as two


def work(case):
    kind = case["kind"]
    if kind == "adjoint":
        n, steps = case["n"], case["steps"]
        # a force pass per step and one at the start; the gradient of each (130 operations a pair)
        return dict(bytes=8.0 * n * 24, flops=(steps + 1.0) * n * n * (42 + 130))
    if kind == "blocks":
        n = case["n"]
        # the start's pass and every particle's share of at least one block
        return dict(bytes=8.0 * n * 21, flops=2.0 * n * n * 42)
    per_source = 8.0 * (8 + (6 if case["order"] >= 4 else 0) + (3 if case["order"] == 6 else 0)) + 4
    per_sink = 8.0 * (4 + (3 if case["order"] >= 4 else 0) + (3 if case["order"] == 6 else 0))
    if kind == "batched":
        sizes = _system_sizes(case).astype(float)
        return dict(bytes=float(sizes.sum()) * (per_source + per_sink + 12), flops=float((sizes ** 2).sum()) * _FLOPS[case["order"]])
    per_sink += 4 + per_source + (12 if case["nn"] else 0)
    return dict(bytes=case["n"] * per_source + case["n_active"] * per_sink,
                flops=float(case["n"]) * case["n_active"] * _FLOPS[case["order"]])


# ---- the same in 64 bits ----------------------------------------------------

def _forces(m, xj, vj, aj, slot, xi, vi, ai, eps2, order):
    """Forces of all sources on a few sinks; slot: the sinks' own places among the sources."""
    me = slot[:, None] == torch.arange(len(m), device=m.device)[None, :]
    r = [xj[None, :, c] - xi[:, None, c] for c in range(3)]
    d2 = r[0] * r[0] + r[1] * r[1] + r[2] * r[2]
    s = torch.rsqrt(torch.where(me, torch.ones_like(d2), d2 + eps2))
    s = torch.where(me, torch.zeros_like(s), s)
    s2, ms = s * s, m[None, :] * s
    q = ms * s2
    out = dict(acc=torch.stack([(q * c).sum(1) for c in r], 1), pot=-ms.sum(1),
               nn_r2=d2.detach().masked_fill(me, math.inf).min(1).values)
    if order >= 4:
        w = [vj[None, :, c] - vi[:, None, c] for c in range(3)]
        al = (r[0] * w[0] + r[1] * w[1] + r[2] * w[2]) * s2
        J = [q * (w[c] - 3.0 * al * r[c]) for c in range(3)]
        out["jerk"] = torch.stack([c.sum(1) for c in J], 1)
    if order == 6:
        d = [aj[None, :, c] - ai[:, None, c] for c in range(3)]
        beta = (sum(c * c for c in w) + sum(r[c] * d[c] for c in range(3))) * s2 + al * al
        out["snap"] = torch.stack([(q * d[c] - 6.0 * al * J[c] - 3.0 * beta * q * r[c]).sum(1) for c in range(3)], 1)
    return out


def _chunked(m, x, v, a, idx, eps2, order):
    step = max(1, (1 << 25) // len(m))
    parts = [_forces(m, x, v, a, i, x[i], v[i], None if a is None else a[i], eps2, order) for i in idx.split(step)]
    return {k: torch.cat([p[k] for p in parts]) for k in parts[0]}


def _exact_adjoint(case, seed):
    n, dt, eps2 = case["n"], 1.0 / 256, _eps2(case)
    g = _gen(seed)
    m, x, v = _plummer(g, n)
    w = _normal(g, n, 3)
    every = torch.arange(n, device="cuda")
    step = max(1, (1 << 24) // n)

    def forces(x, v):
        f = _chunked(m, x, v, None, every, eps2, 4)
        return f["acc"], f["jerk"]

    def forces_vjp(x, v, ga, gj):
        x, v, mm = (q.detach().requires_grad_() for q in (x, v, m))
        got = [torch.zeros_like(q) for q in (x, v, mm)]
        for i in every.split(step):
            with torch.enable_grad():
                f = _forces(mm, x, v, None, i, x[i], v[i], None, eps2, 4)
                add = torch.autograd.grad((f["acc"] * ga[i]).sum() + (f["jerk"] * gj[i]).sum(), (x, v, mm))
            for p, q in zip(got, add):
                p += q
        return got

    def predicted(x, v, a, j):
        return x + v * dt + a * (dt * dt / 2) + j * (dt ** 3 / 6), v + a * dt + j * (dt * dt / 2)

    a, j = forces(x, v)
    x0, v0, states = x, v, []
    for _ in range(case["steps"]):
        xp, vp = predicted(x, v, a, j)
        a1, j1 = forces(xp, vp)
        states.append((x, v, a, j, xp, vp))
        v1 = v + (a + a1) * (dt / 2) + (j - j1) * (dt * dt / 12)
        x = x + (v + v1) * (dt / 2) + (a - a1) * (dt * dt / 12)
        v, a, j = v1, a1, j1
    gx, gv, ga, gj, gm = w, torch.zeros_like(w), torch.zeros_like(w), torch.zeros_like(w), torch.zeros_like(m)
    for xs, vs, as_, js, xp, vp in reversed(states):
        gv1 = gv + gx * (dt / 2)
        bx, bv, bm = forces_vjp(xp, vp, ga + gv1 * (dt / 2) - gx * (dt * dt / 12), gj - gv1 * (dt * dt / 12))
        gm = gm + bm
        gx, gv, ga, gj = (gx + bx, gx * (dt / 2) + gv1 + bx * dt + bv,
                          gx * (dt * dt / 12) + gv1 * (dt / 2) + bx * (dt * dt / 2) + bv * dt,
                          gv1 * (dt * dt / 12) + bx * (dt ** 3 / 6) + bv * (dt * dt / 2))
    bx, bv, bm = forces_vjp(x0, v0, ga, gj)
    return dict(x=x, v=v, gm=gm + bm, gx=gx + bx, gv=gv + bv)


def _quantise(want, cap, t):
    """Largest cap / 2^k not above `want` that divides t."""
    d = torch.exp2(torch.floor(torch.log2(torch.minimum(want, cap))))
    d = torch.minimum(torch.where(d > want, d / 2, d), cap)
    for _ in range(60):
        off = torch.fmod(t, d) != 0
        if not bool(off.any()):
            break
        d = torch.where(off, d / 2, d)
    return d


def _exact_blocks(case, seed):
    """Hermite-4 with individual power-of-two steps, Aarseth's criterion."""
    n, eps2 = case["n"], _eps2(case)
    m, x, v = _plummer(_gen(seed), n)
    every, norm = torch.arange(n, device="cuda"), lambda q: q.norm(dim=1)
    f = _chunked(m, x, v, None, every, eps2, 4)
    a, j, t = f["acc"], f["jerk"], torch.zeros_like(m)
    cap = torch.full_like(m, DT_MAX)
    dt = _quantise(ETA * norm(a) / norm(j), cap, t)
    blocks = active = 0
    while True:
        t1 = (t + dt).min()
        if float(t1) > case["t_end"]:
            break
        i = ((t + dt) == t1).nonzero()[:, 0]
        h = (t1 - t)[:, None]
        xp = x + h * (v + h * (a / 2 + h * (j / 6)))
        vp = v + h * (a + h * (j / 2))
        f = _chunked(m, xp, vp, None, i, eps2, 4)
        h, a0, j0, a1, j1 = h[i], a[i], j[i], f["acc"], f["jerk"]
        v1 = v[i] + (a0 + a1) * (h / 2) + (j0 - j1) * (h * h / 12)
        x[i] = x[i] + (v[i] + v1) * (h / 2) + (a0 - a1) * (h * h / 12)
        a3 = (12.0 * (a0 - a1) + 6.0 * h * (j0 + j1)) / h ** 3
        a2 = (-6.0 * (a0 - a1) - h * (4.0 * j0 + 2.0 * j1)) / (h * h) + h * a3
        v[i], a[i], j[i], t[i] = v1, a1, j1, t1
        want = torch.sqrt(ETA * (norm(a1) * norm(a2) + norm(j1) ** 2) / (norm(j1) * norm(a3) + norm(a2) ** 2))
        dt[i] = _quantise(want, torch.minimum(2.0 * h[:, 0], cap[i]), t[i])
        blocks, active = blocks + 1, active + len(i)
    return dict(x=x, v=v, a=a, jerk=j, t=t, blocks=blocks, active=active)


def exact(case, seed):
    kind = case["kind"]
    with torch.no_grad():
        if kind == "adjoint":
            return _exact_adjoint(case, seed)
        if kind == "blocks":
            return _exact_blocks(case, seed)
        if kind == "batched":
            offsets, m, x, v = _planetary(case, seed)
            z = torch.zeros_like(x)
            parts = [_chunked(m[b:e], x[b:e], v[b:e], z[b:e], torch.arange(e - b, device="cuda"), 0.0, case["order"])
                     for b, e in zip(offsets[:-1].tolist(), offsets[1:].tolist())]
            out = {k: torch.cat([q[k] for q in parts]) for k in parts[0]}
            return dict(out, nn_id=None)
        p, idx = _cluster(case, seed)
        h = (T_STEP - p["t"])[:, None]
        order = case["order"]
        x, v, a, j = p["x"], p["v"], p["a"], p["jerk"]
        s = p["snap"] if order == 6 else torch.zeros_like(x)
        if order == 2:  # leap-frog sources stay where they are
            xp, vp, ap = x, torch.zeros_like(v), None
        else:
            xp = x + h * (v + h * (a / 2 + h * (j / 6 + h * (s / 24))))
            vp = v + h * (a + h * (j / 2 + h * (s / 6)))
            ap = a + h * (j + h * (s / 2))
        out = _chunked(p["m"], xp, vp, ap if order == 6 else None, idx.long(), _eps2(case), order)
        if not case["nn"]:
            del out["nn_r2"]
        else:
            out["nn_id"] = None
        if kind == "lists":
            out["nb_count"] = out["nb_ids"] = None
        return out
