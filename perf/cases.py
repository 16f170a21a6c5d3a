"""The measured work of the library: what a program that steps granular scenes asks of it.

A case is one kind of call (`path`) at one size.  Scenes are jittered lattices of
spheres on a floor (one radius, or radii drawn from [0.4, 0.6] with a contact
envelope) and spheres falling in a walled box, as in the `synth` package; QTT
matrices are random cores of given rank.  All inputs are drawn on the device from
the seed alone.  `exact` restates each path in float64 torch, without the library.

Iterative solves run to a relative residual of 1e-12, so that a result is the
solution of the system and not of the place where an iteration happened to stop.
"""
from __future__ import annotations

import math

import torch

from paper_1808_02558_gb300 import binding, workload

DT = 1e-3
MU = 0.5
GRAVITY = (0.0, 0.0, -9.81)
TOL = 1e-12
FEAT_SCALE = (1.0, 1.0, 1.0, 5e-3, 2.0, 2.0, 2.0, 1.0)
NET_SHAPES = [(64, 8), (64,)] + [(64, 128), (64,)] * 3 + [(3, 64), (3,)]
CORE = {"f64": binding.QP_F64, "f32": binding.QP_F32, "bf16": binding.QP_BF16}


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # contact detection of a time step: 64 000 spheres of several radii
        dict(name="assemble_pile40p", path="assemble", scene="poly", n=40),
        # one operator product, FP32, as a caller's own Krylov loop makes it
        dict(name="apply_f32_pile40p", path="apply", scene="poly", n=40, slots=3, dtype="f32"),
        # the same in FP64 at an odd, medium size
        dict(name="apply_f64_pile21", path="apply", scene="mono", n=21, slots=3, dtype="f64"),
        # a small scene's Newton system, FP64 throughout: latency and barriers
        dict(name="solve_f64_pile8", path="solve", scene="mono", n=8, mixed=0),
        # the large pile's Newton system, FP32 iterations refined in FP64
        dict(name="solve_mixed_pile40p", path="solve", scene="poly", n=40, mixed=1),
        # a whole time step in the walled box: contacts, warm start, PDIP, advance
        dict(name="step_box40", path="step", scene="box", n=40, iters=3),
        # a PDIP iteration that rebuilds its QTT preconditioner (rank <= 10) and uses it
        dict(name="pdip_qtt_pile40p", path="pdip_qtt", scene="poly", n=40, eps=1e-2, rmax=10),
        # a small QTT product in FP64: launches and latency
        dict(name="qtt_f64_d12_r10", path="qtt", d=12, rank=10, core="f64"),
        # the preconditioner's product at the large pile's size (BF16 cores, rank 10)
        dict(name="qtt_bf16_d20_r10", path="qtt", d=20, rank=10, core="bf16"),
        # a high-rank QTT product: dense enough for the tensor cores
        dict(name="qtt_bf16_d20_r64", path="qtt", d=20, rank=64, core="bf16"),
        # a batch of small scenes of mixed sizes solved together
        dict(name="batched_256", path="batched", scenes=256, lo=4, hi=16),
        # training of the learned warm start: loss and gradient over one large scene
        dict(name="net_grad_pile40p", path="net", scene="poly", n=40, grad=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["assemble", "apply", "solve", "solve", "step", "pdip_qtt", "qtt", "qtt", "batched", "net"])
    scene = rng.choice(["mono", "poly", "box"])
    if path == "assemble":
        return dict(path=path, scene=scene, n=_log_int(rng, 5, 40))
    if path == "apply":
        return dict(path=path, scene=scene, n=_log_int(rng, 5, 40), slots=rng.choice([3, 3, 4]),
                    dtype=rng.choice(["f32", "f64"]))
    if path == "solve":
        mixed = rng.choice([0, 1])
        return dict(path=path, scene=rng.choice(["mono", "poly"]), mixed=mixed,
                    n=_log_int(rng, 10, 40) if mixed else _log_int(rng, 4, 20))
    if path == "step":
        return dict(path=path, scene=scene, n=_log_int(rng, 8, 40), iters=rng.choice([1, 2, 3]))
    if path == "pdip_qtt":
        return dict(path=path, scene=rng.choice(["mono", "poly"]), n=_log_int(rng, 8, 40), eps=1e-2,
                    rmax=rng.choice([6, 8, 10]))
    if path == "qtt":
        core = rng.choice(["f64", "f32", "bf16", "bf16"])
        if core == "f64":
            return dict(path=path, d=rng.randint(6, 17), rank=_log_int(rng, 2, 24), core=core)
        return dict(path=path, d=rng.randint(9, 20), rank=_log_int(rng, 2, 64 if core == "bf16" else 24), core=core)
    if path == "batched":
        lo = rng.randint(3, 8)
        return dict(path=path, scenes=_log_int(rng, 6, 256), lo=lo, hi=lo + rng.randint(0, 16 - lo))
    return dict(path=path, scene=scene, n=_log_int(rng, 6, 40), grad=rng.choice([True, False]))


# ------------------------------------------------------------------ inputs
def _generator(seed, tag):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1009 + tag)
    return g


def _uniform(g, *shape):
    return torch.rand(*shape, generator=g, dtype=torch.float64, device="cuda")


def _scene(kind, n, seed, mu=MU, tag=0):
    """Device tensors of one scene in the library's layout, and its scalars.

    The packing (jitter and radii) belongs to the case, so that every seed has the
    same number of contacts; the seed draws the velocities and where in space the
    packing stands."""
    g = _generator(101 * n + len(kind), 1 + 16 * tag)
    site = torch.arange(n, dtype=torch.float64, device="cuda")
    k, j, i = torch.meshgrid(site, site, site, indexing="ij")
    site = torch.stack([i.reshape(-1), j.reshape(-1), k.reshape(-1)])
    M = n * n * n
    walls, delta = (), 0.0
    if kind == "box":
        clear = 0.61
        stag = 0.8 * torch.remainder(site[0] + site[1], 2.0)
        at = clear + site * ((n - 2.0 * clear) / (n - 1))
        at[2] = clear + 2.0 * site[2] + stag
        delta = 0.25
    else:
        at = 0.98 * site
        at[2] += 0.49
        delta = 0.21 if kind == "poly" else 0.0
    pos = at + 0.01 * (2.0 * _uniform(g, 3, M) - 1.0)
    if kind == "mono":
        radius = torch.full((M,), 0.5, dtype=torch.float64, device="cuda")
    else:
        radius = 0.4 + 0.2 * _uniform(g, M)
    g = _generator(seed, 8 + 16 * tag)
    shift = 10.0 * _uniform(g, 3, 1)
    shift[2] = 0.0
    pos = (pos + shift).contiguous()
    if kind == "box":
        x, y = float(shift[0]), float(shift[1])
        walls = ((0, 1, x), (0, -1, x + n), (1, 1, y), (1, -1, y + n))
    vel = 0.1 * torch.randn(3, M, generator=g, dtype=torch.float64, device="cuda")
    mass = (4.0 / 3.0) * math.pi * radius ** 3
    dev = dict(pos=pos, vel=vel, omega=torch.zeros_like(vel), radius=radius, inv_mass=1.0 / mass,
               inv_inertia=1.0 / (0.4 * mass * radius * radius))
    return dict(dev=dev, delta=delta, walls=walls, mu=mu)


def _assemble(ctx, sc, slots=3):
    return ctx.assemble(sc["dev"], 0.0, GRAVITY, DT, sc["delta"], sc["mu"], slots, sc["walls"])


def _iterate(Nc, mu, seed, tag=0):
    """A PDIP iterate inside the cones: compact gamma (Nc, 3) and lambda (2 Nc), off the centre by up to a factor of two."""
    g = _generator(seed, 2 + 16 * tag)
    u = _uniform(g, 5, Nc)
    gn = 0.5 + u[0]
    rad, ang = 0.8 * mu * gn * torch.sqrt(u[1]), 2.0 * math.pi * u[2]
    gamma = torch.stack([gn, rad * torch.cos(ang), rad * torch.sin(ang)], 1)
    f = _constraints(gamma, mu)
    return gamma, -(0.5 + torch.cat([u[3], u[4]])) / f


def _barrier(gamma, lam, mu):
    """The barrier parameter that the library takes at an iterate: 10 times the constraints over their surrogate gap."""
    return 20.0 * gamma.shape[0] / float(-(_constraints(gamma, mu) * lam).sum())


def _pad(x, slots, P):
    out = torch.zeros(P, dtype=x.dtype, device="cuda")
    out[:slots * x.shape[0]].view(-1, slots)[:, :3] = x
    return out


def _cores(case, seed):
    """Random cores whose product keeps a vector's size; ranks no larger than a core's place allows."""
    d, r = case["d"], case["rank"]
    ranks = [min(r, 4 ** min(k, d - k)) for k in range(d + 1)]
    g = torch.Generator()
    g.manual_seed(int(seed) * 1009 + 3)
    return [torch.randn(ranks[k], 4, ranks[k + 1], generator=g, dtype=torch.float64) / math.sqrt(2 * ranks[k + 1])
            for k in range(d)]


def _vector(case, seed):
    dt = torch.float64 if case["core"] == "f64" else torch.float32
    return torch.randn(1 << case["d"], generator=_generator(seed, 4), dtype=torch.float64, device="cuda").to(dt)


def _net_inputs(Nc, seed):
    g = torch.Generator()
    g.manual_seed(int(seed) * 1009 + 5)
    parts = [torch.randn(s, generator=g, dtype=torch.float64).reshape(-1) * math.sqrt(2.0 / s[1]) if len(s) == 2
             else 0.05 * torch.randn(s, generator=g, dtype=torch.float64) for s in NET_SHAPES]
    # messages add up about six neighbours, so the hidden layers keep their size with a smaller second half
    for k in (2, 4, 6):
        parts[k].view(64, 128)[:, 64:] *= 0.2
    params = torch.cat(parts).to(torch.float32).cuda()
    target = torch.randn(3 * Nc, generator=_generator(seed, 6), dtype=torch.float64, device="cuda").to(torch.float32)
    return params, target


def _batch_sides(case):
    lo, hi = case["lo"], case["hi"]
    return [lo + (7 * i) % (hi - lo + 1) for i in range(case["scenes"])]


def _batch_mu(i):
    return 0.2 + 0.6 * ((13 * i) % 97) / 96.0


def _prev_positions(sc):
    """The scene one step earlier: the bodies came from here with their velocity."""
    dev = dict(sc["dev"])
    dev["pos"] = (dev["pos"] - 10.0 * DT * dev["vel"]).contiguous()
    return dict(sc, dev=dev)


# ------------------------------------------------------------------ prepare
def prepare(case, seed):
    path = case["path"]
    s = dict(case=case, path=path, ctx=binding.Context())
    ctx = s["ctx"]
    if path == "qtt":
        s["A"] = ctx.qtt_from_cores([c.numpy() for c in _cores(case, seed)])
        s["x"] = _vector(case, seed)
        s["y"] = torch.empty_like(s["x"])
        return s
    if path == "batched":
        ctxs, states, rhs, gammas = [], [], [], []
        for i, n in enumerate(_batch_sides(case)):
            c, mu = binding.Context(), _batch_mu(i)
            sc = _scene("mono", n, seed, mu, tag=1 + i)
            con = _assemble(c, sc)
            gamma, lam = _iterate(con.Nc, mu, seed, tag=1 + i)
            gamma = _pad(gamma, 3, con.P)
            st = c.state(gamma, lam)
            b = torch.empty_like(gamma)
            c.newton_rhs(st, b)
            ctxs.append(c), states.append(st), rhs.append(b), gammas.append((gamma, lam, sc))
        s["ctxs"], s["states"], s["rhs"], s["keep"] = ctxs, states, rhs, gammas
        s["all"] = torch.empty(sum(b.numel() for b in rhs), dtype=torch.float64, device="cuda")
        s["dx"] = list(s["all"].split([b.numel() for b in rhs]))
        return s
    sc = _scene(case["scene"], case["n"], seed)
    if path == "step":
        prev = _prev_positions(sc)
        con = _assemble(ctx, prev)
        s["prev"] = [workload.view(con, k) for k in ("body_a", "body_b", "plane")]
        s["prev_gamma"] = _pad(_iterate(con.Nc, MU, seed)[0], 3, con.P)
        s["start"] = {k: v.clone() for k, v in sc["dev"].items() if k in ("pos", "vel", "omega")}
        s["scene"] = sc
        con = _assemble(ctx, sc)
        s["gamma"] = torch.zeros(con.P, dtype=torch.float64, device="cuda")
        s["lam"] = torch.zeros(2 * con.Nc, dtype=torch.float64, device="cuda")
        s["opts"] = ctx.pdip_opts(ctx.solve_opts(tol=TOL, maxit=200000, mixed=1, inner_tol=1e-3, max_outer=80))
        return s
    s["scene"] = sc
    if path == "assemble":
        return s
    slots = case.get("slots", 3)
    s["con"] = con = _assemble(ctx, sc, slots)
    if path == "net":
        s["params"], s["target"] = _net_inputs(con.Nc, seed)
        s["grad"] = torch.empty_like(s["params"])
        s["out"] = torch.empty(3 * con.Nc, dtype=torch.float32, device="cuda")
        return s
    if path == "pdip_qtt":
        s["gamma"] = torch.zeros(con.P, dtype=torch.float64, device="cuda")
        s["lam"] = torch.zeros(2 * con.Nc, dtype=torch.float64, device="cuda")
        so = ctx.solve_opts(binding.QP_QTT_PCG, None, tol=TOL, maxit=20000, mixed=1, inner_tol=1e-3, max_outer=80,
                            core_dtype=binding.QP_BF16)
        s["opts"] = ctx.pdip_opts(so, qtt_refresh=1, qtt_eps=case["eps"], qtt_rmax=case["rmax"])
        return s
    gamma, lam = _iterate(con.Nc, MU, seed)
    s["gamma"], s["lam"] = _pad(gamma, slots, con.P), lam
    s["state"] = ctx.state(s["gamma"], s["lam"])
    dt = torch.float32 if case.get("dtype") == "f32" else torch.float64
    if path == "apply":
        s["x"] = torch.randn(con.P, generator=_generator(seed, 7), dtype=torch.float64, device="cuda").to(dt)
        s["y"] = torch.empty_like(s["x"])
        s["dtype"] = CORE[case["dtype"]]
    else:
        s["rhs"] = torch.empty(con.P, dtype=torch.float64, device="cuda")
        s["dx"] = torch.empty_like(s["rhs"])
        s["opts"] = ctx.solve_opts(tol=TOL, maxit=200000, mixed=case["mixed"],
                                   inner_tol=1e-3 if case["mixed"] else 0.0, max_outer=80 if case["mixed"] else 0)
    return s


# ------------------------------------------------------------------ run
CONTACT_ARRAYS = ("body_a", "body_b", "plane", "key", "phi", "frame", "point", "arm_a", "arm_b", "r")


def run(s):
    path, ctx = s["path"], s["ctx"]
    if path == "assemble":
        con = _assemble(ctx, s["scene"])
        return {k: workload.view(con, k) for k in CONTACT_ARRAYS}
    if path == "apply":
        ctx.newton_apply(s["state"], s["x"], s["y"], s["dtype"])
        return s["y"]
    if path == "solve":
        ctx.newton_rhs(s["state"], s["rhs"])
        ctx.newton_solve(s["state"], s["rhs"], s["dx"], s["opts"])
        return dict(rhs=s["rhs"], dx=s["dx"])
    if path == "step":
        dev = s["scene"]["dev"]
        for k, v in s["start"].items():
            dev[k].copy_(v)
        _assemble(ctx, s["scene"])
        st = ctx.state(s["gamma"], s["lam"])
        ctx.pdip_init_warm(st, s["prev"][0], s["prev"][1], s["prev_gamma"], prev_plane=s["prev"][2])
        for _ in range(s["case"]["iters"]):
            ctx.pdip_step(st, s["opts"])
        ctx.advance(st)
        return dict(gamma=s["gamma"], lam=s["lam"], pos=dev["pos"], vel=dev["vel"], omega=dev["omega"])
    if path == "pdip_qtt":
        st = ctx.state(s["gamma"], s["lam"])
        ctx.pdip_init(st)
        ctx.pdip_step(st, s["opts"])
        return dict(gamma=s["gamma"], lam=s["lam"])
    if path == "qtt":
        core = s["case"]["core"]
        ctx.qtt_apply(s["A"], s["x"], s["y"], CORE[core], binding.QP_F64 if core == "f64" else binding.QP_F32)
        return s["y"]
    if path == "batched":
        binding.newton_solve_batched(s["ctxs"], s["states"], s["rhs"], s["dx"], tol=TOL, maxit=100000, inner_tol=1e-3,
                                     max_outer=60)
        return s["all"]
    if s["case"]["grad"]:
        loss = ctx.mpnn_grad(s["params"], FEAT_SCALE, s["target"], s["grad"])
        return dict(loss=loss, grad=s["grad"])
    ctx.mpnn_forward(s["params"], FEAT_SCALE, s["out"])
    return s["out"]


# ------------------------------------------------------------------ work
def _contacts_of(kind, n):
    """Contacts of a scene, to a few per cent."""
    return int(0.89 * n ** 3) if kind == "box" else 3 * n * n * (n - 1) + n * n


def _padded(Nc, slots=3):
    return 1 << max(1, math.ceil(math.log2(max(1, slots * Nc))))


APPLY_FLOPS = 160  # a contact's share of S x: two sides' forces and torques gathered, projected back, and the block


def work(case):
    path = case["path"]
    if path == "qtt":
        d, r = case["d"], case["rank"]
        ranks = [min(r, 4 ** min(k, d - k)) for k in range(d + 1)]
        pairs = sum(ranks[k] * ranks[k + 1] for k in range(d))
        size = 8 if case["core"] == "f64" else 4
        return dict(bytes=2.0 * (size << d) + 4 * pairs * {"f64": 8, "f32": 4, "bf16": 2}[case["core"]],
                    flops=4.0 * pairs * (1 << d))
    if path == "batched":
        Nc = [_contacts_of("mono", n) for n in _batch_sides(case)]
        return dict(bytes=sum(16.0 * _padded(c) + 4 * 8 * _padded(c) / 3 + 180.0 * c for c in Nc),
                    flops=95.0 * APPLY_FLOPS * sum(Nc))
    Nc, M = _contacts_of(case["scene"], case["n"]), case["n"] ** 3
    P = _padded(Nc, case.get("slots", 3))
    geometry = Nc * (18 * 8 + 16) + M * 20  # frame, arms, gap and bodies of each contact; each body's mass and list
    if path == "assemble":
        return dict(bytes=M * 12.0 * 8 + Nc * (17 * 8 + 20.0) + 8 * P, flops=120.0 * Nc + 60 * M)
    if path == "net":
        dense = 2.0 * Nc * (8 * 64 + 3 * 128 * 64 + 64 * 3)
        return dict(bytes=Nc * (8 + 3 + 3) * 8.0, flops=dense * (3 if case["grad"] else 1))
    if path == "apply":
        size = 4 if case["dtype"] == "f32" else 8
        return dict(bytes=2.0 * size * P + geometry * size / 8 + 5 * 8.0 * Nc, flops=float(APPLY_FLOPS) * Nc)
    if path == "solve":
        return dict(bytes=geometry + 2 * 8.0 * P + 5 * 8.0 * Nc, flops=95.0 * APPLY_FLOPS * Nc)
    if path == "step":
        return dict(bytes=geometry + M * 18 * 8.0 + 10 * 8.0 * Nc,
                    flops=case["iters"] * 95.0 * APPLY_FLOPS * Nc)
    d, r = math.log2(P), case["rmax"]
    # about 50 iterations, each with one QTT product whose ranks stay at about half their cap
    return dict(bytes=geometry + 10 * 8.0 * Nc, flops=50.0 * (APPLY_FLOPS * Nc + d * r * r * P))


# ------------------------------------------------------------------ exact, in float64 torch
def _constraints(gamma, mu):
    """Cone constraints, then -gamma_n (2 Nc values)."""
    gn, g1, g2 = gamma.unbind(1)
    return torch.cat([0.5 * (g1 * g1 + g2 * g2 - mu * mu * gn * gn), -gn])


def _cross(u, v):
    return torch.stack([u[:, 1] * v[:, 2] - u[:, 2] * v[:, 1], u[:, 2] * v[:, 0] - u[:, 0] * v[:, 2],
                        u[:, 0] * v[:, 1] - u[:, 1] * v[:, 0]], 1)


def _close_pairs(pos, rad, delta):
    """Pairs a < b with d^2 <= (r_a + r_b + delta)^2, by testing every pair in strips."""
    M, got = pos.shape[1], []
    strip = max(1, (1 << 25) // M)
    for lo in range(0, M, strip):
        hi = min(M, lo + strip)
        d2 = None
        for k in range(3):
            e = pos[k, lo:][None, :] - pos[k, lo:hi][:, None]
            d2 = e * e if d2 is None else d2 + e * e
        reach = (rad[lo:hi][:, None] + rad[lo:][None, :]) + delta
        a, b = torch.nonzero(d2 <= reach * reach, as_tuple=True)
        got.append(torch.stack([a + lo, b + lo])[:, b > a])
    return torch.cat(got, 1)


def _detect(sc):
    """The ordered contact set: ids, gap, frame, points, arms."""
    dev, delta = sc["dev"], sc["delta"]
    pos, rad = dev["pos"], dev["radius"]
    M = rad.shape[0]
    pa, pb = _close_pairs(pos, rad, delta)
    e = (pos[:, pb] - pos[:, pa]).T
    d = torch.sqrt((e[:, 0] * e[:, 0] + e[:, 1] * e[:, 1]) + e[:, 2] * e[:, 2])
    phi = d - (rad[pa] + rad[pb])
    n = e / d[:, None]
    p = pos[:, pa].T + n * (rad[pa] + phi * 0.5)[:, None]
    parts = [(pa, pb, phi, n, p)]
    for w, (axis, sign, off) in enumerate(((2, 1, 0.0),) + tuple(sc["walls"])):
        gap = ((pos[axis] - off) if sign > 0 else (off - pos[axis])) - rad
        b = torch.nonzero(gap <= delta)[:, 0]
        nw = torch.zeros(b.numel(), 3, dtype=torch.float64, device="cuda")
        nw[:, axis] = float(sign)
        pw = pos[:, b].T.clone()
        pw[:, axis] = off + sign * (gap[b] * 0.5)
        parts.append((torch.full_like(b, M + w), b, gap[b], nw, pw))
    a, b, phi, n, p = (torch.cat([q[i] for q in parts]) for i in range(5))
    key = torch.zeros_like(a)
    if a.numel():
        lo, hi = p.amin(0), p.amax(0)
        for ax in range(3):
            ext = hi[ax] - lo[ax]
            if float(ext) > 0.0:
                q = torch.floor(((p[:, ax] - lo[ax]) / ext) * float(1 << 21)).to(torch.int64).clamp(max=(1 << 21) - 1)
                for bit in range(21):
                    key |= ((q >> bit) & 1) << (3 * bit + ax)
    order = torch.sort(b, stable=True)[1]
    for v in (a, key):
        order = order[torch.sort(v[order], stable=True)[1]]
    a, b, phi, n, p = a[order], b[order], phi[order], n[order], p[order]
    plane = torch.where(a >= M, a - M, -1)
    a = a.clamp(max=M)
    axis = torch.argmin(n.abs(), 1)
    c = _cross(n, torch.nn.functional.one_hot(axis, 3).double())
    t1 = c / torch.sqrt((c * c).sum(1))[:, None]
    t2 = _cross(n, t1)
    ra = torch.where((a == M)[:, None], 0.0, p - pos[:, a.clamp(max=M - 1)].T)
    rb = p - pos[:, b].T
    return dict(a=a, b=b, plane=plane, phi=phi, U=torch.stack([n, t1, t2], 2), p=p, ra=ra, rb=rb, M=M)


class _System:
    """N = D^T M^-1 D and r of one or several scenes side by side (compact (Nc, 3) vectors)."""

    def __init__(self, scenes):
        off, self.parts = 0, []
        cat = {k: [] for k in ("a", "b", "U", "Ta", "Tb", "phi", "mu", "vk")}
        mass = []
        for sc in scenes:
            c = _detect(sc)
            dev, M = sc["dev"], c["M"]
            cat["a"].append(c["a"] + off), cat["b"].append(c["b"] + off), cat["U"].append(c["U"])
            for side, arm in (("Ta", c["ra"]), ("Tb", c["rb"])):
                cat[side].append(torch.stack([_cross(arm, c["U"][:, :, u]) for u in range(3)], 2))
            cat["phi"].append(c["phi"])
            cat["mu"].append(torch.full_like(c["phi"], sc["mu"]))
            g = torch.tensor(GRAVITY, dtype=torch.float64, device="cuda")[:, None]
            still = torch.zeros(1, 6, dtype=torch.float64, device="cuda")
            cat["vk"].append(torch.cat([torch.cat([dev["vel"] + DT * g, dev["omega"]]).T, still]))
            m = torch.stack([dev["inv_mass"]] * 3 + [dev["inv_inertia"]] * 3, 1)
            mass.append(torch.cat([m, still]))  # the floor and the walls do not move
            self.parts.append(c)
            off += M + 1
        for k, v in cat.items():
            setattr(self, k, torch.cat(v))
        self.mass = torch.cat(mass)
        self.r = self.project(self.vk)
        self.r[:, 0] += self.phi / DT

    def force(self, x):
        """D x, one row of force and torque a body."""
        out = torch.zeros_like(self.mass)
        f = torch.einsum("ciu,cu->ci", self.U, x)
        out.index_add_(0, self.b, torch.cat([f, torch.einsum("ciu,cu->ci", self.Tb, x)], 1))
        out.index_add_(0, self.a, -torch.cat([f, torch.einsum("ciu,cu->ci", self.Ta, x)], 1))
        return out

    def project(self, w):
        wa, wb = w[self.a], w[self.b]
        return (torch.einsum("ciu,ci->cu", self.U, wb[:, :3] - wa[:, :3]) + torch.einsum("ciu,ci->cu", self.Tb, wb[:, 3:])
                - torch.einsum("ciu,ci->cu", self.Ta, wa[:, 3:]))

    def N(self, x):
        return self.project(self.mass * self.force(x))

    def slope(self, gamma):
        g = gamma.clone()
        g[:, 0] *= -self.mu * self.mu
        return g

    def blocks(self, gamma, lam):
        f, (lc, ln) = _constraints(gamma, self.mu), lam.chunk(2)
        g = self.slope(gamma)
        H = (lc / -f[:lc.numel()])[:, None, None] * g[:, :, None] * g[:, None, :]
        H[:, 0, 0] += ln / gamma[:, 0] - self.mu * self.mu * lc
        H[:, 1, 1] += lc
        H[:, 2, 2] += lc
        return H

    def rhs(self, gamma, lam, t):
        f = _constraints(gamma, self.mu)
        add = self.slope(gamma) / f[:gamma.shape[0], None]
        add[:, 0] += 1.0 / gamma[:, 0]
        return -(self.N(gamma) + self.r) + add / t

    def solve(self, H, b):
        """Block-Jacobi CG until the residual stops falling."""
        own = torch.einsum("ciu,cm,civ->cuv", self.U, self.mass[self.b][:, :1] + self.mass[self.a][:, :1], self.U)
        for T, body in ((self.Tb, self.b), (self.Ta, self.a)):
            own += torch.einsum("ciu,cm,civ->cuv", T, self.mass[body][:, 3:4], T)
        inv = torch.linalg.inv(own + H)
        A = lambda v: self.N(v) + torch.einsum("cuv,cv->cu", H, v)  # noqa: E731
        x = torch.zeros_like(b)
        norm = float(b.norm())
        for _ in range(3):  # restarted from the true residual, for the last digits
            r = b - A(x)
            z = torch.einsum("cuv,cv->cu", inv, r)
            p, rz = z.clone(), (r * z).sum()
            for k in range(1500):
                q = A(p)
                alpha = rz / (p * q).sum()
                x += alpha * p
                r -= alpha * q
                if k % 5 == 0 and float(r.norm()) <= 1e-15 * norm:
                    break
                z = torch.einsum("cuv,cv->cu", inv, r)
                new = (r * z).sum()
                p, rz = z + (new / rz) * p, new
        return x

    def pdip_step(self, gamma, lam):
        """One primal-dual iteration with the library's default factors."""
        Nc = gamma.shape[0]
        f = _constraints(gamma, self.mu)
        t = _barrier(gamma, lam, self.mu)

        def residual(g, m):
            dual = self.N(g) + self.r + self.slope(g) * m[:Nc, None]
            dual[:, 0] -= m[Nc:]
            cent = -m * _constraints(g, self.mu) - 1.0 / t
            return math.sqrt(float((dual * dual).sum() + (cent * cent).sum()))

        before = residual(gamma, lam)
        dg = self.solve(self.blocks(gamma, lam), self.rhs(gamma, lam, t))
        slope = torch.cat([(self.slope(gamma) * dg).sum(1), -dg[:, 0]])
        dl = -lam - 1.0 / (t * f) - (lam / f) * slope
        s = 0.99 * min(1.0, float(torch.where(dl < 0, -lam / dl, math.inf).amin()))
        for _ in range(60):
            if bool((_constraints(gamma + s * dg, self.mu) < 0).all()):
                break
            s *= 0.5
        for _ in range(60):
            if residual(gamma + s * dg, lam + s * dl) <= (1.0 - 0.01 * s) * before:
                break
            s *= 0.5
        return gamma + s * dg, lam + s * dl


def _exact_qtt(case, seed):
    d = case["d"]
    x = _vector(case, seed).double().reshape(1, -1)  # (rank, remaining columns and done rows)
    kind = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}[case["core"]]
    for k, c in enumerate(_cores(case, seed)):
        r0, _, r1 = c.shape
        G = c.to(torch.float32).to(kind).double().cuda() if case["core"] != "f64" else c.cuda()
        G = G.reshape(r0, 2, 2, r1).permute(1, 3, 0, 2).reshape(2 * r1, 2 * r0)  # (i, b) from (a, j)
        done, left = 1 << k, 1 << (d - k - 1)
        x = x.reshape(r0, done, 2, left).permute(0, 2, 1, 3).reshape(2 * r0, done * left)
        x = (G @ x).reshape(2, r1, done, left).permute(1, 2, 0, 3).reshape(r1, -1)
    return x.reshape(-1)


def _exact_net(case, seed):
    sc = _scene(case["scene"], case["n"], seed)
    sy = _System([sc])
    c = sy.parts[0]
    Nc = c["a"].numel()
    params, target = _net_inputs(Nc, seed)
    theta, at = [], 0
    for s in NET_SHAPES:
        m = math.prod(s)
        theta.append(params[at:at + m].to(torch.bfloat16).double().reshape(s).requires_grad_())
        at += m
    u = sy.r.clone()
    u[:, 0] -= c["phi"] / DT
    x = torch.cat([c["U"][:, :, 0], (c["phi"] / DT)[:, None], u, torch.full_like(c["phi"], MU)[:, None]], 1)
    x = x * torch.tensor(FEAT_SCALE, dtype=torch.float32).double().cuda()
    on = torch.ones(c["M"] + 1, 1, dtype=torch.float64, device="cuda")
    on[c["M"]] = 0.0
    h = torch.relu(x @ theta[0].T + theta[1])
    for k in (2, 4, 6):
        m = torch.zeros(c["M"] + 1, 64, dtype=torch.float64, device="cuda")
        m = m.index_add(0, c["a"], h).index_add(0, c["b"], h) * on
        h = torch.relu(torch.cat([h, m[c["a"]] + m[c["b"]]], 1) @ theta[k].T + theta[k + 1])
    out = h @ theta[8].T + theta[9]
    if not case["grad"]:
        return out.detach().reshape(-1)
    loss = ((out - target.double().reshape(-1, 3)) ** 2).mean()
    loss.backward()
    return dict(loss=float(loss.detach()), grad=torch.cat([t.grad.reshape(-1) for t in theta]))


def exact(case, seed):
    path = case["path"]
    if path == "qtt":
        return _exact_qtt(case, seed)
    if path == "net":
        return _exact_net(case, seed)
    if path == "batched":
        scenes = [_scene("mono", n, seed, _batch_mu(i), tag=1 + i) for i, n in enumerate(_batch_sides(case))]
        sy = _System(scenes)
        Nc = [c["a"].numel() for c in sy.parts]
        at = [_iterate(m, sc["mu"], seed, tag=1 + i) for i, (m, sc) in enumerate(zip(Nc, scenes))]
        t = torch.cat([torch.full((m, 1), _barrier(g, v, sc["mu"]), dtype=torch.float64, device="cuda")
                       for m, (g, v), sc in zip(Nc, at, scenes)])
        gamma = torch.cat([g for g, _ in at])
        lam = torch.cat([m[:len(m) // 2] for _, m in at] + [m[len(m) // 2:] for _, m in at])
        dx = sy.solve(sy.blocks(gamma, lam), sy.rhs(gamma, lam, t))
        return torch.cat([_pad(v, 3, _padded(v.shape[0])) for v in dx.split(Nc)])
    sc = _scene(case["scene"], case["n"], seed)
    sy = _System([sc])
    c = sy.parts[0]
    Nc = c["a"].numel()
    slots = case.get("slots", 3)
    P = _padded(Nc, slots)
    if path == "assemble":
        return dict(body_a=None, body_b=None, plane=None, key=None, phi=c["phi"],
                    frame=c["U"].permute(2, 1, 0).reshape(-1), point=c["p"].T.reshape(-1),
                    arm_a=c["ra"].T.reshape(-1), arm_b=c["rb"].T.reshape(-1), r=_pad(sy.r, 3, P))
    if path == "step":
        before = _detect(_prev_positions(sc))
        old = _iterate(before["a"].numel(), MU, seed)[0]
        name = lambda q: ((q["a"] + q["plane"].clamp(min=0)) << 32) + q["b"]  # noqa: E731
        k, order = torch.sort(name(before))
        want = name(c)
        at = torch.searchsorted(k, want).clamp(max=k.numel() - 1)
        gamma = torch.where((k[at] == want)[:, None], old[order[at]], torch.tensor([1.0, 0.0, 0.0], device="cuda").double())
        gamma[:, 0].clamp_(min=1.0)
        tang = gamma[:, 1:].norm(dim=1)
        cap = 0.9 * MU * gamma[:, 0]
        gamma[:, 1:] *= torch.where(tang > cap, cap / tang.clamp(min=1e-300), 1.0)[:, None]
        lam = -1.0 / _constraints(gamma, MU)
        for _ in range(case["iters"]):
            gamma, lam = sy.pdip_step(gamma, lam)
        after = (sy.vk + sy.mass * sy.force(gamma))[:c["M"]].T
        return dict(gamma=_pad(gamma, 3, P), lam=lam, pos=sc["dev"]["pos"] + DT * after[:3], vel=after[:3],
                    omega=after[3:])
    if path == "pdip_qtt":
        gamma = torch.zeros(Nc, 3, dtype=torch.float64, device="cuda")
        gamma[:, 0] = 1.0
        gamma, lam = sy.pdip_step(gamma, -1.0 / _constraints(gamma, MU))
        return dict(gamma=_pad(gamma, 3, P), lam=lam)
    gamma, lam = _iterate(Nc, MU, seed)
    H = sy.blocks(gamma, lam)
    if path == "apply":
        x = torch.randn(P, generator=_generator(seed, 7), dtype=torch.float64, device="cuda")
        x = x.to(torch.float32).double() if case["dtype"] == "f32" else x
        y = x.clone()
        rows = x[:slots * Nc].view(Nc, slots)[:, :3]
        y[:slots * Nc].view(Nc, slots)[:, :3] = sy.N(rows) + torch.einsum("cuv,cv->cu", H, rows)
        return y
    rhs = sy.rhs(gamma, lam, _barrier(gamma, lam, MU))
    return dict(rhs=_pad(rhs, 3, P), dx=_pad(sy.solve(H, rhs), 3, P))
