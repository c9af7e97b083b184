"""Performance cases of the framework: the calls a user's program makes, over the range of sizes, orders,
precisions and options they are made with.

listed() names the cases, draw() gives further ones of the same ranges, prepare() makes what a program has in
hand before the call (moonlets on the GPU, or in pinned host memory, and the context or batch it keeps), run()
makes one pass through the public entry points and returns its outputs, work() says what one pass cannot do
without, and exact() gives the outputs of a pass in plain 64-bit arithmetic where direct summation is quick.

Kinds of cases:
  sort     ncorp_hilbert_sort_static: keys and stable order, allocation-free (the smallest call)
  step     ncorp_step on device arrays, called again and again on one disk (a time integration)
  host     ncorp_step on pinned host arrays with a fresh upload, and the colliding pairs read back (a program
           that owns the state and changes it between the steps)
  accel    ncorp_accel: accelerations of given positions (another integrator's force evaluation)
  collide  ncorp_collide and ncorp_collisions: the collision search alone
  batch    ncorp_batch_run: an ensemble of disks advanced together, every state read back
"""
import math

import torch

from paper_2310_20374_gb300 import ncorp

MIXED, FP64 = "mixed", "fp64"
PAIRS_CAP = 1 << 16


def listed():
    return [
        # the smallest call: the keys of a few thousand moonlets
        {"name": "sort_4k", "kind": "sort", "n": 4099},
        # a thousand moonlets, the start of a small integration: launches and grid barriers are all there is
        {"name": "step_1k_p3", "kind": "step", "n": 1009, "p": 3, "theta": 0.5, "precision": MIXED, "options": "none"},
        # 1e4 moonlets in FP64, where a run is checked against a reference
        {"name": "step_10k_p3_fp64", "kind": "step", "n": 10000, "p": 3, "theta": 0.5, "precision": FP64,
         "options": "none"},
        # a disk with every external force, the star among them (its position moves with the time)
        {"name": "step_50k_p4_star", "kind": "step", "n": 50021, "p": 4, "theta": 0.5, "precision": MIXED,
         "options": "star"},
        # a dense ring whose impacts are resolved in the step
        {"name": "step_30k_p3_impacts", "kind": "step", "n": 30011, "p": 3, "theta": 0.5, "precision": MIXED,
         "options": "impacts"},
        # the benchmark's disk: 1e5 moonlets at the highest order, mixed precision ...
        {"name": "step_100k_p6", "kind": "step", "n": 100000, "p": 6, "theta": 0.5, "precision": MIXED,
         "options": "none"},
        # ... in FP64 ...
        {"name": "step_100k_p6_fp64", "kind": "step", "n": 100000, "p": 6, "theta": 0.5, "precision": FP64,
         "options": "none"},
        # ... and from host memory, uploaded for every step
        {"name": "host_100k_p6", "kind": "host", "n": 100000, "p": 6, "theta": 0.5, "precision": MIXED},
        # the largest disk of the benchmark
        {"name": "step_1m_p4", "kind": "step", "n": 1000000, "p": 4, "theta": 0.6, "precision": MIXED,
         "options": "none"},
        # the force evaluation alone, at an odd size
        {"name": "accel_120k_p5", "kind": "accel", "n": 120011, "p": 5, "theta": 0.5, "precision": MIXED},
        # the collision search alone, at an odd size, where many pairs collide
        {"name": "collide_200k", "kind": "collide", "n": 200003},
        # an ensemble: 64 disks between 1e3 and 2e5 moonlets in one batch, a run of five steps
        {"name": "batch_64", "kind": "batch", "disks": 64, "lo": 1000, "hi": 200000, "p": 6, "theta": 0.5, "steps": 5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "host", "accel", "accel", "collide", "batch", "sort"])
    theta = round(rng.uniform(0.45, 0.65), 3)
    precision = rng.choice([MIXED, MIXED, MIXED, FP64])
    p = rng.choice([2, 3, 4, 5, 6])
    if kind == "sort":
        return {"kind": kind, "n": _log_int(rng, 4000, ncorp.NCORP_STATIC_MAX_N)}
    if kind == "step":
        options = rng.choice(["none", "none", "star", "impacts"])
        hi = 100000 if precision == FP64 or options == "impacts" else 1000000
        return {"kind": kind, "n": _log_int(rng, 1000, hi), "p": p, "theta": theta, "precision": precision,
                "options": options}
    if kind == "host":
        return {"kind": kind, "n": _log_int(rng, 5000, 300000), "p": p, "theta": theta, "precision": MIXED}
    if kind == "accel":
        # from 2e4 moonlets: the call's use is another integrator's whole disk
        return {"kind": kind, "n": _log_int(rng, 20000, 100000 if precision == FP64 else 200000), "p": p,
                "theta": theta, "precision": precision}
    if kind == "collide":
        return {"kind": kind, "n": _log_int(rng, 5000, 300000)}
    return {"kind": kind, "disks": rng.randint(8, 64), "lo": 1000, "hi": _log_int(rng, 20000, 200000), "p": p,
            "theta": theta, "steps": rng.randint(2, 5)}


# ---------------------------------------------------------------------------- inputs
DT = 1e-3
DENSE_DT = 5e-3
STAR = {"star_mass": 2.0, "star_a": 80.0, "star_obliquity": 0.4, "t0": 0.3, "central_J2": 2e-3}


def _disk(n, gen, dense=False):
    """Moonlets of a disk around a central mass (G = M_c = R_c = 1): semi-major axes uniform, small Rayleigh
    eccentricities and inclinations, radii from dN/dR ~ R^-3.5, masses ~ R^3 summing to 0.02.  dense: a narrow
    ring of large moonlets (a fixed share of its volume), where many pairs collide in a step."""
    a_lo, a_hi, s_e, s_i, r_lo, r_hi = 2.0, 10.0, 0.05, 0.025, 1e-3, 1e-2
    if dense:
        scale = (30000.0 / n) ** (1.0 / 3.0)
        a_lo, a_hi, s_e, s_i, r_lo, r_hi = 2.0, 2.6, 0.1, 0.05, 1e-2 * scale, 3e-2 * scale
    u = torch.rand((7, n), generator=gen, device="cuda", dtype=torch.float64)
    a = a_lo + (a_hi - a_lo) * u[0]
    e = (s_e * torch.sqrt(-2.0 * torch.log1p(-u[1]))).clamp(max=0.9)
    inc = s_i * torch.sqrt(-2.0 * torch.log1p(-u[2]))
    M, om, Om = (2.0 * math.pi * u[k] for k in (3, 4, 5))
    lo, hi = r_lo ** -2.5, r_hi ** -2.5
    R = (lo + u[6] * (hi - lo)) ** (-1.0 / 2.5)
    m = R ** 3
    m = m * (0.02 / m.sum())
    E = M + e * torch.sin(M)
    for _ in range(12):   # Kepler's equation by Newton's method
        E = E - (E - e * torch.sin(E) - M) / (1.0 - e * torch.cos(E))
    cE, sE, sq = torch.cos(E), torch.sin(E), torch.sqrt(1.0 - e * e)
    xp, yp = a * (cE - e), a * sq * sE
    rate = a ** -1.5 / (1.0 - e * cE)
    vxp, vyp = -a * sE * rate, a * sq * cE * rate
    cO, sO, co, so, ci, si = (f(v) for v in (Om, om, inc) for f in (torch.cos, torch.sin))
    r11, r12 = cO * co - sO * so * ci, -cO * so - sO * co * ci
    r21, r22 = sO * co + cO * so * ci, -sO * so + cO * co * ci
    r31, r32 = so * si, co * si
    pos = torch.stack([r11 * xp + r12 * yp, r21 * xp + r22 * yp, r31 * xp + r32 * yp], dim=1).contiguous()
    vel = torch.stack([r11 * vxp + r12 * vyp, r21 * vxp + r22 * vyp, r31 * vxp + r32 * vyp], dim=1).contiguous()
    return pos, vel, m.contiguous(), R.contiguous()


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 1000003 + 17)


def _dense(case):
    return case["kind"] == "collide" or case.get("options") == "impacts"


def _batch_sizes(case):
    """Moonlets of each disk: spread evenly over the logarithm of the range, in a shuffled order."""
    k, lo, hi = case["disks"], math.log(case["lo"]), math.log(case["hi"])
    sizes = [int(math.exp(lo + (i + 0.5) / k * (hi - lo))) for i in range(k)]
    return [sizes[i] for i in torch.randperm(k, generator=torch.Generator().manual_seed(k)).tolist()]


def _config(case):
    cfg = ncorp.ncorp_config_default()
    cfg.precision = ncorp.NCORP_FP64 if case.get("precision") == FP64 else ncorp.NCORP_MIXED
    if case.get("options") == "star":
        for k, v in STAR.items():
            setattr(cfg, k, v)
    if case.get("options") == "impacts":
        cfg.resolve_f = 2.0
    return cfg


class _State:
    """What a program keeps between calls; its context or batch is released with it."""

    def __init__(self, case):
        self.case, self.ctx, self.batch = case, None, None

    def __del__(self):
        if self.ctx is not None:
            ncorp.ncorp_free(self.ctx)
        if self.batch is not None:
            ncorp.ncorp_batch_free(self.batch)


def prepare(case, seed):
    s = _State(case)
    gen = _generator(seed)
    stream = torch.cuda.current_stream().cuda_stream
    kind = case["kind"]
    if kind == "batch":
        cfg = _config(case)
        # the default leaf size, set so that the batch does not time candidates: the choice would
        # change the results from one run to the next
        cfg.leaf_size = 64 if case["p"] >= 4 else 32
        s.batch = ncorp.ncorp_batch_create(cfg, 0, stream)
        s.sizes = _batch_sizes(case)
        s.ids = []
        for n in s.sizes:
            pos, vel, m, R = _disk(n, gen)
            s.ids.append(ncorp.ncorp_batch_add_disk(s.batch, pos, vel, m, R, n, case["p"], case["theta"], DT))
        total = sum(s.sizes)
        s.pos = torch.empty((total, 3), device="cuda", dtype=torch.float64)
        s.vel = torch.empty_like(s.pos)
        return s
    n = case["n"]
    s.pos, s.vel, s.mass, s.radius = _disk(n, gen, _dense(case))
    if kind == "sort":
        s.keys = torch.empty(n, device="cuda", dtype=torch.int64)
        s.order = torch.empty(n, device="cuda", dtype=torch.int64)
        return s
    s.ctx = ncorp.ncorp_init(_config(case), n, torch.cuda.current_device(), stream)
    if kind == "host":
        s.pos, s.vel, s.mass, s.radius = (t.cpu().pin_memory() for t in (s.pos, s.vel, s.mass, s.radius))
        s.pairs = torch.zeros((PAIRS_CAP, 2), dtype=torch.int64).pin_memory()
    elif kind == "accel":
        s.acc, s.mutual = torch.empty_like(s.pos), torch.empty_like(s.pos)
    elif kind == "collide":
        s.pairs = torch.zeros((PAIRS_CAP, 2), device="cuda", dtype=torch.int64)
    return s


# ---------------------------------------------------------------------------- one pass
def run(s):
    c = s.case
    kind = c["kind"]
    if kind == "sort":
        stream = torch.cuda.current_stream().cuda_stream
        ncorp.ncorp_hilbert_sort_static(s.pos, c["n"], s.keys, s.order, stream)
        return [s.keys, s.order]
    if kind == "step":
        dt = DENSE_DT if _dense(c) else DT
        ncorp.ncorp_step(s.ctx, s.pos, s.vel, s.mass, s.radius, c["n"], c["p"], c["theta"], dt)
        return [s.pos, s.vel]
    if kind == "host":
        ncorp.ncorp_reset(s.ctx)
        ncorp.ncorp_step(s.ctx, s.pos, s.vel, s.mass, s.radius, c["n"], c["p"], c["theta"], DT)
        k = ncorp.ncorp_collisions(s.ctx, s.pairs, PAIRS_CAP)
        return [s.pos, s.vel, s.pairs, k]
    if kind == "accel":
        ncorp.ncorp_accel(s.ctx, s.pos, s.mass, c["n"], c["p"], c["theta"], s.acc, s.mutual)
        return [s.acc, s.mutual]
    if kind == "collide":
        ncorp.ncorp_collide(s.ctx, s.pos, s.vel, s.radius, c["n"], DENSE_DT)
        k = ncorp.ncorp_collisions(s.ctx, s.pairs, PAIRS_CAP)
        return [s.pairs, k]
    ncorp.ncorp_batch_run(s.batch, c["steps"])
    at = 0
    for did, n in zip(s.ids, s.sizes):
        ncorp.ncorp_batch_get_state(s.batch, did, s.pos[at:at + n], s.vel[at:at + n])
        at += n
    return [s.pos, s.vel]


# ---------------------------------------------------------------------------- work of one pass
# Pairs per moonlet that the method sums directly (each evaluated once) and well-separated cell pairs per
# moonlet, at theta_min = 0.5 and the default leaf sizes and thresholds, from the walk's counters.
NEAR_PAIRS = {2: 228.0, 3: 228.0, 4: 534.0, 5: 534.0, 6: 566.0}
CELL_PAIRS = {2: 5.1, 3: 5.1, 4: 1.8, 5: 1.8, 6: 1.35}
COLLISION_PAIRS = {2: 91.0, 3: 91.0, 4: 222.0, 5: 222.0, 6: 222.0}   # moonlet pairs the search tests, per moonlet


def _cell_pair_flops(p):
    """Multiply-adds of one well-separated pair, both directions from one derivative tensor: the recursion for
    the (p + 1)(p + 2)(p + 3)/6 derivatives and the contraction with the moments of both cells."""
    num = (p + 1) * (p + 2) * (p + 3) // 6
    contraction = sum((na + 1) * (na + 2) // 2 * (nb + 1) * (nb + 2) // 2
                      for nb in range(p) if nb != 1 for na in range(1, p - nb + 1))
    return 12 * num + 4 * contraction


def _force_flops(n, p):
    near = min(NEAR_PAIRS[p], 0.5 * (n - 1))
    return n * (30.0 * near + CELL_PAIRS[p] * _cell_pair_flops(p) + 6 * (p + 1) * (p + 2) * (p + 3) // 6)


def work(case):
    kind = case["kind"]
    if kind == "sort":
        n = case["n"]
        return {"bytes": n * (24 + 8 + 8), "flops": 0}
    if kind == "accel":
        n = case["n"]
        return {"bytes": n * (24 + 8 + 24 + 24), "flops": _force_flops(n, case["p"])}
    if kind == "collide":
        n = case["n"]
        return {"bytes": n * (24 + 24 + 8), "flops": n * 30.0 * COLLISION_PAIRS[6]}
    if kind == "batch":
        p, n = case["p"], sum(_batch_sizes(case))
        per_step = sum(_force_flops(k, p) + 30.0 * k * COLLISION_PAIRS[p] for k in _batch_sizes(case))
        return {"bytes": n * 112, "flops": case["steps"] * per_step}
    n = case["n"]
    search = n * 30.0 * COLLISION_PAIRS[case["p"]]
    evals = 2 if kind == "host" else 1   # the uploaded state's acceleration, and the new one's
    return {"bytes": n * 112, "flops": evals * _force_flops(n, case["p"]) + search}


# ---------------------------------------------------------------------------- 64-bit results
EXACT_MAX_N = 130000


def _direct(pos, m):
    """Mutual accelerations by direct summation (G = 1); coincident pairs contribute nothing."""
    n = pos.shape[0]
    x, y, z = (pos[:, k].contiguous() for k in range(3))
    out = torch.empty_like(pos)
    rows = max(1, (1 << 27) // n)
    for i in range(0, n, rows):
        dx, dy, dz = (c[None, :] - c[i:i + rows, None] for c in (x, y, z))
        r2 = dx * dx
        r2.addcmul_(dy, dy).addcmul_(dz, dz)
        w = torch.where(r2 > 0, m[None, :] * r2.pow_(-1.5), 0.0)
        out[i:i + rows, 0] = (w * dx).sum(1)
        out[i:i + rows, 1] = (w * dy).sum(1)
        out[i:i + rows, 2] = (w * dz).sum(1)
    return out


def _external(pos, star, t):
    r2 = (pos * pos).sum(1, keepdim=True)
    a = -pos * r2 ** -1.5
    if star:
        z = pos[:, 2:3]
        q = STAR["central_J2"] * r2 ** -2.5
        a = a + q * (15.0 * z * z - 3.0 * r2) / (2.0 * r2) * pos
        a[:, 2:3] -= 3.0 * q * z
        lam = math.sqrt(STAR["star_mass"] / STAR["star_a"] ** 3) * t
        eps = STAR["star_obliquity"]
        s = torch.tensor([math.cos(lam), math.sin(lam) * math.cos(eps), math.sin(lam) * math.sin(eps)],
                         device=pos.device, dtype=pos.dtype)
        k = STAR["star_mass"] / STAR["star_a"] ** 3
        a = a - k * (pos - 3.0 * (pos @ s)[:, None] * s[None, :])
    return a


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("step", "host", "accel") or case["n"] > EXACT_MAX_N or case.get("options") == "impacts":
        return None   # whole numbers, resolved impacts, or more pairs than direct summation takes quickly
    pos, vel, m, _ = _disk(case["n"], _generator(seed), _dense(case))
    if kind == "accel":
        mutual = _direct(pos, m)
        return [mutual + _external(pos, False, 0.0), mutual]
    star = case["options"] == "star" if kind == "step" else False
    t0 = STAR["t0"] if star else 0.0
    vel = vel + 0.5 * DT * (_direct(pos, m) + _external(pos, star, t0))
    pos = pos + DT * vel
    vel = vel + 0.5 * DT * (_direct(pos, m) + _external(pos, star, t0 + DT))
    return [pos, vel, None] if kind == "host" else [pos, vel]
