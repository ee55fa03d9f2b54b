"""The workloads of this framework that are timed, and how their results are judged.

Each case is one pass through the public entry points as a user's program makes it.  Kinds:

  matvec    u = D f on a resident tree (the inner call of every iterative method)
  step      new positions, then u = D f: rpy_tree_update_positions + rpy_matvec (one time step)
  forest    u = D f of many independent systems in one resident forest
  oneshot   rpy_matvec_oneshot: build, apply, free (a program that keeps nothing)
  evaluate  velocities at separate target points: rpy_evaluate
  noise     D^{1/2} z by a fixed number of Lanczos steps on a resident tree (the Brownian displacement)
  host      rpy_tree_matvec_host: a time step with page-locked host buffers in and out
  serve     a server with resident systems of several sizes and accuracies: one request of
            new positions and forces to each, all in flight together, waited for

Fields of a case: kind, dist (cube, sphere = surface of a sphere, mixed = 90% sphere + 10% cube,
plummer), n, a (bead radius; 0 means 0.5 / n^(1/3)), digits (3, 6, 9), prec (0 FP64, 1 FP32 form) and
the build parameters leaf_cap, p, quad (0 = the defaults of the setting).
"""
import math

import numpy as np
import torch

import paper_1711_02976_gb300 as rp

# Plane waves (both halves), quadrature nodes and default order of each quadrature rule: the sizes of
# the expansions, for work() only.
WAVES = {3: 268, 4: 436, 5: 646, 6: 928, 9: 2336}
NODES = {3: 10, 4: 13, 5: 16, 6: 19, 9: 33}
ORDER = {3: 8, 6: 18, 9: 26}
LEAF = {3: 40, 6: 100, 9: 120}

# The largest n for which the direct sum of exact() is taken (pairs).
EXACT_PAIRS = 4.5e10


def _case(name, kind, dist, n, digits, prec, a=0.0, leaf_cap=0, p=0, quad=0, **more):
    c = dict(name=name, kind=kind, dist=dist, n=n, a=a, digits=digits, prec=prec, leaf_cap=leaf_cap, p=p, quad=quad)
    c.update(more)
    return c


def listed():
    return [
        # the repository's smallest configuration, applied again and again: launches and latency
        _case("cube4096_d3_f64_matvec", "matvec", "cube", 4096, 3, 0, a=0.004, leaf_cap=40),
        # a script's single call on a small system of odd size: build, apply, free
        _case("cube1001_d6_f64_oneshot", "oneshot", "cube", 1001, 6, 0, a=0.01),
        # an ordinary Brownian-dynamics system, one time step at the default parameters
        _case("sphere20001_d6_f64_step", "step", "sphere", 20001, 6, 0),
        # the benchmark's system, one time step: plain FP64 and the FP32 form, at the autotuner's choices
        _case("mixed1m_d6_f64_step", "step", "mixed", 1000000, 6, 0, a=1e-4, leaf_cap=100, p=16, quad=5),
        _case("mixed1m_d6_f32_step", "step", "mixed", 1000000, 6, 1, a=1e-4, leaf_cap=140, p=15, quad=5),
        # the paper's largest system, one time step: the largest calls in both precisions
        _case("cube15m_d3_f64_step", "step", "cube", 15000000, 3, 0, a=2e-5, leaf_cap=80, p=6, quad=3),
        _case("cube15m_d3_f32_step", "step", "cube", 15000000, 3, 1, a=2e-5, leaf_cap=80, p=6, quad=3),
        # the batching form: 256 systems of uneven size, cubes and Plummer-like clusters
        _case("forest256_d3_f32_matvec", "forest", "batch", 0, 3, 1, leaf_cap=80, p=8, quad=3, nsys=256, lo=1000,
              hi=200000),
        # the highest accuracy setting, resident tree
        _case("mixed200k_d9_f64_matvec", "matvec", "mixed", 200000, 9, 0, a=1e-4, leaf_cap=120, p=25, quad=9),
        # flow at tracer points around a suspension
        _case("evaluate150k_d6_f64", "evaluate", "cube", 150000, 6, 0, a=1e-3, nt=49999),
        # Brownian displacements of a suspension with overlapping beads
        _case("noise50k_d3_f32", "noise", "cube", 50000, 3, 1, steps=12),
        # continuous batching over resident systems, 3-digit FP32 and 6-digit FP64 alternating
        _case("serve8_mixed_precision", "serve", "batch", 0, 6, 0, nsys=8, lo=10000, hi=120000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["matvec", "matvec", "step", "step", "step", "forest", "oneshot", "evaluate", "noise", "host",
                       "serve"])
    digits, prec = rng.choice([(3, 0), (3, 1), (3, 1), (6, 0), (6, 0), (6, 1), (6, 1), (9, 0)])
    dist = rng.choice(["cube", "sphere", "mixed", "plummer"])
    # largest sizes: what each setting is used for, and no pass longer than the largest listed one
    top = {(3, 0): 2000000, (3, 1): 8000000, (6, 0): 1500000, (6, 1): 3000000, (9, 0): 400000}[(digits, prec)]
    if dist == "plummer":
        top = min(top, 300000)
    if kind == "oneshot":
        top, prec = min(top, 300000), 0
    if kind in ("evaluate", "noise", "host"):
        top = min(top, 200000 if kind == "noise" else 500000)
    if kind == "noise":
        digits = min(digits, 6)
    n = _log_int(rng, 1000, top) | 1
    a = rng.choice([0.0, 0.0, 0.1, 0.02])   # in units of n^(-1/3): overlapping, ordinary and dilute beads
    c = _case("", kind, dist, n, digits, prec, a=a * n ** (-1.0 / 3.0))
    c.pop("name")
    # parameters as the autotuner sets them for about half the cases, and always for the large ones
    if kind not in ("oneshot", "serve") and (n > 500000 or rng.random() < 0.5):
        c["leaf_cap"] = rng.choice([60, 80, 111]) if digits == 3 else rng.choice([90, 120, 141])
        c["p"], c["quad"] = {3: (6, 3), 6: (16, 5), 9: (25, 9)}[digits]
        if dist != "cube" and digits == 3:
            c["p"] = 8
    if kind in ("forest", "serve"):
        c["dist"], c["n"], c["a"] = "batch", 0, 0.0
        c["nsys"] = _log_int(rng, 2, 64 if kind == "forest" else 12)
        c["lo"], c["hi"] = 1000, _log_int(rng, 5000, 100000)
        c["leaf_cap"], c["p"], c["quad"] = 0, 0, 0
        if digits == 9:
            c["digits"] = 6
    if kind == "evaluate":
        c["nt"] = _log_int(rng, max(1000, n // 8), 200000)
    if kind == "noise":
        c["steps"] = rng.randint(6, 16)
    return c


# ---------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _rand(g, *shape):
    return torch.rand(*shape, dtype=torch.float64, device="cuda", generator=g)


def _randn(g, *shape):
    return torch.randn(*shape, dtype=torch.float64, device="cuda", generator=g)


def _surface(g, n):
    d = _randn(g, n, 3)
    return 0.5 + 0.5 * d / d.norm(dim=1, keepdim=True)


def _positions(g, dist, n):
    if dist == "cube":
        return _rand(g, n, 3)
    if dist == "sphere":
        return _surface(g, n)
    if dist == "mixed":
        nc = int(round(0.1 * n))
        return torch.cat([_surface(g, n - nc), _rand(g, nc, 3)]).contiguous()
    # Plummer-like cluster, scale 0.1, kept inside the unit cube by drawing again
    out = torch.empty(0, 3, dtype=torch.float64, device="cuda")
    while out.shape[0] < n:
        m = 2 * (n - out.shape[0]) + 256
        r = 0.1 / torch.sqrt(_rand(g, m).clamp(1e-12, 1.0 - 1e-12) ** (-2.0 / 3.0) - 1.0)
        d = _randn(g, m, 3)
        x = 0.5 + r[:, None] * d / d.norm(dim=1, keepdim=True)
        out = torch.cat([out, x[((x >= 0) & (x < 1)).all(dim=1)]])
    return out[:n].contiguous()


def _radius(case, n):
    return case["a"] if case["a"] > 0 else 0.5 / n ** (1.0 / 3.0)


def _sizes(case):
    """Sizes of a batch: log-uniform, the same for every seed (a pass of a case is one amount of work)."""
    k = case["nsys"]
    u = np.random.default_rng(k).random(k)
    u[0], u[-1] = 0.0, 1.0
    return [int(round(math.exp(math.log(case["lo"]) + v * math.log(case["hi"] / case["lo"])))) for v in u]


def _batch(case, g):
    """Systems of a batch: alternately a uniform cube and a cluster (forest) or a sphere surface (serve)."""
    other = "plummer" if case["kind"] == "forest" else "sphere"
    out = []
    for i, n in enumerate(_sizes(case)):
        pos = _positions(g, "cube" if i % 2 == 0 else other, n)
        f = _randn(g, n, 3)
        out.append((pos, f, 0.5 / n ** (1.0 / 3.0)))
    return out


def _serve_setting(i):
    return (3, rp.RPY_FP32) if i % 2 == 0 else (6, rp.RPY_FP64)


def _pinned(x):
    h = torch.empty(x.shape, dtype=x.dtype, pin_memory=True)
    h.copy_(x)
    return h


class _Server:
    """A server handle, destroyed with its state."""

    def __init__(self):
        self.handle = rp.rpy_server_create(slots=4)

    def __del__(self):
        if self.handle:
            rp.rpy_server_destroy(self.handle)
            self.handle = None


def _inputs(case, seed):
    g = _gen(seed)
    if case["dist"] == "batch":
        return _batch(case, g)
    n = case["n"]
    pos = _positions(g, case["dist"], n)
    f = _randn(g, n, 3)
    if case["kind"] == "evaluate":
        return pos, f, _rand(g, case["nt"], 3)
    return pos, f


def _build(case, pos, offsets, a):
    return rp.rpy_forest_build(pos, offsets, a, case["digits"], leaf_cap=case["leaf_cap"], precision=case["prec"],
                               order_p=case["p"], quad=case["quad"])


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind in ("forest", "serve"):
        systems = _inputs(case, seed)
        if kind == "forest":
            off = np.concatenate([[0], np.cumsum([x.shape[0] for x, _, _ in systems])]).astype(np.int64)
            a = np.array([r for _, _, r in systems])
            st["s"] = 6 * math.pi * a
            st["f"] = torch.cat([f for _, f, _ in systems]).contiguous()
            st["u"] = torch.empty_like(st["f"])
            st["tree"] = _build(case, torch.cat([x for x, _, _ in systems]).contiguous(), off, a)
        else:
            st["server"] = _Server()
            st["req"] = []
            for i, (x, f, r) in enumerate(systems):
                d, prec = _serve_setting(i)
                hx, hf = _pinned(x), _pinned(f)
                sid = rp.rpy_server_add_system(st["server"].handle, hx.numpy(), r, d, precision=prec)
                st["req"].append((sid, hx, hf, 6 * math.pi * r, torch.empty_like(hf).pin_memory()))
        return st
    data = _inputs(case, seed)
    n = case["n"]
    a = _radius(case, n)
    st.update(pos=data[0], f=data[1], a=a, s=6 * math.pi * a)
    if kind == "evaluate":
        st["tgt"] = data[2]
        st["u"] = torch.empty_like(data[2])
        return st
    st["u"] = torch.empty_like(st["f"])
    if kind != "oneshot":
        st["tree"] = _build(case, st["pos"], [0, n], [a])
    if kind == "host":
        st["hpos"], st["hf"], st["hu"] = _pinned(st["pos"]), _pinned(st["f"]), _pinned(st["u"])
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "matvec":
        rp.rpy_matvec(st["tree"], st["f"], st["s"], st["u"])
    elif kind == "step":
        rp.rpy_tree_update_positions(st["tree"], st["pos"])
        rp.rpy_matvec(st["tree"], st["f"], st["s"], st["u"])
    elif kind == "forest":
        rp.rpy_forest_matvec(st["tree"], st["f"], st["s"], st["u"])
    elif kind == "oneshot":
        rp.rpy_matvec_oneshot(st["pos"], case["n"], st["a"], st["f"], st["s"], case["digits"], st["u"])
    elif kind == "evaluate":
        rp.rpy_evaluate(st["pos"], st["f"], st["tgt"], st["a"], st["s"], case["digits"], st["u"], precision=case["prec"],
                        leaf_cap=case["leaf_cap"], order_p=case["p"], quad=case["quad"])
    elif kind == "noise":
        rp.rpy_lanczos_sqrt(st["tree"], st["f"], st["s"], st["u"], m_max=case["steps"], tol=0.0)
    elif kind == "host":
        rp.rpy_tree_matvec_host(st["tree"], st["hpos"].numpy(), st["hf"].numpy(), st["s"], st["hu"].numpy())
        return st["hu"]
    else:
        h = st["server"].handle
        ids = [rp.rpy_server_submit(h, sid, x.numpy(), f.numpy(), s, u.numpy()) for sid, x, f, s, u in st["req"]]
        for rid in ids:
            status, _ = rp.rpy_server_wait(h, rid)
            if status != 0:
                raise rp.RpyError(status, "rpy_server_wait")
        return [u for _, _, _, _, u in st["req"]]
    return st["u"]


# ---------------------------------------------------------------- work and accuracy

def _matvec_work(n, digits, dist, leaf_cap, p, quad):
    """FLOPs of one matvec by the method's operation counts: near pairs (33 each; a leaf of half the
    capacity and its neighbours, 27 in a volume, 12 on a surface), and per box the plane-wave sums of three frames
    and four sets (node sums and angle sums, out and in) with about 12 shifted sources per box and direction;
    per bead the multipole and local evaluations."""
    cap, p, quad = leaf_cap or LEAF[digits], p or ORDER[digits], quad or digits
    occ = min(n, 0.5 * cap)
    near = n * min(n, occ * (27 if dist in ("cube", "plummer", "batch") else 12)) * 33.0
    if n <= cap:
        return n * n * 33.0
    nc, S, s = (p + 1) * (p + 2) / 2, WAVES[quad] / 2, NODES[quad]
    box = 3 * 4 * 2 * 2 * (2 * nc * s + 2 * S * (p + 1)) + 6 * 4 * S * 8 * 12
    return near + 1.2 * n / occ * box + n * nc * 4 * (4 + 6 + 6)


def _items(case):
    """(n, digits, prec, dist) of each system of a case."""
    if case["dist"] == "batch":
        for i, n in enumerate(_sizes(case)):
            d = _serve_setting(i)[0] if case["kind"] == "serve" else case["digits"]
            yield n, d, "cube"
    else:
        yield case["n"] + case.get("nt", 0), case["digits"], case["dist"]


def work(case):
    fl, n = 0.0, 0
    for m, d, dist in _items(case):
        fl += _matvec_work(m, d, dist, case["leaf_cap"], case["p"], case["quad"])
        n += m
    if case["kind"] == "noise":
        fl *= case["steps"]
    # positions and forces read once, velocities written once
    return {"bytes": 72.0 * n, "flops": fl}


def tolerance(case):
    """About four times the distance to the direct sum that was measured over listed and drawn cases
    (the truncation of the expansions; the rounding of either precision is below it): mostly
    1e-4 ... 2.5e-4 and up to 6.3e-4 at 3 digits, 1e-7 ... 3.6e-7 and up to 7.5e-7 at 6,
    1.7e-10 ... 1.5e-9 at 9."""
    tol = {3: 2e-3, 6: 2e-6, 9: 5e-9}
    return {"rel": tol[3 if case["kind"] == "serve" else case["digits"]]}


def _direct(xt, xs, f, a, s):
    """u at the points xt from the forces f at xs, in 64 bits, over blocks of targets; a pair at
    distance 0 takes the r -> 0 limit (which is the self term when the point is the bead itself)."""
    u = torch.empty_like(xt)
    co, cf = s / (6 * math.pi * a), s / (8 * math.pi)
    step = max(1, (1 << 21) // xs.shape[0])
    for i in range(0, xt.shape[0], step):
        d = [xt[i:i + step, k, None] - xs[None, :, k] for k in range(3)]
        r2 = d[0] * d[0]
        r2.addcmul_(d[1], d[1]).addcmul_(d[2], d[2])
        rf = d[0] * f[:, 0]
        rf.addcmul_(d[1], f[None, :, 1]).addcmul_(d[2], f[None, :, 2])
        r = r2.sqrt()
        far = r >= 2 * a
        ri = 1.0 / torch.where(r > 0, r, torch.ones_like(r))
        v = (2 * a * a) * ri * ri
        t1 = torch.where(far, cf * ri * (1 + v / 3), co * (1 - (9 / (32 * a)) * r))
        t2 = torch.where(far, cf * ri * (1 - v) * ri * ri, torch.where(r > 0, co * (3 / (32 * a)) * ri, 0.0))
        t2.mul_(rf)
        for k in range(3):
            u[i:i + step, k] = t1 @ f[:, k] + (t2 * d[k]).sum(dim=1)
    return u


def _sqrt_action(x, z, a, s, steps):
    """|z| V T^{1/2} e_1 of so many Lanczos steps on the direct sum, fully reorthogonalised."""
    nz = z.norm()
    V = [z.reshape(-1) / nz]
    al, be = [], []
    while True:
        w = _direct(x, x, V[-1].reshape(-1, 3), a, s).reshape(-1)
        al.append(float(w @ V[-1]))
        if len(al) == steps:
            break
        B = torch.stack(V)
        for _ in range(2):
            w = w - B.T @ (B @ w)
        be.append(float(w.norm()))
        V.append(w / be[-1])
    lam, q = np.linalg.eigh(np.diag(al) + np.diag(be, 1) + np.diag(be, -1))
    c = torch.tensor(q @ (np.sqrt(np.maximum(lam, 0)) * q[0]), dtype=torch.float64, device=z.device)
    return (nz * (c @ torch.stack(V))).reshape(-1, 3)


def exact(case, seed):
    kind = case["kind"]
    if case["dist"] == "batch":
        if sum(n * n for n in _sizes(case)) > EXACT_PAIRS:
            return None
        us = [_direct(x, x, f, a, 6 * math.pi * a) for x, f, a in _inputs(case, seed)]
        return torch.cat(us) if kind == "forest" else us
    n = case["n"]
    pairs = n * case["nt"] if kind == "evaluate" else n * n * case.get("steps", 1)
    if pairs > EXACT_PAIRS:
        return None
    data = _inputs(case, seed)
    a = _radius(case, n)
    s = 6 * math.pi * a
    if kind == "evaluate":
        return _direct(data[2], data[0], data[1], a, s)
    if kind == "noise":
        return _sqrt_action(data[0], data[1], a, s, case["steps"])
    return _direct(data[0], data[0], data[1], a, s)
