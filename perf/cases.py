"""The work a program hands to this library, as cases that can be timed and checked.

A case is a dict of plain values.  Its "path" names the entry point:
  poisson  Plan.execute / execute_f64 / execute_host: one solve u = scale dx^2 G * f
  ragged   Plan.execute on many independent solves of different box edges
  ifactor  Plan.ifactor: y = M E_Q(alpha) M x, once per alpha of the case
  step     RKPlan.step: one IF-HERK step
  refresh  RKPlan.refresh: velocity refresh u = C^T (-L^-1 C u)
  ops      RKPlan.op: every staggered-grid operator once
Geometry (boxes, block lists) comes from the case alone, field values from the case and
the seed.  `exact` evaluates the same sums in 64 bits with torch alone: the lattice Green's
function from its Bessel integral, free-space convolutions by zero-padded FFTs.
"""
import math

import numpy as np
import torch

from paper_1601_00035_gb300 import lgf

DEV = "cuda"
UINF = (0.0, 0.0, -0.18686)  # free stream of the Re = 500 ring
RE = 500.0


def listed():
    return [
        # the smallest solve: one scalar 32^3 box of Gaussian blobs (launch latency counts)
        {"name": "blobs32", "path": "poisson", "shape": "blobs", "edge": 32, "B": 16, "ncomp": 1},
        # the same solve for callers that need FP64 data and transforms
        {"name": "blobs32_f64", "path": "poisson", "shape": "blobs", "edge": 32, "B": 16, "ncomp": 1, "f64": True},
        # an odd box edge on 8^3 blocks, dense source, launched without a graph
        {"name": "blobs77_b8", "path": "poisson", "shape": "blobs", "edge": 77, "B": 8, "ncomp": 1},
        # streamfunction of a thin-core vortex ring in a 128^3 box, three components, one graph
        {"name": "ring128", "path": "poisson", "shape": "ring", "edge": 128, "B": 16, "ncomp": 3, "graph": True,
         "R": 32.0, "sigma": 3.0, "tilt": 1.49, "azimuth": 0.6, "threshold": 1e-14},
        # the same solve for a program whose fields live in page-locked host memory
        {"name": "ring128_host", "path": "poisson", "shape": "ring", "edge": 128, "B": 16, "ncomp": 3, "graph": True,
         "R": 32.0, "sigma": 3.0, "tilt": 1.49, "azimuth": 0.6, "threshold": 1e-14, "host": True},
        # integrating factors of one velocity field at three time steps (tap radius 7, 9, 15)
        {"name": "ifactor128", "path": "ifactor", "edge": 128, "B": 16, "ncomp": 3, "alphas": "0.05,0.2,1.0"},
        # a batch of independent ring solves, box edges 24..192, one graph
        {"name": "ragged64", "path": "ragged", "n": 64, "emin": 24, "emax": 192, "B": 16, "graph": True, "geometry": 5},
        # pressure solve of a projection: scalar, shell-shaped support, targets one block wider
        {"name": "shell256", "path": "poisson", "shape": "shell", "B": 16, "ncomp": 1, "graph": True,
         "R": 50.0, "sigma": 10.0, "tilt": 0.9, "azimuth": 2.1, "threshold": 1e-6},
        # the stencils of a stage on the same ring's blocks
        {"name": "ops256", "path": "ops", "B": 16, "R": 50.0, "sigma": 10.0, "tilt": 0.9, "azimuth": 2.1,
         "threshold": 1e-6},
        # velocity refresh of that ring: a vector solve between two curls
        {"name": "refresh256", "path": "refresh", "B": 16, "R": 50.0, "sigma": 10.0, "tilt": 0.9, "azimuth": 2.1,
         "threshold": 1e-6},
        # one full time step of that ring, replayed as a graph
        {"name": "step256", "path": "step", "B": 16, "R": 50.0, "sigma": 10.0, "tilt": 0.9, "azimuth": 2.1,
         "threshold": 1e-6, "scheme": 0, "graph": True},
        # the thin ring (core 1/80 of the radius) whose box is too wide for the whole-box FFTs:
        # the block-sparse solve
        {"name": "thinring", "path": "poisson", "shape": "shell", "B": 16, "ncomp": 1, "graph": True, "method": 1,
         "R": 400.0, "sigma": 5.0, "tilt": 0.9, "azimuth": 2.1, "threshold": 1e-6},
    ]


def draw(rng):
    def logu(a, b):
        return math.exp(rng.uniform(math.log(a), math.log(b)))

    def ring(lo, hi, thick):
        R = logu(lo, hi)
        return {"R": round(R, 2), "sigma": round(R * thick, 2), "tilt": round(rng.uniform(0.0, 1.57), 3),
                "azimuth": round(rng.uniform(0.0, 6.28), 3), "threshold": 1e-6}

    graph = rng.random() < 0.5
    kind = rng.choice(["blobs", "blobs", "ring", "shell", "thin", "ifactor", "ragged", "step", "refresh", "ops"])
    if kind == "blobs":
        f64 = rng.random() < 0.25
        return {"path": "poisson", "shape": "blobs", "edge": int(round(logu(24, 96 if f64 else 160))),
                "B": rng.choice([8, 16, 32]), "ncomp": rng.choice([1, 1, 3]), "f64": f64, "graph": graph}
    if kind == "ring":
        e = int(round(logu(48, 160)))
        R = round(rng.uniform(0.15, 0.25) * e, 2)
        return {"path": "poisson", "shape": "ring", "edge": e, "B": rng.choice([8, 16]), "ncomp": 3, "graph": graph,
                "R": R, "sigma": round(R / rng.uniform(5, 11), 2), "tilt": round(rng.uniform(0.0, 1.57), 3),
                "azimuth": round(rng.uniform(0.0, 6.28), 3), "threshold": 1e-14, "host": rng.random() < 0.25}
    if kind == "shell":
        return {"path": "poisson", "shape": "shell", "B": rng.choice([8, 16]), "ncomp": rng.choice([1, 1, 3]),
                "graph": graph, **ring(20, 60, rng.uniform(0.1, 0.2))}
    if kind == "thin":
        return {"path": "poisson", "shape": "shell", "B": 16, "ncomp": 1, "graph": graph, "method": 1,
                "far_tc": rng.random() < 0.3, **ring(60, 400, 0.0), "sigma": round(rng.uniform(3.0, 5.0), 2)}
    if kind == "ifactor":
        B = rng.choice([8, 16, 16])
        return {"path": "ifactor", "edge": int(round(logu(32, 160))), "B": B, "ncomp": rng.choice([1, 3]),
                "alphas": "%.4f" % logu(0.02, 0.08 if B == 8 else 1.0)}
    if kind == "ragged":
        return {"path": "ragged", "n": rng.randint(4, 64), "emin": 24, "emax": rng.choice([64, 96, 128, 192]),
                "B": rng.choice([8, 16, 32]), "graph": graph, "geometry": rng.randint(0, 1 << 20)}
    c = {"path": kind, "B": rng.choice([8, 16, 16]), **ring(18, 56, rng.uniform(0.12, 0.2))}
    if kind == "step":
        c.update(scheme=rng.choice([0, 1, 2]), graph=graph)
    return c


# ---------------------------------------------------------------------------
# fields
# ---------------------------------------------------------------------------
def _axes(tilt, azimuth):
    """Rows: the ring frame's x, y, z axes (z = the ring axis, tilted from e_z)."""
    ct, st, cp, sp = math.cos(tilt), math.sin(tilt), math.cos(azimuth), math.sin(azimuth)
    return torch.tensor([[ct * cp, ct * sp, -st], [-sp, cp, 0.0], [st * cp, st * sp, ct]], dtype=torch.float64,
                        device=DEV)


def _swirl(seed, n=4):
    """Azimuthal modes of the circulation: amplitudes and phases that the seed sets."""
    r = np.random.default_rng(seed)
    return 1.0 + 0.1 * r.uniform(-1, 1), 0.15 * r.uniform(-1, 1, n), r.uniform(0, 2 * math.pi, n)


def _ring(pts, R, sigma, M, modes=None):
    """Vorticity [n, 3] of a Gaussian-core ring at points [n, 3] in its centre's frame."""
    p = pts @ M.T
    rho = torch.hypot(p[:, 0], p[:, 1]).clamp_min(1e-300)
    w = torch.exp(-(p[:, 2] ** 2 + (rho - R) ** 2) / sigma ** 2) / (math.pi * sigma ** 2)
    if modes is not None:
        amp, a, ph = modes
        th = torch.atan2(p[:, 1], p[:, 0])
        w = w * (amp + sum(float(a[m]) * torch.cos((m + 1) * th + float(ph[m])) for m in range(len(a))))
    z = torch.zeros_like(w)
    return torch.stack([-w * p[:, 1] / rho, w * p[:, 0] / rho, z], 1) @ M


def _cells(blocks, B):
    """Cell indices [nblk * B^3, 3] of the listed blocks in field order, FP64 on the GPU."""
    r = torch.arange(B, dtype=torch.float64, device=DEV)
    z, y, x = torch.meshgrid(r, r, r, indexing="ij")
    loc = torch.stack([x, y, z], -1).reshape(1, -1, 3)
    b = torch.as_tensor(blocks, dtype=torch.float64, device=DEV).reshape(-1, 1, 3)
    return (b * B + loc).reshape(-1, 3)


def _ring_field(blocks, B, c, centre, modes):
    """Edge-sampled ring vorticity [nblk, 3, B, B, B] in FP64."""
    M, pts = _axes(c["tilt"], c["azimuth"]), _cells(blocks, B) - centre
    out = torch.empty((len(blocks), 3, B, B, B), dtype=torch.float64, device=DEV)
    for q in range(3):
        shift = torch.zeros(3, dtype=torch.float64, device=DEV)
        shift[q] = 0.5
        out[:, q] = _ring(pts - shift, c["R"], c["sigma"], M, modes)[:, q].reshape(-1, B, B, B)
    return out


def _box_blocks(edge, B):
    n = (edge + B - 1) // B
    z, y, x = np.meshgrid(*[np.arange(n)] * 3, indexing="ij")
    return np.stack([x.ravel(), y.ravel(), z.ravel()], 1).astype(np.int32)


def _active(cand, B, c, centre):
    w = _ring_field(cand, B, c, centre, None).abs().flatten(1).amax(1)
    return cand[(w > c["threshold"] * w.max()).cpu().numpy()]


def _ring_blocks(c):
    """Blocks near the torus of a ring centred at the origin that hold vorticity above the threshold."""
    B = c["B"]
    reach = 6.0 * c["sigma"] + B
    g = np.arange(-int((c["R"] + reach) // B) - 2, int((c["R"] + reach) // B) + 3)
    z, y, x = np.meshgrid(g, g, g, indexing="ij")
    cand = np.stack([x.ravel(), y.ravel(), z.ravel()], 1).astype(np.int32)
    p = ((cand + 0.5) * B) @ _axes(c["tilt"], c["azimuth"]).cpu().numpy().T
    near = np.hypot(np.hypot(p[:, 0], p[:, 1]) - c["R"], p[:, 2]) < reach
    return _active(cand[near], B, c, 0.0)


def _dilate(blocks):
    o = np.array([[x, y, z] for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)])
    return np.unique((blocks[:, None] + o).reshape(-1, 3), axis=0).astype(np.int32)


def _geometry(c):
    """(source blocks, target blocks, ring centre) of a Poisson case."""
    B = c["B"]
    if c["shape"] == "shell":
        src = _ring_blocks(c)
        return src, _dilate(src), 0.0
    dst = _box_blocks(c["edge"], B)
    return (_active(dst, B, c, c["edge"] / 2) if c["shape"] == "ring" else dst), dst, c["edge"] / 2


def _blobs(c, seed, blocks):
    """Three Gaussian blobs per component, zero outside the box's cells."""
    B, e, r = c["B"], c["edge"], np.random.default_rng(seed)
    p = _cells(blocks, B)
    inside = (p < e).all(1)
    out = []
    for _ in range(c["ncomp"]):
        f = torch.zeros(len(p), dtype=torch.float64, device=DEV)
        for _ in range(3):
            amp = r.uniform(-1, 1)
            cen = torch.tensor(e / 2 - 0.5 + r.uniform(-e / 4, e / 4, 3), device=DEV)
            f += amp * torch.exp(-((p - cen) ** 2).sum(1) / (2 * (3 * e / 32) ** 2))
        out.append((f * inside).reshape(-1, B, B, B))
    return torch.stack(out, 1)


def _source(c, seed, src, centre):
    f = _blobs(c, seed, src) if c["shape"] == "blobs" else _ring_field(src, c["B"], c, centre, _swirl(seed))
    return f[:, :c["ncomp"]].to(torch.float64 if c.get("f64") else torch.float32).contiguous()


def _ragged(c):
    """Per solve: edge and ring parameters, set by the case's geometry number."""
    r, out = np.random.default_rng(c["geometry"]), []
    for _ in range(c["n"]):
        e = int(round(math.exp(r.uniform(math.log(c["emin"]), math.log(c["emax"])))))
        R = r.uniform(4.0, max(4.0, min(40.0, (e / 2 - 2) / 1.75)))
        out.append({"path": "poisson", "shape": "ring", "edge": e, "B": c["B"], "ncomp": 1, "R": R, "sigma": R / 8,
                    "tilt": r.uniform(0.3, 1.57), "azimuth": r.uniform(0, 6.28), "threshold": 1e-14})
    return out


def _rk(c):
    dx = 1.0 / c["R"]
    return dx, 0.01721 * 50.0 * dx  # a fixed CFL number


def _rk_plan(c, soln):
    dx, dt = _rk(c)
    return lgf.RKPlan(c["B"], soln, dx, dt, RE, scheme=c.get("scheme", 0), use_graph=bool(c.get("graph")))


def _xsoln(soln):
    """The dilation in the order RKPlan.blocks(0) gives: the solution blocks first."""
    order = {tuple(b): None for b in soln.tolist()}
    for b in soln.tolist():
        for z in (-1, 0, 1):
            for y in (-1, 0, 1):
                for x in (-1, 0, 1):
                    order.setdefault((b[0] + x, b[1] + y, b[2] + z))
    return np.array(list(order), dtype=np.int32)


def _velocity(c, seed, soln, xs):
    """Velocity [nblk, 3, B, B, B] of the perturbed ring, from its vorticity in 64 bits."""
    B, (dx, _) = c["B"], _rk(c)
    box = _Box(xs, B)
    w = box.dense(soln, _ring_field(soln, B, c, 0.0, _swirl(seed)) / dx ** 2)
    a = box.masked(_convolve(w, -dx * dx))
    return box.blocks(xs, _curl_t(a, dx)).float().contiguous()


# ---------------------------------------------------------------------------
# the timed calls
# ---------------------------------------------------------------------------
def _table(pairs, B):
    K = max(lgf.required_max_offset(s, d, B) for s, d in pairs)
    return lgf.Table(lgf.LAPLACE7, max_offset=K)


def prepare(case, seed):
    c, B = case, case["B"]
    if c["path"] == "poisson":
        src, dst, centre = _geometry(c)
        f = _source(c, seed, src, centre)
        o = torch.zeros((len(dst), c["ncomp"], B, B, B), dtype=f.dtype, device=DEV)
        split = c.get("method", 0) == 1
        t = lgf.Table(lgf.LAPLACE7, max_offset=31) if split else _table([(src, dst)], B)
        plan = lgf.Plan(t, [lgf.Solve(B, c["ncomp"], src, dst, scale=-1.0)], use_graph=bool(c.get("graph")),
                        precision=int(bool(c.get("f64"))), method=int(split), far_precision=int(bool(c.get("far_tc"))))
        call = "execute_host" if c.get("host") else "execute_f64" if c.get("f64") else "execute"
        if c.get("host"):
            f, o = f.cpu().pin_memory(), o.cpu().pin_memory()
        return {"path": "poisson", "call": getattr(plan, call), "src": [f], "dst": [o]}
    if c["path"] == "ragged":
        solves, src, dst, pairs = [], [], [], []
        for j, q in enumerate(_ragged(c)):
            sb, db, centre = _geometry(q)
            pairs.append((sb, db))
            solves.append(lgf.Solve(B, 1, sb, db, scale=-1.0))
            src.append(_source(q, seed * 1000 + j, sb, centre))
            dst.append(torch.zeros((len(db), 1, B, B, B), device=DEV))
        plan = lgf.Plan(_table(pairs, B), solves, use_graph=bool(c.get("graph")))
        return {"path": "poisson", "call": plan.execute, "src": src, "dst": dst}
    if c["path"] == "ifactor":
        blocks = _box_blocks(c["edge"], B)
        x = _if_field(c, seed, blocks)
        plans = [lgf.Plan(lgf.Table(lgf.IFACTOR, alpha=float(a)), [lgf.Solve(B, c["ncomp"], blocks, None)])
                 for a in c["alphas"].split(",")]
        return {"path": "ifactor", "plans": plans, "x": x, "y": [torch.zeros_like(x) for _ in plans]}
    soln = _ring_blocks(c)
    plan = _rk_plan(c, soln)
    u = _velocity(c, seed, soln, plan.blocks(0))
    st = {"path": c["path"], "plan": plan, "u": u, "out": torch.zeros_like(u)}
    if c["path"] == "ops":
        st["out"] = [torch.zeros_like(u) for _ in range(5)]
        st["out"][2] = torch.zeros_like(u[:, :1])
        st["cell"] = u[:, :1].contiguous()
    return st


def run(state):
    if state["path"] == "poisson":
        state["call"](state["src"], state["dst"])
        return state["dst"]
    if state["path"] == "ifactor":
        for p, y in zip(state["plans"], state["y"]):
            p.ifactor(state["x"], y)
        return state["y"]
    plan, u, out = state["plan"], state["u"], state["out"]
    if state["path"] == "step":
        plan.step(u, out, UINF)
    elif state["path"] == "refresh":
        plan.refresh(u, out)
    else:
        plan.op(lgf.OP_CURL, u, out[0])
        plan.op(lgf.OP_CURL_T, u, out[1])
        plan.op(lgf.OP_DIV_T, u, out[2])
        plan.op(lgf.OP_GRAD, state["cell"], out[3])
        plan.op(lgf.OP_NONLINEAR, u, out[4], 1.0, UINF)
    return out


def _if_field(c, seed, blocks):
    """Smooth velocity-like field: a few Gaussian eddies per component, zero outside the box's cells."""
    return _blobs({**c, "shape": "blobs"}, seed, blocks).float().contiguous()


def work(case):
    """Each input read once, each output written once; flops: per solve the smaller of the padded-box
    FFTs (2.5 P log2 P each way, P = the box of twice the extents) and 1500 per target point (near
    spectra and interpolated far field), 12 R + 6 per point for an integrating factor of radius R."""
    c, B = case, case["B"]

    def solve(src, dst, nc):
        ext = np.concatenate([src, dst])
        P = float(np.prod(2.0 * B * (ext.max(0) - ext.min(0) + 1)))
        return nc * min(5.0 * P * math.log2(P), 1500.0 * len(dst) * B ** 3), nc * (len(src) + len(dst)) * B ** 3

    if c["path"] == "poisson":
        src, dst, _ = _geometry(c)
        fl, n = solve(src, dst, c["ncomp"])
        return {"bytes": (8 if c.get("f64") else 4) * n, "flops": fl}
    if c["path"] == "ragged":
        w = [solve(*_geometry(q)[:2], 1) for q in _ragged(c)]
        return {"bytes": 4 * sum(n for _, n in w), "flops": sum(f for f, _ in w)}
    if c["path"] == "ifactor":
        n = c["ncomp"] * len(_box_blocks(c["edge"], B)) * B ** 3
        al = [float(a) for a in c["alphas"].split(",")]
        return {"bytes": 4 * n * (1 + len(al)), "flops": float(sum(n * (12 * _radius(a) + 6) for a in al))}
    soln = _ring_blocks(c)
    xs = _xsoln(soln)
    n = len(xs) * B ** 3
    if c["path"] == "ops":
        return {"bytes": 4 * n * (3 + 1 + 3 + 3 + 1 + 3 + 3), "flops": float(n * (12 + 12 + 6 + 6 + 90))}
    if c["path"] == "refresh":
        return {"bytes": 24 * n, "flops": solve(soln, xs, 3)[0] + 24.0 * n}
    dx, dt = _rk(c)
    e = _exponents(c.get("scheme", 0), dt / (dx * dx * RE))
    ifs = sum(3 * n * (12 * _radius(a) + 6) * k for a, k in zip(e, (3, 2, 1)) if a > 0)
    return {"bytes": 24 * n, "flops": float(3 * (solve(soln, xs, 1)[0] + 110.0 * n) + ifs)}


# ---------------------------------------------------------------------------
# 64-bit results
# ---------------------------------------------------------------------------
def _bessel(x, nmax):
    """e^{-x} I_n(x), n = 0..nmax, for a vector of x > 0: [len(x), nmax + 1].  Up to 5e7 the cosine
    coefficients of exp(x (cos t - 1)) by an FFT, beyond it Hankel's series."""
    out = torch.empty((len(x), nmax + 1), dtype=torch.float64, device=DEV)
    small = x < 5e7
    for lo, hi, M in ((0.0, 1e4, 1 << 13), (1e4, 5e7, 1 << 17)):
        idx = torch.nonzero((x >= lo) & (x < hi)).flatten()
        M = max(M, 1 << (4 * nmax + 64).bit_length())
        s = torch.sin(torch.arange(M, dtype=torch.float64, device=DEV) * (math.pi / M)) ** 2
        for part in idx.split(64) if len(idx) else ():
            f = torch.exp(-2.0 * x[part, None] * s)
            out[part] = torch.fft.rfft(f).real[:, :nmax + 1] / M
    big = torch.nonzero(~small).flatten()
    if len(big):
        mu = 4.0 * torch.arange(nmax + 1, dtype=torch.float64, device=DEV) ** 2
        xb = x[big, None]
        term = torch.ones((len(big), nmax + 1), dtype=torch.float64, device=DEV)
        tot = term.clone()
        for k in range(1, 14):
            term = term * (-(mu - (2 * k - 1) ** 2) / (k * 8.0 * xb))
            tot += term
        out[big] = tot / torch.sqrt(2 * math.pi * xb)
    return out


def _lgf_box(nx, ny, nz):
    """G(a, b, c) = -int_0^inf prod e^{-2t} I(2t) dt for 0 <= a < nx, ..: [nz, ny, nx].  Trapezoid in
    log t, which converges geometrically: the integrand is analytic for |Im log t| < pi / 2."""
    h = 0.2
    t = torch.exp(torch.arange(-41.0, 80.0, h, dtype=torch.float64, device=DEV))
    f = _bessel(2.0 * t, max(nx, ny, nz) - 1)
    fyx = (f[:, :ny, None] * f[:, None, :nx]).reshape(len(t), -1)
    return -((f[:, :nz] * (h * t)[:, None]).T @ fyx).reshape(nz, ny, nx)


def _even(n):
    """A length >= n with small prime factors."""
    while True:
        m = n
        for p in (2, 3, 5, 7):
            while m % p == 0:
                m //= p
        if m == 1 and n % 2 == 0:
            return n
        n += 1


def _convolve(f, scale, G=None):
    """scale * sum_m G(n - m) f(m) on f's own box; f [.., nz, ny, nx] FP64."""
    E = f.shape[-3:]
    L = [_even(2 * e - 1) for e in E]
    if G is None:
        G = _lgf_box(E[2], E[1], E[0])
    k = torch.zeros(L, dtype=torch.float64, device=DEV)
    iy, ix = (torch.cat([torch.arange(e, device=DEV), torch.arange(e - 1, 0, -1, device=DEV)]) for e in E[1:])
    py, px = (torch.cat([torch.arange(e, device=DEV), torch.arange(l - e + 1, l, device=DEV)]) for e, l in zip(E[1:], L[1:]))
    for z in range(E[0]):
        plane = G[z][iy][:, ix]
        for zz in {z, (L[0] - z) % L[0]}:
            k[zz].index_put_((py[:, None], px[None]), plane)
    kh = torch.fft.rfftn(k)
    del k
    out = torch.empty_like(f)
    for o, s in zip(out.reshape(-1, *E), f.reshape(-1, *E)):
        sh = torch.fft.rfftn(s, s=L)
        sh *= kh
        o.copy_(torch.fft.irfftn(sh, s=L)[:E[0], :E[1], :E[2]])
        del sh
    return out.mul_(scale)


class _Box:
    """A dense box around a block list, with a block's margin of zeros on every side."""

    def __init__(self, blocks, B, margin=1):
        self.B, self.lo = B, blocks.min(0) - margin
        self.nb = (blocks.max(0) + margin + 1 - self.lo)[::-1]  # z, y, x
        self.mask = self.dense(blocks, torch.ones((len(blocks), 1, B, B, B), dtype=torch.float64, device=DEV))

    def _index(self, blocks):
        p = torch.as_tensor(np.asarray(blocks) - self.lo, device=DEV).long()
        return (p[:, 2] * int(self.nb[1]) + p[:, 1]) * int(self.nb[2]) + p[:, 0]

    def dense(self, blocks, v):
        """[nblk, c, B, B, B] -> [c, Z, Y, X] FP64."""
        B, nc = self.B, v.shape[1]
        nz, ny, nx = (int(n) for n in self.nb)
        d = torch.zeros((nz * ny * nx, nc, B, B, B), dtype=torch.float64, device=DEV)
        d[self._index(blocks)] = v.to(DEV, torch.float64)
        d = d.reshape(nz, ny, nx, nc, B, B, B).permute(3, 0, 4, 1, 5, 2, 6)
        return d.reshape(nc, nz * B, ny * B, nx * B)

    def blocks(self, blocks, d):
        B, nc = self.B, d.shape[0]
        nz, ny, nx = (int(n) for n in self.nb)
        v = d.reshape(nc, nz, B, ny, B, nx, B).permute(1, 3, 5, 0, 2, 4, 6).reshape(nz * ny * nx, nc, B, B, B)
        return v[self._index(blocks)]

    def masked(self, d):
        return d * self.mask


def _at(f, q, d):
    """f at n + d e_q (axes x, y, z are the last, second and third from the end)."""
    return torch.roll(f, -d, dims=-(1 + q))


def _curl(f, dx):
    out = torch.empty_like(f)
    for q in range(3):
        r, s = (q + 1) % 3, (q + 2) % 3
        out[q] = (f[r] - _at(f[r], s, 1) + _at(f[s], r, 1) - f[s]) / dx
    return out


def _curl_t(e, dx):
    out = torch.empty_like(e)
    for q in range(3):
        r, s = (q + 1) % 3, (q + 2) % 3
        out[q] = (_at(e[r], s, -1) - e[r] + e[s] - _at(e[s], r, -1)) / dx
    return out


def _grad_t(f, dx):
    return sum(_at(f[q], q, -1) - f[q] for q in range(3))[None] / dx


def _grad(c, dx):
    return torch.stack([_at(c[0], q, 1) - c[0] for q in range(3)]) / dx


def _nonlinear(f, dx):
    e, out = _curl(f, dx), torch.empty_like(f)
    for q in range(3):
        r, s = (q + 1) % 3, (q + 2) % 3
        a = e[r] * (f[s] + _at(f[s], q, 1))
        b = e[s] * (f[r] + _at(f[r], q, 1))
        out[q] = 0.25 * (a + _at(a, s, -1) - b - _at(b, r, -1))
    return out


def _taps(alpha, n):
    return _bessel(torch.tensor([2.0 * alpha], dtype=torch.float64, device=DEV), n)[0]


def _radius(alpha):
    """Largest k whose tap times the centre tap squared is at least 1e-14."""
    g = [0.0] * 41
    for j in range(400):  # cosine coefficients on the host
        th = 2 * math.pi * j / 400
        w = math.exp(2 * alpha * (math.cos(th) - 1)) / 400
        for k in range(41):
            g[k] += w * math.cos(k * th)
    return max(k for k in range(41) if g[k] * g[0] ** 2 >= 1e-14)


def _ifactor(d, alpha):
    """E_Q(alpha) along the three axes of a dense box (zero outside it)."""
    for ax in (-1, -2, -3):
        n = d.shape[ax]
        g = _taps(alpha, 40)
        i = torch.arange(n, device=DEV)
        k = (i[:, None] - i[None]).abs()
        T = torch.where(k <= 40, g[k.clamp_max(40)], torch.zeros((), dtype=torch.float64, device=DEV))
        d = (d.transpose(ax, -1) @ T).transpose(ax, -1)
    return d


def _tableau(scheme):
    r3 = math.sqrt(3.0)
    return ([[0.5], [r3 / 3, (3 - r3) / 3], [(3 + r3) / 6, -r3 / 3, (3 + r3) / 6]],
            [[1 / 3], [-1.0, 2.0], [0.0, 0.75, 0.25]],
            [[8 / 15], [0.25, 5 / 12], [0.25, 0.0, 0.75]])[scheme]


def _exponents(scheme, alpha):
    a = _tableau(scheme)
    c = [0.0, sum(a[0]), sum(a[1]), 1.0]
    return [(c[i + 1] - c[i]) * alpha if c[i + 1] - c[i] > 1e-12 else 0.0 for i in range(3)]


def _step(u, box, soln, scheme, dx, dt):
    """One IF-HERK step on the dense box."""
    a = _tableau(scheme)
    supp = box.dense(soln, torch.ones((len(soln), 1, box.B, box.B, box.B), dtype=torch.float64, device=DEV))
    M, ex = box.masked, _exponents(scheme, dt / (dx * dx * RE))
    G = _lgf_box(u.shape[3], u.shape[2], u.shape[1])
    uinf = torch.tensor(UINF, dtype=torch.float64, device=DEV)[:, None, None, None]

    def H(i, x):
        return M(_ifactor(M(x), ex[i])) if ex[i] > 0 else x

    def g_of(v, aii):
        return -aii * dt * supp * _nonlinear(M(v + uinf), dx)

    def project(r, g):
        d = M(_convolve(supp * M(_grad_t(r, dx)), -dx * dx, G))
        gd = M(_grad(d, dx))
        return r - gd, g - gd

    g = g_of(u, a[0][0])
    t, w = project(u + g, g)
    w11 = w / (a[0][0] * dt)
    u1 = H(0, t)
    g = g_of(u1, a[1][1])
    t, w = project(H(0, u + dt * a[1][0] * w11) + g, g)
    w22 = w / (a[1][1] * dt)
    u2 = H(1, t)
    g = g_of(u2, a[2][2])
    r = H(1, H(0, u + dt * a[2][0] * w11) + dt * a[2][1] * w22) + g
    return H(2, project(r, g)[0])


def _solve(c, seed):
    src, dst, centre = _geometry(c)
    f = _source(c, seed, src, centre)
    box = _Box(np.concatenate([src, dst]), c["B"], margin=0)
    return box.blocks(dst, _convolve(box.dense(src, f), -1.0))


def exact(case, seed):
    c, B = case, case["B"]
    if c["path"] == "poisson":
        return [_solve(c, seed)]
    if c["path"] == "ragged":
        return [_solve(q, seed * 1000 + j) for j, q in enumerate(_ragged(c))]
    if c["path"] == "ifactor":
        blocks = _box_blocks(c["edge"], B)
        box = _Box(blocks, B, margin=0)
        x = box.dense(blocks, _if_field(c, seed, blocks))
        return [box.blocks(blocks, _ifactor(x, float(a))) for a in c["alphas"].split(",")]
    soln = _ring_blocks(c)
    xs = _xsoln(soln)
    dx, dt = _rk(c)
    box = _Box(xs, B)
    u = box.dense(xs, _velocity(c, seed, soln, xs))
    if c["path"] == "step":
        return box.blocks(xs, _step(u, box, soln, c["scheme"], dx, dt))
    keep = box.dense(soln, torch.ones((len(soln), 1, B, B, B), dtype=torch.float64, device=DEV))
    if c["path"] == "refresh":
        w = box.masked(_curl(u, dx)) * keep
        return box.blocks(xs, _curl_t(box.masked(_convolve(w, -dx * dx)), dx))
    uinf = torch.tensor(UINF, dtype=torch.float64, device=DEV)[:, None, None, None]
    out = [_curl(u, dx), _curl_t(u, dx), _grad_t(u, dx), _grad(u[:1], dx),
           keep * _nonlinear(box.masked(u + uinf), dx)]
    return [box.blocks(xs, o) for o in out]
