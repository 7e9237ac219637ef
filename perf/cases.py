"""What the speed of this library is measured on: single right-hand sides, SSP-RK3
steps and short whole solves through the public entry points of `weno` and `serve`.

The states are flows as they stand inside a run, not only its first instant: the
repository's initial data (Riemann tubes, the shock-density interaction, four
quadrants) with smooth waves of several lengths laid over them, so that the stencils
meet jumps, smooth variation and critical points together.
"""
import math

import numpy as np
import torch

from paper_2603_26272_gb300 import serve, weno

GAMMA = 1.4
EPS = MU0 = 1e-40

# A case: what is called ("rhs", "step", "step_host", "solve", "serve"), the system, the
# shape, the order, the precision, the boundary condition and the weight options.
_BASE = dict(call="rhs", system="euler", ndim=1, nbatch=1, nx=200, ny=1, order=6,
             precision="fp64", bc="transmissive", ai=True, alpha="field", data="tube", t=0.0)


def _case(**kw):
    c = dict(_BASE)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call a user's own time integrator makes: one right-hand side of a
        # 200-cell shock tube (launches and latency)
        _case(name="rhs_tube_200"),
        # a whole short solve of the 200-point periodic advection problem
        _case(name="solve_advection_200", call="solve", system="advection", bc="periodic",
              data="wave", t=0.5),
        # the first steps of the 1600-cell shock-density run: one 1D problem, short of filling the GPU
        _case(name="solve_shock_density_1600", call="solve", nx=1600, data="shock_density", t=0.05),
        # a parameter study: a batch of 64 Riemann problems of 1600 cells, one step
        _case(name="step_riemann_64x1600", call="step", nbatch=64, nx=1600),
        # small 2D grids, where a step does not fill the GPU
        _case(name="step_2d_128", call="step", ndim=2, nx=128, ny=128, data="quadrant"),
        # an odd, ragged, periodic grid
        _case(name="rhs_2d_501x333", ndim=2, nx=501, ny=333, bc="periodic", data="smooth"),
        # a state that lives in host memory: copy in, one step, copy out
        _case(name="step_host_2d_512", call="step_host", ndim=2, nx=512, ny=512, data="quadrant"),
        # weights without the affine-invariant descaler, as the paper's tables have them
        _case(name="rhs_2d_512_plain_weights", ndim=2, nx=512, ny=512, ai=False, data="quadrant"),
        # the widest member of the family
        _case(name="rhs_2d_512_order10", ndim=2, nx=512, ny=512, order=10, data="quadrant"),
        # the headline grid, one step in each precision mode
        _case(name="step_2d_2048", call="step", ndim=2, nx=2048, ny=2048, data="quadrant"),
        _case(name="step_2d_4096_fp32", call="step", ndim=2, nx=4096, ny=4096,
              precision="fp32_recon", data="quadrant"),
        # continuous batching: eight small solves of mixed shape and precision served together
        _case(name="serve_mixed_8", call="serve", nbatch=8, nx=4096, ny=256, data="tube", t=8.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["1d", "1d", "scalar", "2d", "2d", "2d", "2d"])
    call = rng.choice(["rhs", "step", "step"])
    if kind == "scalar":
        system = rng.choice(["advection", "burgers", "buckley_leverett"])
        return _case(call=call, system=system, nx=_log(rng, 80, 16384), nbatch=_log(rng, 1, 64),
                     bc="transmissive" if system == "buckley_leverett" else "periodic",
                     order=rng.choice([6, 6, 4, 8, 10]), data="wave")
    order = rng.choice([6, 6, 6, 6, 4, 8, 10])
    precision = rng.choice(["fp64", "fp64", "fp32_recon"]) if order == 6 else "fp64"
    opts = dict(call=call, order=order, precision=precision,
                bc=rng.choice(["transmissive", "transmissive", "periodic"]),
                ai=precision == "fp32_recon" or rng.random() < 0.85,
                alpha="single" if rng.random() < 0.15 else "field")
    if kind == "1d":
        return _case(nx=_log(rng, 100, 16384), nbatch=_log(rng, 1, 64),
                     data="smooth" if opts["bc"] == "periodic" else
                     rng.choice(["tube", "shock_density"]), **opts)
    top = 1024 if order > 6 else 2048
    if call == "step" and rng.random() < 0.2:
        opts["call"] = "step_host"
        top = 512
    return _case(ndim=2, nx=_log(rng, 48, top), ny=_log(rng, 48, top),
                 data="smooth" if opts["bc"] == "periodic" else "quadrant", **opts)


# ---------------------------------------------------------------------------
# Inputs.  Plain tensors on `dev`; the same numbers on every device are not needed,
# only the same numbers for the same seed on the same machine.
# ---------------------------------------------------------------------------
_DOMAIN = {"tube": (-5.0, 5.0), "shock_density": (-5.0, 5.0), "wave": (-1.0, 1.0),
           "quadrant": (0.0, 1.0), "smooth": (0.0, 1.0)}


def _waves(rng, nb, x, y, amp, kmax=8, modes=6):
    """A smooth field of relative size `amp` per problem: `modes` Fourier modes of up to
    `kmax` periods over the domain, shorter ones weaker; x, y in [0, 1] -> [nb][ny][nx]."""
    out = torch.zeros(nb, y.numel(), x.numel(), dtype=torch.float64, device=x.device)
    for b in range(nb):
        k = rng.integers(-kmax, kmax + 1, size=(modes, 2))
        ph = rng.uniform(0, 2 * math.pi, size=modes)
        for (kx, ky), f in zip(k.tolist(), ph.tolist()):
            a = amp / modes / (1.0 + 0.25 * math.hypot(kx, ky))
            ex = 2 * math.pi * kx * x + f
            ey = 2 * math.pi * ky * y
            out[b] += a * (torch.cos(ey)[:, None] * torch.sin(ex)[None, :] +
                           torch.sin(ey)[:, None] * torch.cos(ex)[None, :])
    return out


def _state(c, seed, dev):
    """The state [nbatch][ncomp][ny][nx] and the domain of case c."""
    rng = np.random.default_rng([seed, c["nx"], c["ny"], c["nbatch"]])
    nb, ny, nx, data = c["nbatch"], c["ny"], c["nx"], c["data"]
    a, b = _DOMAIN[data]
    x = (torch.arange(nx, dtype=torch.float64, device=dev) + 0.5) / nx
    y = (torch.arange(ny, dtype=torch.float64, device=dev) + 0.5) / ny
    X, Y = x[None, None, :], y[None, :, None]

    def col(v):
        return torch.as_tensor(v, dtype=torch.float64, device=dev).reshape(nb, 1, 1)

    if c["system"] != "euler":
        if c["system"] == "buckley_leverett":  # saturations in [0, 1] with a jump
            s = 0.5 + 0.4 * _waves(rng, nb, x, y, 1.0, kmax=4)
            s = torch.where(X < col(rng.uniform(0.3, 0.7, nb)), s, 0.3 * s)
            return s.reshape(nb, 1, 1, nx).contiguous(), (a, b)
        u = 0.5 + torch.sin(2 * math.pi * (X + col(rng.uniform(0, 1, nb))))
        return (u + _waves(rng, nb, x, y, 0.5)).reshape(nb, 1, 1, nx).contiguous(), (a, b)

    one = torch.ones(nb, ny, nx, dtype=torch.float64, device=dev)
    if data == "shock_density":
        xx = a + (b - a) * X
        left = (xx < -4.0 + col(rng.uniform(0.0, 2.0, nb))) & (one > 0)
        rho = torch.where(left, 3.857143 * one, 1.0 + 0.2 * torch.sin(5.0 * xx) * one)
        u, v, p = torch.where(left, 2.629369 * one, 0 * one), 0 * one, torch.where(left, 10.33333 * one, one)
    elif data == "smooth":
        rho, u, v, p = 1.5 * one, 0.2 * one, -0.1 * one, 1.5 * one
    else:  # tube: two states; quadrant: four
        n = 2 if data == "tube" else 4
        st = np.stack([rng.uniform(0.1, 2.0 if n == 2 else 1.5, (n, nb)), rng.uniform(-1, 1, (n, nb)),
                       rng.uniform(-1, 1, (n, nb)), rng.uniform(0.1, 2.0 if n == 2 else 1.5, (n, nb))])
        at = col(rng.uniform(0.3, 0.7, nb)) if n == 2 else 0.5
        right, up = X > at, Y > (0.5 if n == 4 else 2.0)

        def pick(q):
            lo = torch.where(right, col(st[q, 0]), col(st[q, 1]))
            if n == 2:
                return lo * one
            return torch.where(up, torch.where(right, col(st[q, 2]), col(st[q, 3])), lo) * one

        rho, u, v, p = (pick(q) for q in range(4))
    w = 0.2 if data != "shock_density" else 0.05
    rho = rho * (1 + _waves(rng, nb, x, y, w))
    p = p * (1 + _waves(rng, nb, x, y, w))
    u = u + _waves(rng, nb, x, y, w)
    if c["ndim"] == 1:
        U = torch.stack([rho, rho * u, p / (GAMMA - 1) + 0.5 * rho * u * u], dim=1)
    else:
        v = v + _waves(rng, nb, x, y, w)
        U = torch.stack([rho, rho * u, rho * v, p / (GAMMA - 1) + 0.5 * rho * (u * u + v * v)], dim=1)
    return U.contiguous(), (a, b)


def _desc(c, dom):
    return weno.make_desc(system=c["system"], ndim=c["ndim"], nbatch=c["nbatch"], nx=c["nx"],
                          ny=c["ny"], x0=dom[0], x1=dom[1], y0=dom[0], y1=dom[1], bc_x=c["bc"],
                          bc_y=c["bc"], gamma=GAMMA, cfl=0.5, eps=EPS, mu0=MU0, ai=c["ai"],
                          precision=c["precision"], alpha_mode=c["alpha"], order=c["order"])


def _served(c):
    """The solves of a serving case: alternating 1D tubes and 2D quadrants of sizes up to
    (nx, ny x ny), alternating precision, each over about c["t"] steps."""
    for k in range(c["nbatch"]):
        prec = "fp32_recon" if (k // 2) % 2 else "fp64"
        if k % 2 == 0:
            n = max(64, c["nx"] >> (k // 2)) + k
            yield _case(nx=n, precision=prec, data="tube"), c["t"] * 0.5 * (10.0 / n) / 3.0
        else:
            n = max(32, c["ny"] - 32 * (k // 2))
            yield (_case(ndim=2, nx=n, ny=n, precision=prec, data="quadrant"),
                   c["t"] * 0.5 / n / 6.0)


def prepare(case, seed):
    c, dev = case, "cuda"
    if c["call"] == "serve":
        reqs = []
        for k, (q, t) in enumerate(_served(c)):
            U, dom = _state(q, seed + 100 * k, dev)
            reqs.append((_desc(q, dom), U.cpu().numpy(), t))
        return {"call": "serve", "reqs": reqs,
                "engine": serve.Engine(256 << 20, max_slots=64, max_tiles=1 << 16)}
    U, dom = _state(c, seed, dev)
    d = _desc(c, dom)
    s = {"call": c["call"], "d": d, "U0": U, "U": torch.empty_like(U), "t": c["t"]}
    if c["call"] == "step_host":
        s["U0"] = U.cpu().pin_memory()
        s["U"] = torch.empty_like(s["U0"]).pin_memory()
        s["ws"] = weno.workspace(d, host=True)
    else:
        s["ws"] = weno.workspace(d)
    return s


def run(s):
    call = s["call"]
    if call == "rhs":
        return weno.rhs(s["d"], s["U0"], out=s["U"], ws=s["ws"])
    if call == "serve":
        e, out = s["engine"], {}
        slots = [e.admit(d, U, t) for d, U, t in s["reqs"]]
        left = set(slots)
        while left:
            e.run(4)
            for slot in e.poll()[0]:
                if slot in left:
                    left.discard(slot)
                    U, t, n, _ = e.retire(slot)
                    out["solve%d" % slots.index(slot)] = {"U": U, "t": t, "steps": n}
        return out
    s["U"].copy_(s["U0"])
    if call == "step":
        weno.step(s["d"], s["U"], ws=s["ws"], sync=False)
        return s["U"]
    if call == "step_host":
        dt = weno.step_host(s["d"], s["U"], ws=s["ws"])
        return {"U": s["U"], "dt": np.array(dt)}
    t, n = weno.solve(s["d"], s["U"], s["t"], ws=s["ws"])
    return {"U": s["U"], "t": np.array(t), "steps": np.array(n)}


def _stage_work(c):
    """Operations of one right-hand side, from the steps of the method."""
    r = c["order"] // 2
    recon = (r + 1) * (r * r + 5 * r + 6) + 10 * r  # indicators, candidates, weights; tau, mu
    cells = c["nbatch"] * c["nx"] * c["ny"]
    if c["system"] != "euler":
        return cells * (2 * recon + 8 * r)
    m = 3 if c["ndim"] == 1 else 4
    face = 2 * m * recon + 2 * r * 2 * m * m + 2 * m * m + 40  # fields, projections, back, Roe state
    return cells * (c["ndim"] * face + 20)


def work(case):
    c = case
    if c["call"] == "serve":
        total = {"bytes": 0.0, "flops": 0.0}
        for q, _ in _served(c):
            total["bytes"] += 16.0 * (3 if q["ndim"] == 1 else 4) * q["nx"] * q["ny"]
            total["flops"] += 3.0 * c["t"] * _stage_work(q)
        return total
    nc = 1 if c["system"] != "euler" else (3 if c["ndim"] == 1 else 4)
    stages = 1
    if c["call"] in ("step", "step_host"):
        stages = 3
    elif c["call"] == "solve":  # about this many CFL steps
        a, b = _DOMAIN[c["data"]]
        speed = {"advection": 1.0, "shock_density": 4.6}.get(
            c["system"] if c["system"] != "euler" else c["data"], 3.0)
        stages = 3 * max(1, math.ceil(c["t"] * speed * c["nx"] / (0.5 * (b - a))))
    return {"bytes": 16.0 * nc * c["nbatch"] * c["nx"] * c["ny"],
            "flops": float(stages * _stage_work(c))}


# ---------------------------------------------------------------------------
# The same results from plain 64-bit torch: arXiv 2603.26272 written out step by step
# (Section 3 and the Appendix tables), with explicit eigenvector matrices.
# ---------------------------------------------------------------------------
_D = {2: [1, 4, 1], 3: [1, 9, 9, 1], 4: [1, 16, 36, 16, 1], 5: [1, 25, 100, 100, 25, 1]}
_C = {2: [[-1, 3], [1, 1], [3, -1]],
      3: [[2, -7, 11], [-1, 5, 2], [2, 5, -1], [11, -7, 2]],
      4: [[-3, 13, -23, 25], [1, -5, 13, 3], [-1, 7, 7, -1], [3, 13, -5, 1], [25, -23, 13, -3]],
      5: [[12, -63, 137, -163, 137], [-3, 17, -43, 77, 12], [2, -13, 47, 27, -3],
          [-3, 27, 47, -13, 2], [12, 77, -43, 17, -3], [137, -163, 137, -63, 12]]}
_CDEN = {2: 2, 3: 6, 4: 12, 5: 60}
_BDEN = {2: 1, 3: 6, 4: 240, 5: 10080}


def _rev(B):
    return [row[::-1] for row in B[::-1]]


def _indicator_tables(r):
    if r == 2:
        return [[[1, -1], [-1, 1]]] * 3
    if r == 3:
        B0 = [[8, -19, 11], [-19, 50, -31], [11, -31, 20]]
        B1 = [[8, -13, 5], [-13, 26, -13], [5, -13, 8]]
        return [B0, B1, _rev(B0), [[44, -73, 29], [-73, 122, -49], [29, -49, 20]]]
    if r == 4:
        B0 = [[547, -1941, 2321, -927], [-1941, 7043, -8623, 3521], [2321, -8623, 11003, -4701],
              [-927, 3521, -4701, 2107]]
        B1 = [[267, -821, 801, -247], [-821, 2843, -2983, 961], [801, -2983, 3443, -1261],
              [-247, 961, -1261, 547]]
        return [B0, B1, _rev(B1), _rev(B0),
                [[7107, -16901, 13521, -3727], [-16901, 40643, -32863, 9121],
                 [13521, -32863, 26843, -7501], [-3727, 9121, -7501, 2107]]]
    B0 = [[45316, -208501, 364863, -288007, 86329], [-208501, 965926, -1704396, 1358458, -411487],
          [364863, -1704396, 3042786, -2462076, 758823], [-288007, 1358458, -2462076, 2041126, -649501],
          [86329, -411487, 758823, -649501, 215836]]
    B1 = [[13816, -60871, 99213, -70237, 18079], [-60871, 277126, -464976, 337018, -88297],
          [99213, -464976, 812586, -611976, 165153], [-70237, 337018, -611976, 485446, -140251],
          [18079, -88297, 165153, -140251, 45316]]
    B2 = [[13816, -51001, 67923, -38947, 8209], [-51001, 209926, -299076, 179098, -38947],
          [67923, -299076, 462306, -299076, 67923], [-38947, 179098, -299076, 209926, -51001],
          [8209, -38947, 67923, -51001, 13816]]
    Bd = [[942016, -2964751, 3597813, -2004757, 429679], [-2964751, 9449926, -11584896, 6499258, -1399537],
          [3597813, -11584896, 14319786, -8079576, 1746873],
          [-2004757, 6499258, -8079576, 4577926, -992851], [429679, -1399537, 1746873, -992851, 215836]]
    return [B0, B1, B2, _rev(B1), _rev(B0), Bd]


def _recon(v, r, ai):
    """The numerical flux at the face from the 2r stencil values v (eqs. (11)-(22), p = 1)."""
    B, f0 = _indicator_tables(r), v[r - 1]
    betas = []
    for k in range(r + 1):
        g = [v[k + m] - v[k] for m in range(r)]
        q = 0.0
        for i in range(1, r):
            row = 0.0
            for j in range(i, r):
                row = row + (1 if i == j else 2) * B[k][i][j] * g[j]
            q = q + g[i] * row
        betas.append((q / _BDEN[r]).clamp_min(0.0))
    betas[r] = sum(betas) / (r + 1)
    mean = sum(w - f0 for w in v) / (2 * r) + f0
    tau = sum((-1) ** (j + 1) * math.comb(2 * r - 1, j) * (v[j] - f0) for j in range(2 * r)) ** 2
    mu = sum((w - mean).abs() for w in v) / (2 * r) + MU0 if ai else torch.ones_like(f0)
    num, den = 0.0, 0.0
    for k in range(r + 1):
        a = _D[r][k] * (1.0 + tau / (betas[k] + EPS * mu * mu))
        cand = sum(_C[r][k][m] * (v[k + m] - f0) for m in range(r)) / _CDEN[r]
        num, den = num + a * cand, den + a
    return f0 + num / den


def _pad(U, r, bc, dim):
    if bc == "periodic":
        n = U.shape[dim]
        at = torch.arange(-r, n + r, device=U.device) % n
    else:
        at = torch.arange(-r, U.shape[dim] + r, device=U.device).clamp(0, U.shape[dim] - 1)
    return U.index_select(dim, at)


def _primitives(U):
    rho, E = U[:, 0], U[:, -1]
    vel = [U[:, 1 + k] / rho for k in range(U.shape[1] - 2)]
    q2 = sum(w * w for w in vel)
    p = (GAMMA - 1) * (E - 0.5 * rho * q2)
    return rho, vel, p, (E + p) / rho


def _alpha(U, k):
    rho, vel, p, _ = _primitives(U)
    cs, u = torch.sqrt(GAMMA * p / rho), vel[k]

    def top(w):
        return w.abs().flatten(1).amax(1).reshape(-1, 1, 1)
    return [top(u - cs)] + [top(u)] * len(vel) + [top(u + cs)]


def _bl_speed(u):
    D = u * u + 0.25 * (1 - u) ** 2
    return 0.5 * u * (1 - u) / (D * D)


def _bl_peak():
    def slope(u):
        D = u * u + 0.25 * (1 - u) ** 2
        return (1 - 2 * u) * D - 2 * u * (1 - u) * (2 * u - 0.5 * (1 - u))
    lo, hi = 0.0, 1.0
    for _ in range(100):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if slope(mid) > 0 else (lo, mid)
    return 0.5 * (lo + hi)


def _scalar_alpha(c, U):
    if c["system"] == "advection":
        return torch.ones(U.shape[0], 1, 1, dtype=U.dtype, device=U.device)
    lo, hi = U.flatten(1).amin(1), U.flatten(1).amax(1)
    if c["system"] == "burgers":
        s = torch.maximum(lo.abs(), hi.abs())
    else:
        peak = torch.full_like(lo, _bl_peak())
        s = torch.maximum(_bl_speed(lo).abs(), _bl_speed(hi).abs())
        s = torch.where((lo <= peak) & (peak <= hi), torch.maximum(s, _bl_speed(peak)), s)
    return s.reshape(-1, 1, 1)


def _faces(c, U, k):
    """Interface fluxes along direction k (0: x, 1: y): one more face than cells."""
    r, dim = c["order"] // 2, (2, 1)[k]  # dimension of a component [nb][ny][nx]
    P = _pad(U, r, c["bc"], dim + 1)
    n = U.shape[dim + 1] + 1

    def cell(q, j):
        return q.narrow(dim, j, n)

    if c["system"] != "euler":
        u = P[:, 0]
        f = {"advection": lambda w: w, "burgers": lambda w: 0.5 * w * w,
             "buckley_leverett": lambda w: w * w / (w * w + 0.25 * (1 - w) ** 2)}[c["system"]](u)
        A = _scalar_alpha(c, U)
        fp = [0.5 * (cell(f, j) + A * cell(u, j)) for j in range(2 * r)]
        fm = [0.5 * (cell(f, j) - A * cell(u, j)) for j in range(2 * r)]
        return (_recon(fp, r, c["ai"]) + _recon(fm[::-1], r, c["ai"])).unsqueeze(1)
    rho, vel, p, H = _primitives(P)
    F = torch.stack([P[:, 1 + k]] + [P[:, 1 + m] * vel[k] + (p if m == k else 0.0)
                                     for m in range(len(vel))] + [(P[:, -1] + p) * vel[k]], dim=1)
    sl, sr = (torch.sqrt(cell(rho, j)) for j in (r - 1, r))

    def roe(q):
        return (sl * cell(q, r - 1) + sr * cell(q, r)) / (sl + sr)
    W, h = [roe(q) for q in vel], roe(H)
    q2 = sum(w * w for w in W)
    cs = torch.sqrt((GAMMA - 1) * (h - 0.5 * q2))
    un, one, nil = W[k], torch.ones_like(h), torch.zeros_like(h)
    b1 = (GAMMA - 1) / (cs * cs)
    b2 = 0.5 * b1 * q2
    m = len(vel)

    def acoustic(s):  # the row of L and the column of R of u + s c
        L = [0.5 * (b2 - s * un / cs)] + [0.5 * (-b1 * w + (s / cs if i == k else 0.0))
                                          for i, w in enumerate(W)] + [0.5 * b1]
        R = [one] + [w + (s * cs if i == k else 0.0) for i, w in enumerate(W)] + [h + s * un * cs]
        return L, R
    fields = [acoustic(-1.0), ([1 - b2] + [b1 * w for w in W] + [-b1], [one] + W + [0.5 * q2])]
    if m == 2:
        t = 1 - k
        fields.append(([-W[t]] + [one if i == t else nil for i in range(2)] + [nil],
                       [nil] + [one if i == t else nil for i in range(2)] + [W[t]]))
    fields.append(acoustic(1.0))
    A = _alpha(U, k)
    if c["alpha"] == "single":
        A = [torch.stack(A).amax(0)] * len(A)
    out = [0.0] * (m + 2)
    for (L, R), al in zip(fields, A):
        w = [sum(L[q] * cell(P[:, q], j) for q in range(m + 2)) for j in range(2 * r)]
        g = [sum(L[q] * cell(F[:, q], j) for q in range(m + 2)) for j in range(2 * r)]
        fp = [0.5 * (g[j] + al * w[j]) for j in range(2 * r)]
        fm = [0.5 * (g[j] - al * w[j]) for j in range(2 * r)][::-1]
        e = _recon(fp, r, c["ai"]) + _recon(fm, r, c["ai"])
        out = [out[q] + R[q] * e for q in range(m + 2)]
    return torch.stack(out, dim=1)


def _rhs(c, U, d):
    total = 0.0
    for k in range(c["ndim"]):
        F = _faces(c, U, k)
        total = total - torch.diff(F, dim=(3, 2)[k]) / d[k]
    return total


def _dt(c, U, d):
    if c["system"] != "euler":
        return 0.5 * d[0] / _scalar_alpha(c, U).reshape(-1)
    s = [torch.maximum(a[0], a[-1]).reshape(-1) for a in (_alpha(U, k) for k in range(c["ndim"]))]
    return 0.5 * d[0] / s[0] if c["ndim"] == 1 else 0.5 / (s[0] / d[0] + s[1] / d[1])


def _rk3(c, U, dt, d):
    h = dt.reshape(-1, 1, 1, 1)
    U1 = U + h * _rhs(c, U, d)
    U2 = 0.75 * U + 0.25 * (U1 + h * _rhs(c, U1, d))
    return U / 3.0 + (2.0 / 3.0) * (U2 + h * _rhs(c, U2, d))


def _solve(c, U, t_end, d):
    t, n = 0.0, 0
    while t < t_end:
        dt = float(_dt(c, U, d))
        last = not dt < t_end - t
        dt = t_end - t if last else dt
        U = _rk3(c, U, torch.full((1,), dt, dtype=U.dtype, device=U.device), d)
        t, n = (t_end if last else t + dt), n + 1
    return U, t, n


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"

    def grid(c, dom):
        return [(dom[1] - dom[0]) / c["nx"], (dom[1] - dom[0]) / c["ny"]]
    if case["call"] == "serve":
        out = {}
        for k, (q, t_end) in enumerate(_served(case)):
            U, dom = _state(q, seed + 100 * k, dev)
            U, t, n = _solve(q, U, t_end, grid(q, dom))
            out["solve%d" % k] = {"U": U.cpu().numpy(), "t": t, "steps": n}
        return out
    U, dom = _state(case, seed, dev)
    d = grid(case, dom)
    if case["call"] == "rhs":
        return _rhs(case, U, d)
    if case["call"] == "solve":
        U, t, n = _solve(case, U, case["t"], d)
        return {"U": U, "t": np.array([t]), "steps": np.array([n])}
    dt = _dt(case, U, d)
    U = _rk3(case, U, dt, d)
    return U if case["call"] == "step" else {"U": U, "dt": dt.cpu().numpy()}
