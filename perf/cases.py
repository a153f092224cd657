"""Performance cases: what users of the library have it do, over the sizes they do it at.

A case is one call sequence through the Python binding (a level step, a
hierarchy root step, a batch of Riemann problems, a training step), on inputs
of the shapes and distributions of the repository's configurations.  listed()
names them; draw() gives others of the same ranges.  prepare() makes what a
program has in hand before the call, run() is one call sequence, work() counts
what it cannot do without, and exact() states the same results in plain 64-bit
torch, without the library.
"""
import functools
import math

import numpy as np
import torch

import paper_1307_2265_gb300 as ez
from paper_1307_2265_gb300 import hierarchy, synth

G = 5.0 / 3.0
NG = 3
CFL = 0.4
OPTIONS = ez.OPT_STEEPEN | ez.OPT_FLATTEN | ez.OPT_DIFFUSE


def listed():
    return [
        # the smallest configuration: one 32^3 periodic grid, white noise, in each
        # precision (the default is FP64); latency and launches decide it
        {"name": "grid32_fp64", "kind": "grid", "nx": 32, "ny": 32, "nz": 32, "precision": "fp64", "recipe": "white"},
        {"name": "grid32_fp32", "kind": "grid", "nx": 32, "ny": 32, "nz": 32, "precision": "fp32", "recipe": "white"},
        # one 256^3 periodic grid of Mach-3 turbulence, the FP32 path
        {"name": "grid256_fp32", "kind": "grid", "nx": 256, "ny": 256, "nz": 256, "precision": "fp32",
         "recipe": "turbulent"},
        # a ragged grid with external boundaries (tunnels, blast boxes): ghosts
        # filled each step, transverse ghost layers swept, FP64
        {"name": "walls_fp64", "kind": "grid", "nx": 100, "ny": 75, "nz": 50, "precision": "fp64", "recipe": "white",
         "walls": True},
        # the same in FP32 with the reconstruction options on, the way
        # strong-shock problems (double Mach reflection) are run
        {"name": "walls_options_fp32", "kind": "grid", "nx": 240, "ny": 125, "nz": 61, "precision": "fp32",
         "recipe": "blast", "walls": True, "options": True},
        # the headline: one AMR level of 4000 uneven patches, 1.9e8 cells, with
        # the plain and with the learned Newton guess
        {"name": "level4000_fp32", "kind": "level", "patches": 4000, "lo": 8, "hi": 64, "layout": 3,
         "precision": "fp32"},
        {"name": "level4000_learned", "kind": "level", "patches": 4000, "lo": 8, "hi": 64, "layout": 3,
         "precision": "fp32", "learned": True},
        # a level in FP64, the path that reproduces the reference bit for bit
        {"name": "level400_fp64", "kind": "level", "patches": 400, "lo": 8, "hi": 64, "layout": 7,
         "precision": "fp64"},
        # cold supersonic gas with the dual-energy field
        {"name": "level1000_dual", "kind": "level", "patches": 1000, "lo": 8, "hi": 64, "layout": 11,
         "precision": "fp32", "dual": True},
        # a subcycled root step of a static hierarchy: ghost interpolation,
        # sibling copies, flux registers and correction, projection
        {"name": "hierarchy64", "kind": "hierarchy", "root": 64, "levels": 3, "precision": "fp32"},
        # batched Riemann problems in FP64: the roots a training set is made of
        {"name": "riemann_fp64", "kind": "riemann", "n": 1 << 20, "precision": "fp64"},
        # one Adam step of the learned guess at its training batch
        {"name": "train16384", "kind": "train", "batch": 16384},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grid", "grid", "grid", "level", "level", "level", "hierarchy", "riemann", "train"])
    if kind == "grid":
        prec = rng.choice(["fp64", "fp32"])
        most = 6e6 if prec == "fp64" else 1.7e7
        while True:
            n = [_logint(rng, 8, 400) for _ in range(3)]
            if n[0] * n[1] * n[2] <= most:
                break
        c = {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "precision": prec,
             "recipe": rng.choice(["white", "turbulent", "blast"])}
        if rng.random() < 0.5:
            c["walls"] = True
        if rng.random() < 0.3:
            c["options"] = True
        return c
    if kind == "level":
        prec = rng.choice(["fp64", "fp32", "fp32"])
        lo, hi = rng.choice([(8, 64), (16, 32), (4, 40), (30, 64)])
        c = {"kind": kind, "patches": _logint(rng, 10, 250 if prec == "fp64" else 1500), "lo": lo, "hi": hi,
             "layout": rng.randrange(1 << 20), "precision": prec}
        more = rng.choice(["", "", "learned" if prec == "fp32" else "", "dual", "options"])
        if more:
            c[more] = True
        return c
    if kind == "hierarchy":
        root, levels = rng.choice([(32, 1), (48, 1), (64, 1), (64, 2), (96, 1), (96, 2), (128, 1), (128, 2), (64, 3)])
        c = {"kind": kind, "root": root, "levels": levels, "precision": "fp32", "layout": rng.randrange(1000)}
        if rng.random() < 0.3:
            c["learned"] = True
        return c
    if kind == "riemann":
        return {"kind": kind, "n": _logint(rng, 1000, 4_000_000), "precision": rng.choice(["fp64", "fp32"])}
    return {"kind": kind, "batch": _logint(rng, 100, 60_000)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _conserved(rho, v, p):
    E = p / (G - 1.0) + 0.5 * rho * ((v[0] * v[0] + v[1] * v[1]) + v[2] * v[2])
    return [rho, rho * v[0], rho * v[1], rho * v[2], E]


def _rand(seed, *shape):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    return torch.randn(*shape, dtype=torch.float64, device="cuda", generator=g)


def _grf(seed, nz, ny, nx):
    """Zero-mean, unit-variance periodic Gaussian random field, P(k) ~ k^-4."""
    f = torch.fft.rfftn(_rand(seed, nz, ny, nx))
    k = [torch.fft.fftfreq(s, dtype=torch.float64, device="cuda") * s for s in (nz, ny)]
    k.append(torch.arange(nx // 2 + 1, dtype=torch.float64, device="cuda"))
    k2 = k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + k[2][None, None, :] ** 2
    k2[0, 0, 0] = 1.0
    amp = 1.0 / k2
    amp[0, 0, 0] = 0.0
    f = torch.fft.irfftn(f * amp, s=(nz, ny, nx))
    return f / f.std()


def _grid_active(case, seed):
    """Active fields (z, y, x) of a single grid: white noise, turbulence or blasts."""
    s = (case["nz"], case["ny"], case["nx"])
    c0 = math.sqrt(G)
    if case["recipe"] == "white":
        r = _rand(seed, 4, *s)
        rho = torch.exp(0.5 * r[0] - 0.125)
        return _conserved(rho, r[1:] * (c0 / math.sqrt(3.0)), torch.ones_like(rho))
    if case["recipe"] == "turbulent":
        rho = torch.exp(_grf(4 * seed, *s) - 0.5)
        v = torch.stack([_grf(4 * seed + 1 + i, *s) for i in range(3)])
        v = v * (3.0 * c0 / torch.sqrt((v * v).sum(0).mean()))
        return _conserved(rho, v, torch.ones_like(rho))
    rho = torch.clamp(torch.exp(_grf(4 * seed, *s) - 0.5), 1e-2, 1e2)
    p = torch.full_like(rho, 1e-3)
    rng = np.random.default_rng(seed)
    ax = [torch.arange(m, dtype=torch.float64, device="cuda") for m in s]
    for _ in range(16):
        c, rad = rng.uniform(0, 1, 3) * s, rng.uniform(4, 24) * min(1.0, min(s) / 96.0)
        d = [torch.minimum((a - ci).abs(), m - (a - ci).abs()) ** 2 for a, ci, m in zip(ax, c, s)]
        inside = d[0][:, None, None] + d[1][None, :, None] + d[2][None, None, :] <= rad * rad
        p = torch.where(inside, torch.clamp(p, min=1e3 * 10.0 ** rng.uniform(-2, 0)), p)
    return _conserved(rho, torch.zeros(3, *s, dtype=torch.float64, device="cuda"), p)


def _sizes(case):
    rng = np.random.default_rng(case["layout"])
    return rng.integers(case["lo"], case["hi"] + 1, size=(case["patches"], 3))


def _level_active(case, seed, cells):
    """Active cells of all patches, packed: white noise at rms Mach 1 (Mach 10
    and cold with dual energy, where E - KE is a small part of E)."""
    r = _rand(seed, 4, cells)
    rho = torch.exp(0.5 * r[0] - 0.125)
    mach = 10.0 if case.get("dual") else 1.0
    return _conserved(rho, r[1:] * (mach * math.sqrt(G / 3.0)), torch.ones_like(rho))


def _packed_to_stored(sizes):
    """Storage index of every packed active cell (patch by patch, x fastest)."""
    n = torch.from_numpy(sizes).cuda()
    cells, vols = n.prod(1), (n + 2 * NG).prod(1)
    off = torch.cumsum(vols, 0) - vols
    first = torch.cumsum(cells, 0) - cells
    pid = torch.repeat_interleave(torch.arange(len(n), device="cuda"), cells)
    c = torch.arange(int(cells.sum()), device="cuda") - first[pid]
    nx, ny = n[:, 0][pid], n[:, 1][pid]
    z = c // (nx * ny)
    c -= z * (nx * ny)
    y = c // nx
    x = c - y * nx
    return off[pid] + (x + NG) + (nx + 2 * NG) * ((y + NG) + (ny + 2 * NG) * (z + NG)), off.cpu().numpy()


@functools.lru_cache(maxsize=1)
def _net_params():
    """Weights of a learned guess, trained on the host from a fixed seed (a
    program trains its network once and keeps it)."""
    rng = np.random.default_rng(5)
    s = [torch.from_numpy(a) for a in synth.riemann_states(rng, 1 << 15, 0.7, 1.0, 0.5, gamma=G)]
    o = _riemann64(*s)
    rl, ul, pl, rr, ur, pr = (a.numpy() for a in s)
    ic = np.sqrt(np.sqrt(rl * rr) / (G * np.sqrt(pl * pr)))
    a, b, d = 0.5 * np.log(rl / rr), 0.5 * np.log(pl / pr), 0.5 * (ul - ur) * ic
    x = np.stack([a, d, b, -a, -d, -b], 1)
    t = np.clip(np.log(o["pstar"].numpy() / np.sqrt(pl * pr)), -6.0, 6.0)
    W = [rng.normal(0, math.sqrt(2 / 6), (64, 6)), np.zeros(64), rng.normal(0, math.sqrt(2 / 64), (64, 64)),
         np.zeros(64), rng.normal(0, 1 / 8, 64), np.zeros(1)]
    m, v = [np.zeros_like(w) for w in W], [np.zeros_like(w) for w in W]
    sig = lambda q: 1.0 / (1.0 + np.exp(-q))  # noqa: E731
    for it in range(1, 801):
        i = rng.integers(0, len(t), 512)
        z1 = x[i] @ W[0].T + W[1]
        h1 = z1 * sig(z1)
        z2 = h1 @ W[2].T + W[3]
        h2 = z2 * sig(z2)
        e = (h2 @ W[4] + W[5][0] - t[i]) * (2.0 / 512)
        dz2 = e[:, None] * W[4] * (sig(z2) * (1 + z2 * (1 - sig(z2))))
        dz1 = (dz2 @ W[2]) * (sig(z1) * (1 + z1 * (1 - sig(z1))))
        for k, g in enumerate([dz1.T @ x[i], dz1.sum(0), dz2.T @ h1, dz2.sum(0), h2.T @ e, e.sum(keepdims=True)]):
            m[k] = 0.9 * m[k] + 0.1 * g
            v[k] = 0.999 * v[k] + 0.001 * g * g
            W[k] = W[k] - 4e-3 * (0.02 ** (it / 800)) * (m[k] / (1 - 0.9 ** it)) / (np.sqrt(v[k] / (1 - 0.999 ** it)) + 1e-8)
    return {k: np.round(w * 1024.0) / 1024.0 for k, w in zip(("W1", "b1", "W2", "b2", "w3", "b3"), W)}


def _net0(seed):
    """Fresh weights of the network a training run starts from."""
    rng = np.random.default_rng(seed)
    return {"W1": rng.normal(0, math.sqrt(2 / 6), (64, 6)), "b1": np.zeros(64),
            "W2": rng.normal(0, math.sqrt(2 / 64), (64, 64)), "b2": np.zeros(64),
            "w3": rng.normal(0, 1 / 8, 64), "b3": np.zeros(1)}


def _params(case, net):
    options = (OPTIONS if case.get("options") else 0) | (ez.OPT_DUAL if case.get("dual") else 0)
    return ez.Params(gamma=G, cfl=CFL, precision=ez.FP64 if case["precision"] == "fp64" else ez.FP32, options=options,
                     guess=ez.GUESS_MLP if net is not None else ez.GUESS_PLAIN,
                     mlp=net.blob if net is not None else None)


BC = (ez.BC_REFLECT, ez.BC_OUTFLOW, ez.BC_PERIODIC)


def _layout(case):
    R, k = case["root"], case["levels"]
    regions = [(R // 8, R - R // 8), (R // 4, R - R // 4), (3 * R // 8, R - 3 * R // 8)][:k]
    return synth.hierarchy_layout(R, regions, list(range(16, 33, 2)), seed=case.get("layout", 0))


def _riemann_inputs(case, seed):
    # left and right states as the training runs log them: lognormal density and
    # pressure, velocities of about Mach 1
    r = _rand(seed, 6, case["n"])
    rl, rr, pl, pr = (torch.exp(r[i]) for i in (0, 3, 2, 5))
    s = [rl, r[1] * torch.sqrt(G * pl / rl), pl, rr, r[4] * torch.sqrt(G * pr / rr), pr]
    dt = torch.float64 if case["precision"] == "fp64" else torch.float32
    return [a.to(dt).contiguous() for a in s]


def _train_inputs(case, seed):
    s = _riemann_inputs({"n": case["batch"], "precision": "fp64"}, seed)
    o = _riemann64(*s)
    rl, ul, pl, rr, ur, pr = s
    ic = torch.sqrt(torch.sqrt(rl * rr) / (G * torch.sqrt(pl * pr)))
    a, b, d = 0.5 * torch.log(rl / rr), 0.5 * torch.log(pl / pr), 0.5 * (ul - ur) * ic
    x = torch.stack([a, d, b, -a, -d, -b], 1)
    t = torch.log(torch.clamp(o["pstar"], min=1e-6) / torch.sqrt(pl * pr))
    return x.float(), t.float()


def prepare(case, seed):
    kind = case["kind"]
    net = ez.MLP(params=_net_params()) if case.get("learned") else None
    if kind == "grid":
        n = (case["nx"], case["ny"], case["nz"])
        st = [torch.nn.functional.pad(f, (NG,) * 6).reshape(-1) for f in _grid_active(case, seed)]
        table = ez.patch_table([n], [0], 1.0 / max(n), flags=0 if case.get("walls") else ez.PATCH_PERIODIC)
        return {"case": case, "batch": ez.PatchBatch(table, st), "params": _params(case, net), "step": 0}
    if kind == "level":
        sizes = _sizes(case)
        idx, off = _packed_to_stored(sizes)
        act = _level_active(case, seed, len(idx))
        if case.get("dual"):   # the gas energy: E - KE at uniform unit pressure
            act.append(torch.full_like(act[0], 1.0 / (G - 1.0)))
        total = int(np.prod(sizes + 2 * NG, axis=1).sum())
        st = []
        while act:
            f = torch.zeros(total, dtype=torch.float64, device="cuda")
            f[idx] = act.pop(0)
            st.append(f)
        table = ez.patch_table(sizes, off, 1.0 / 64, flags=ez.PATCH_PERIODIC)
        batch = ez.PatchBatch(table, st[:5], ge=st[5] if len(st) > 5 else None)
        return {"case": case, "batch": batch, "params": _params(case, net), "step": 0, "net": net}
    if kind == "hierarchy":
        lay = _layout(case)
        h = hierarchy.Hierarchy(lay, synth.hierarchy_fields(lay, config=1000 + seed, gamma=G), 1.0 / case["root"])
        return {"case": case, "h": h, "params": _params(case, net), "net": net,
                "out": [lev["batch"].U for lev in h.levels]}
    if kind == "riemann":
        return {"case": case, "s": _riemann_inputs(case, seed), "params": _params(case, None)}
    x, t = _train_inputs(case, seed)
    return {"case": case, "net": ez.MLP(params=_net0(seed)), "x": x, "t": t}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("grid", "level"):
        b, p = state["batch"], state["params"]
        if case.get("walls"):
            ez.timestep_cfl(b, p, out=b.dt_dev)
            ez.step_boundary(b, p, state["step"], b.dt_dev, BC)
        else:
            ez.evolve(b, p, 1, step0=state["step"])
        state["step"] += 1
        return {"dt": b.dt_dev, "U": b.U} if b.ge is None else {"dt": b.dt_dev, "U": b.U, "ge": b.ge}
    if kind == "hierarchy":
        dt = state["h"].root_step(state["params"])
        return {"dt": dt, "levels": state["out"]}
    if kind == "riemann":
        return ez.riemann_solve(*state["s"], state["params"])
    net = state["net"]
    loss = net.train_step(state["x"], state["t"], 2e-3)
    return {"loss": loss, "weights": net.master, "m": net.m, "v": net.v, "grad": net.grad}


def work(case):
    """Bytes: fields read and written once by the timestep and by each of the
    three sweeps.  Flops: per cell-sweep about 330 for the reconstruction,
    tracing, two Newton steps, flux and update, more with the options."""
    kind = case["kind"]
    if kind in ("grid", "level"):
        cells = case["nx"] * case["ny"] * case["nz"] if kind == "grid" else int(np.prod(_sizes(case), axis=1).sum())
        nf = 6 if case.get("dual") else 5
        return {"bytes": cells * (40 + 3 * 16 * nf),
                "flops": cells * (25 + 3 * (330 + 60 * bool(case.get("options")) + 40 * bool(case.get("dual"))))}
    if kind == "hierarchy":
        up = sum(int(np.prod(L["n"], axis=1).sum()) * 2 ** l for l, L in enumerate(_layout(case)))
        return {"bytes": up * 280, "flops": up * 1015}
    if kind == "riemann":
        return {"bytes": case["n"] * (11 * (8 if case["precision"] == "fp64" else 4) + 4), "flops": case["n"] * 180}
    return {"bytes": case["batch"] * 28 + 4673 * 28 + 19456, "flops": case["batch"] * 3 * 2 * (6 * 64 + 64 * 64 + 64)}


# ---------------------------------------------------------------------------
# the same results in plain 64-bit torch
# ---------------------------------------------------------------------------
def _riemann64(rl, ul, pl, rr, ur, pr, floor=1e-30):
    """Two-shock p* by Newton and the state at x/t = 0."""
    W_ = torch.where
    g2 = (G + 1.0) / (2.0 * G)
    CL, CR = torch.sqrt(G * pl * rl), torch.sqrt(G * pr * rr)
    ps = torch.clamp((CR * pl + CL * pr + CL * CR * (ul - ur)) / (CL + CR), min=floor)

    def side(q, p, C):
        W = C * torch.sqrt(torch.clamp(1.0 + g2 * (q / p - 1.0), min=1e-6))
        return W, 2.0 * W * W * W / (W * W + C * C)

    for _ in range(25):
        WL, ZL = side(ps, pl, CL)
        WR, ZR = side(ps, pr, CR)
        f = (ur + (ps - pr) / WR) - (ul - (ps - pl) / WL)
        ps = torch.clamp(ps - ZL * ZR * f / (ZL + ZR), min=floor)
    WL, ZL = side(ps, pl, CL)
    WR, ZR = side(ps, pr, CR)
    us = (ZL * (ul - (ps - pl) / WL) + ZR * (ur + (ps - pr) / WR)) / (ZL + ZR)
    left = us >= 0.0
    r, u, p, W = W_(left, rl, rr), W_(left, ul, ur), W_(left, pl, pr), W_(left, WL, WR)
    sg = W_(left, 1.0, -1.0)
    rs = torch.clamp(1.0 / (1.0 / r - (ps - p) / (W * W)), min=floor)
    rs = W_(rs > floor, rs, torch.full_like(rs, floor))
    head = u - sg * torch.sqrt(G * p / r)
    tail = us - sg * torch.sqrt(G * ps / rs)
    w_r = W_(sg * head >= 0.0, 0.0, W_(sg * tail <= 0.0, 1.0, -head / (tail - head)))
    w = W_(ps > p, W_(sg * (u - sg * W / r) >= 0.0, 0.0, 1.0), w_r)
    return {"pstar": ps, "ustar": us, "rho": r + w * (rs - r), "u": u + w * (us - u), "p": p + w * (ps - p)}


def _flux64(r, u, p, t1, t2):
    m = r * u
    return [m, m * u + p, m * t1, m * t2, u * (p / (G - 1.0) + 0.5 * r * (u * u + t1 * t1 + t2 * t2) + p)]


def _hll64(L, R):
    W_ = torch.where
    cl, cr = torch.sqrt(G * L[2] / L[0]), torch.sqrt(G * R[2] / R[0])
    SL, SR = torch.minimum(L[1] - cl, R[1] - cr), torch.maximum(L[1] + cl, R[1] + cr)
    FL, FR = _flux64(*L), _flux64(*R)
    cons = lambda s: [s[0], s[0] * s[1], s[0] * s[3], s[0] * s[4], s[2] / (G - 1.0) + 0.5 * s[0] * (s[1] ** 2 + s[3] ** 2 + s[4] ** 2)]  # noqa: E731
    return [W_(SL >= 0, a, W_(SR <= 0, b, (SR * a - SL * b + SL * SR * (y - x)) / (SR - SL)))
            for a, b, x, y in zip(FL, FR, cons(L), cons(R))]


def _sweep64(U, ge, d, dtdx, nb, inside, options):
    """One split sweep.  U: conserved fields; nb(q, k): the value k cells along
    the sweep; inside: cells that count as active along it (None: all)."""
    W_ = torch.where
    a1, a2 = (1 if d == 0 else 0), (1 if d == 2 else 2)
    rho, mn, m1, m2, E = U[0], U[1 + d], U[1 + a1], U[1 + a2], U[4]
    e = E - 0.5 * (mn * mn + m1 * m1 + m2 * m2) / rho
    if ge is not None:
        e = W_(e < 1e-3 * E, ge, e)
    q = [rho, mn / rho, torch.clamp((G - 1.0) * e, min=1e-30), m1 / rho, m2 / rho]
    if ge is not None:
        q.append(ge / rho)
    c = torch.sqrt(G * q[2] / q[0])

    def slope(x):
        l, r = x - nb(x, -1), nb(x, 1) - x
        m = torch.minimum(0.5 * (l + r).abs(), 2.0 * torch.minimum(l.abs(), r.abs()))
        return W_(l * r > 0, W_(l + r >= 0, m, -m), torch.zeros_like(x))

    if options:   # detectors of contact steepening and flattening
        rp, rm, pp, pm = nb(q[0], 1), nb(q[0], -1), nb(q[2], 1), nb(q[2], -1)
        Dm, Dp = q[0] - 2 * rm + nb(q[0], -2), nb(q[0], 2) - 2 * rp + q[0]
        dr, rmin, pmin = rp - rm, torch.minimum(rp, rm), torch.minimum(pp, pm)
        ok = (Dm * Dp < 0) & (dr.abs() >= 0.01 * rmin) & ((pp - pm).abs() / pmin <= 0.1 * G * (dr.abs() / rmin))
        eta = W_(ok, torch.clamp(20.0 * (-(Dp - Dm) / (6.0 * W_(ok, dr, torch.ones_like(dr))) - 0.05), 0.0, 1.0), 0.0)
        d1, d2 = pp - pm, nb(q[2], 2) - nb(q[2], -2)
        f = W_(d2 != 0, torch.clamp(10.0 * (d1 / W_(d2 != 0, d2, torch.ones_like(d2)) - 0.75), 0.0, 1.0), 1.0)
        flat = W_((nb(q[1], -1) - nb(q[1], 1) > 0) & (d1.abs() > 0.33 * pmin), f, torch.zeros_like(f))
    uc = q[1]
    lam = [uc - c, uc, uc + c]
    side = {1: [], -1: []}   # per variable: functions averaging over a domain of the zone's right / left edge
    for v, x in enumerate(q):
        dq = slope(x)
        face = 0.5 * (x + nb(x, 1)) - (nb(dq, 1) - dq) / 6.0
        ql, qr = nb(face, -1), face
        if options and v == 0:
            ql = W_(eta > 0, ql * (1 - eta) + (nb(x, -1) + 0.5 * nb(dq, -1)) * eta, ql)
            qr = W_(eta > 0, qr * (1 - eta) + (nb(x, 1) - 0.5 * nb(dq, 1)) * eta, qr)
        if options:
            ql, qr = flat * x + (1 - flat) * ql, flat * x + (1 - flat) * qr
        ext = (qr - x) * (x - ql) <= 0
        dd, q6 = qr - ql, 6.0 * (x - 0.5 * (ql + qr))
        nl = W_(ext, x, W_(dd * q6 > dd * dd, 3 * x - 2 * qr, ql))
        nr = W_(ext, x, W_(-(dd * dd) > dd * q6, 3 * x - 2 * ql, qr))
        dd, q6 = nr - nl, 6.0 * (x - 0.5 * (nl + nr))
        side[1].append((nr, dd, q6))
        side[-1].append((nl, dd, q6))
    st = {}
    for s in (1, -1):
        def avg(v, sig, s=s):
            edge, dd, q6 = side[s][v]
            return edge - s * 0.5 * sig * (dd - s * (1 - sig * (2.0 / 3.0)) * q6)

        sig = [torch.clamp(s * l * dtdx, min=0.0) for l in lam]
        ref, slow = (2, 0) if s > 0 else (0, 2)
        r, u, p = (avg(v, sig[ref]) for v in range(3))
        r, p = torch.clamp(r, min=1e-30), torch.clamp(p, min=1e-30)
        C = torch.sqrt(G * p * r)
        bs = W_(sig[slow] > 0, s * (0.5 / C) * ((u - avg(1, sig[slow])) - s * (p - avg(2, sig[slow])) / C), 0.0)
        b0 = W_(sig[1] > 0, (p - avg(2, sig[1])) / (C * C) + 1.0 / r - 1.0 / avg(0, sig[1]), 0.0)
        rho_e = 1.0 / (1.0 / r - (bs + b0))
        out = [W_(rho_e > 1e-30, rho_e, torch.full_like(r, 1e-30)), u - s * C * bs,
               torch.clamp(p + C * C * bs, min=1e-30), avg(3, sig[1]), avg(4, sig[1])]
        if ge is not None:
            out.append(avg(5, sig[1]))
        st[s] = out
    # interface j+1/2: left state from zone j, right state from zone j+1
    L, R = st[1], [nb(x, 1) for x in st[-1]]
    o = _riemann64(L[0], L[1], L[2], R[0], R[1], R[2])
    up = o["ustar"] >= 0
    F = _flux64(o["rho"], o["u"], o["p"], W_(up, L[3], R[3]), W_(up, L[4], R[4]))
    uf = o["u"]
    Fg = F[0] * W_(up, L[5], R[5]) if ge is not None else None
    zL, zR = q, [nb(x, 1) for x in q]
    if options:
        nu = 0.1 * torch.clamp(zL[1] - zR[1], min=0.0)
        cons = lambda s: [s[0], s[0] * s[1], s[0] * s[3], s[0] * s[4], s[2] / (G - 1.0) + 0.5 * s[0] * (s[1] ** 2 + s[3] ** 2 + s[4] ** 2)]  # noqa: E731
        F = [x + nu * (a - b) for x, a, b in zip(F, cons(zL), cons(zR))]
    bad = rho + dtdx * (nb(F[0], -1) - F[0]) <= 0
    if inside is not None:
        bad = bad & inside
    if bool(bad.any()):   # HLL re-flux of both faces of such cells
        face = bad | nb(bad, 1)
        H = _hll64(zL[:5], zR[:5])
        F = [W_(face, h, x) for h, x in zip(H, F)]
        if ge is not None:
            Fg = W_(face, F[0] * W_(F[0] >= 0, zL[5], zR[5]), Fg)
            uf = W_(face, 0.5 * (zL[1] + zR[1]), uf)
    new = [None] * 5
    for k, f in zip((0, 1 + d, 1 + a1, 1 + a2, 4), F):
        up_ = U[k] + dtdx * (nb(f, -1) - f)
        new[k] = up_ if inside is None else W_(inside, up_, U[k])
    if ge is None:
        return new, None
    g = ge + dtdx * (nb(Fg, -1) - Fg) - dtdx * q[2] * (uf - nb(uf, -1))
    en = new[4] - 0.5 * (new[1] ** 2 + new[2] ** 2 + new[3] ** 2) / new[0]
    emax = torch.maximum(new[4], torch.maximum(nb(new[4], -1), nb(new[4], 1)))
    return new, W_((new[0] > 0) & (en > 0.1 * emax), en, g)


def _rate64(U, dx):
    rho = U[0]
    c = torch.sqrt(G * torch.clamp((G - 1.0) * (U[4] - 0.5 * (U[1] ** 2 + U[2] ** 2 + U[3] ** 2) / rho), min=1e-30) / rho)
    return sum((c + (U[1 + i] / rho).abs()) / dx for i in range(3)).max()


def _fill64(f, axis_sign):
    """Reflecting x, outflow y, periodic z ghosts of a padded (z, y, x) block."""
    n = [s - 2 * NG for s in f.shape[::-1]]
    i = [torch.arange(-NG, m + NG, device=f.device) for m in n]
    x = i[0] % (2 * n[0])
    mirror = (i[0] < 0) | (i[0] >= n[0])
    x = torch.where(x < n[0], x, 2 * n[0] - 1 - x) + NG
    y, z = torch.clamp(i[1], 0, n[1] - 1) + NG, i[2] % n[2] + NG
    f = f[z][:, y][:, :, x]
    return torch.where(mirror[None, None, :], axis_sign * f, f)


def _exact_grid(case, seed):
    dx = 1.0 / max(case["nx"], case["ny"], case["nz"])
    act = _grid_active(case, seed)
    walls = bool(case.get("walls"))
    dt = CFL / _rate64(act, dx)
    U = act
    if walls:
        U = [_fill64(torch.nn.functional.pad(f, (NG,) * 6), -1.0 if k == 1 else 1.0) for k, f in enumerate(act)]
    stored = [torch.zeros(tuple(s + 2 * NG for s in act[0].shape), dtype=torch.float64, device="cuda")
              for _ in range(5)] if not walls else U
    for d in range(3):
        dim = 2 - d
        inside = None
        if walls:
            i = torch.arange(U[0].shape[dim], device="cuda")
            shape = [1, 1, 1]
            shape[dim] = -1
            inside = ((i >= NG) & (i < len(i) - NG)).reshape(shape)
        U, _ = _sweep64(U, None, d, dt / dx, lambda q, k, dim=dim: torch.roll(q, -k, dim), inside,
                        bool(case.get("options")))
        if walls:
            # a sweep covers the transverse ghosts of the axes still to come;
            # those of the axes done keep their values
            cov = torch.ones_like(U[0], dtype=torch.bool)
            for e in range(d):
                cov &= _active_along(U[0], 2 - e)
            U = [torch.where(cov, new, old) for new, old in zip(U, stored)]
            stored = U
    if not walls:
        U = [torch.nn.functional.pad(f, (NG,) * 6) for f in U]
    return {"dt": dt.reshape(1), "U": [f.reshape(-1) for f in U]}


def _active_along(f, dim):
    i = torch.arange(f.shape[dim], device=f.device)
    shape = [1, 1, 1]
    shape[dim] = -1
    return ((i >= NG) & (i < len(i) - NG)).reshape(shape)


def _exact_level(case, seed):
    sizes = _sizes(case)
    idx, off = _packed_to_stored(sizes)
    act = _level_active(case, seed, len(idx))
    dx = 1.0 / 64
    dt = CFL / _rate64(act, dx)
    dual = bool(case.get("dual"))
    out = [torch.zeros(int(np.prod(sizes + 2 * NG, axis=1).sum()), dtype=torch.float64, device="cuda")
           for _ in range(6 if dual else 5)]
    cells = np.prod(sizes, axis=1)
    ends = np.concatenate([[0], np.cumsum(cells)])
    a = 0
    while a < len(sizes):
        b = a + 1
        while b < len(sizes) and ends[b + 1] - ends[a] <= 12_000_000:
            b += 1
        lo, hi = int(ends[a]), int(ends[b])
        U = [f[lo:hi] for f in act]
        ge = torch.full_like(U[0], 1.0 / (G - 1.0)) if dual else None
        n = torch.from_numpy(sizes[a:b]).cuda()
        first = torch.from_numpy(ends[a:b] - lo).cuda()
        pid = torch.repeat_interleave(torch.arange(b - a, device="cuda"), n.prod(1))
        c = torch.arange(hi - lo, device="cuda")
        stride = [torch.ones_like(n[:, 0]), n[:, 0], n[:, 0] * n[:, 1]]
        for d in range(3):
            i, m, s = ((c - first[pid]) // stride[d][pid]) % n[:, d][pid], n[:, d][pid], stride[d][pid]
            at = {k: c + ((i + k) % m - i) * s for k in (-2, -1, 1, 2)}
            U, ge = _sweep64(U, ge, d, dt / dx, lambda q, k, at=at: q[at[k]], None, bool(case.get("options")))
        for f, u in zip(out, U + ([ge] if dual else [])):
            f[idx[lo:hi]] = u
        a = b
    r = {"dt": dt.reshape(1), "U": out[:5]}
    return {**r, "ge": out[5]} if dual else r


def _exact_train(case, seed):
    x, t = (a.double() for a in _train_inputs(case, seed))
    net = {k: torch.from_numpy(v).cuda().float().double() for k, v in _net0(seed).items()}
    w0 = torch.cat([v.reshape(-1) for v in net.values()])
    w = w0.clone().requires_grad_(True)
    at, p = 0, {}
    for k, v in net.items():
        p[k] = w[at:at + v.numel()].reshape(v.shape)
        at += v.numel()
    silu = torch.nn.functional.silu
    y = silu(silu(x @ p["W1"].T + p["b1"]) @ p["W2"].T + p["b2"]) @ p["w3"] + p["b3"]
    loss = ((y - t) ** 2).mean()
    g, = torch.autograd.grad(loss, w)
    return {"loss": loss.detach().reshape(1), "weights": w0 - 2e-3 * g / (g.abs() + 1e-8), "m": 0.1 * g,
            "v": 0.001 * g * g, "grad": g}


def exact(case, seed):
    kind = case["kind"]
    if kind == "grid":
        return _exact_grid(case, seed)
    if kind == "level":
        return _exact_level(case, seed)
    if kind == "riemann":
        o = _riemann64(*(a.double() for a in _riemann_inputs(case, seed)))
        return {**o, "iters": None}
    if kind == "train":
        return _exact_train(case, seed)
    return None   # a subcycled hierarchy step
