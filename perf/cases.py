"""The work that users of this library have it do, as cases that a program can time and check.

Each case is one call, or a few calls that belong together, through the public entry points
(`paper_2501_12497_gb300.api` and `.autograd`): the projector pair, the motion operators and
their gradients, the reweighted regulariser, Solve-OF, and whole solves, from the 64x64x8
plain-method problem to the 1024x1024x64 one. Sizes are those of the benchmark workloads and
tests; `draw` gives other sizes, shapes and options of the same ranges.

The oracle values of `exact` are plain torch arithmetic in FP64 on the same inputs. Solve-OF and
the whole solves have none: what they return after a fixed number of iterations is defined by the
iteration itself, not by a formula.
"""
import math

import numpy as np
import torch

from paper_2501_12497_gb300 import api, autograd

H = 1.0  # pixel size


def listed():
    return [
        # the plain method's configuration: the smallest calls, where launches and latency count
        dict(name="tomo_64x64x8_f64", kind="tomo", nx=64, ny=64, nt=8, na=16, nb=64, fp64=True),
        # a gradient step of the joint problem by autograd (the differentiation form): H u and the flow
        # residual, then the gradients in u, s and s'
        dict(name="gradstep_256x256x32", kind="gradstep", nx=256, ny=256, nt=32, na=30, nb=363, fp64=False),
        # the same on odd frames with unequal numbers of views (rows that no vector load divides)
        dict(name="gradstep_181x149x9", kind="gradstep", nx=181, ny=149, nt=9, na=23, nb=257, ragged=True, fp64=False),
        # H and H^T of the large single problem, as each Golub-Kahan step applies them
        dict(name="tomo_1024x1024x64", kind="tomo", nx=1024, ny=1024, nt=64, na=90, nb=1448, fp64=False),
        # the flat fan beam of the fan workload
        dict(name="fan_256x256x32", kind="tomo", nx=256, ny=256, nt=32, na=30, nb=363, fp64=False, fan=2.0, db=1.6),
        # the image step's regulariser on the large problem
        dict(name="reg_1024x1024x64", kind="reg", nx=1024, ny=1024, nt=64, fp64=False),
        # derivative fields, linearised residual and reverse flow of the large problem
        dict(name="motion_1024x1024x64", kind="motion", nx=1024, ny=1024, nt=64, dr=1, fp64=False),
        # optical flow alone on the precision-form frames (31 pairs, 20 GKS iterations)
        dict(name="solve_of_256x256x32", kind="solve_of", nx=256, ny=256, nt=32, of_iters=20, fp64=False),
        # the first outer iterations of whole solves at the three sizes
        dict(name="solve_64x64x8_f64", kind="solve", nx=64, ny=64, nt=8, na=16, nb=64, outer=3, fp64=True),
        dict(name="solve_256x256x32", kind="solve", nx=256, ny=256, nt=32, na=30, nb=363, outer=2, fp64=False),
        dict(name="solve_1024x1024x64", kind="solve", nx=1024, ny=1024, nt=64, na=90, nb=1448, outer=2, fp64=False),
        # independent problems of uneven size solved together
        dict(name="batch_4_to_256", kind="batch", nx=256, ny=256, nt=8, na=10, nb=363, count=4, outer=2, fp64=False),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["tomo", "tomo", "gradstep", "gradstep", "reg", "motion", "solve_of", "solve", "batch"])
    solver = kind in ("solve_of", "solve", "batch")
    fp64 = rng.random() < 0.25
    top = 256 if solver or fp64 else 1024
    nx = _log(rng, 32, top)
    ny = nx if rng.random() < 0.4 or kind == "batch" else _log(rng, 32, top)
    if rng.random() < 0.5:  # the sizes in use are mostly multiples of 8
        nx, ny = nx - nx % 8, ny - ny % 8
    most = (1 << 20) if solver else (1 << 22) if fp64 else (1 << 25)
    nt = min(_log(rng, 2, 64), max(2, most // (nx * ny)))
    case = dict(kind=kind, nx=nx, ny=ny, nt=nt, fp64=fp64)
    if kind in ("tomo", "gradstep", "solve", "batch"):
        n = max(nx, ny)
        case.update(na=_log(rng, 8 if solver else 4, 45 if solver else 90), nb=math.ceil(math.sqrt(2) * n))
        if not solver:
            case["ragged"] = rng.random() < 0.3  # frames with unequal numbers of angles
            if rng.random() < 0.25:
                case.update(fan=2.0, db=1.6, nb=math.ceil(1.45 * n))
            else:
                case["db"] = rng.choice([1.0, 1.0, 1.0, 0.75, 1.5])
    if kind in ("gradstep", "reg"):
        case["round"] = rng.random() < 0.2  # M(s) by rounding and clipping
    if kind == "motion":
        case["dr"] = rng.choice([1, 1, 2, 3])
    if kind == "solve_of":
        case["of_iters"] = rng.choice([10, 20])
    if kind == "solve":
        case["outer"] = 2
        case["tv"] = rng.random() < 0.25  # D1-OF
        case["scale"] = 2 if nx % 2 == ny % 2 == 0 and rng.random() < 0.25 else 1  # Solve-OF on halved frames
    if kind == "batch":
        case.update(count=rng.choice([2, 3, 5]), outer=2, nt=min(nt, 12))
    return case


def members(case):
    """The problems of a batch: frames of 1, 3/4 and 1/2 of the largest, more of them and more views in turn."""
    out = []
    for i in range(case["count"]):
        n = max(24, case["nx"] * (4 - i % 3) // 4)
        out.append(dict(case, kind="solve", nx=n, ny=n, nt=case["nt"] + 2 * i, na=case["na"] + 5 * i, nb=math.ceil(math.sqrt(2) * n)))
    return out


# ------------------------------------------------------------------ inputs
def _dtype(case):
    return torch.float64 if case["fp64"] else torch.float32


def _geometry(case):
    """Angles per frame and their values: shifted intervals, as in the workloads."""
    nt, na = case["nt"], case["na"]
    n = np.array([na + (t % 3 if case.get("ragged") else 0) for t in range(nt)], np.int32)
    ang = np.concatenate([np.deg2rad(np.arange(k) * 180.0 / k + t * 180.0 / (k * nt)) for t, k in enumerate(n)])
    return n, ang


def _distances(case):
    n = max(case["nx"], case["ny"])
    return (case["fan"] * n, 0.5 * case["fan"] * n) if case.get("fan") else None


def _problem(case):
    prec = api.MOF_FP64 if case["fp64"] else api.MOF_FP32
    if "na" in case:
        n, ang = _geometry(case)
        p = api.mof_problem_create(case["nx"], case["ny"], case["nt"], case["nb"], n, ang, H, case.get("db", 1.0), prec,
                                   fan=_distances(case))
    else:
        nt = case["nt"]
        p = api.mof_problem_create(case["nx"], case["ny"], nt, 1, [1] * nt, [0.0] * nt, precision=prec)
    if case.get("round"):
        api.mof_set_warp(p, 1)
    return p


def _ellipses(case, seed):
    """Ellipses in rigid motion: rows (cx, cy, a, b, phi, rho, vx, vy, omega) in pixels."""
    rng = np.random.default_rng(seed)
    nx, ny, nt = case["nx"], case["ny"], case["nt"]
    out, scale = [], min(nx, ny) / 256.0
    for _ in range(8):
        a, b = rng.uniform(16, 60, 2) * scale
        sp, d = rng.uniform(0.3, 1.5), rng.uniform(0, 2 * np.pi)
        room = 0.25
        cx, cy = rng.uniform(-room, room) * nx, rng.uniform(-room, room) * ny
        vx, vy = sp * np.cos(d), sp * np.sin(d)
        lim = 0.12 * min(nx, ny)  # the whole path stays near its middle
        cut = min(1.0, lim / max(1e-9, 0.5 * nt * sp))
        out.append((cx - 0.5 * nt * vx * cut, cy - 0.5 * nt * vy * cut, a, b, rng.uniform(0, np.pi), rng.uniform(0.2, 1.0),
                    vx * cut, vy * cut, np.deg2rad(rng.uniform(-2, 2))))
    return out


def _at(e, t):
    return e[0] + t * e[6], e[1] + t * e[7], e[2], e[3], e[4] + t * e[8], e[5]


def _frames(case, seed):
    """The phantom's frames: ellipses with edges about a pixel wide on a smooth background."""
    nx, ny, nt, dev = case["nx"], case["ny"], case["nt"], "cuda"
    x = torch.arange(nx, device=dev, dtype=torch.float32) - 0.5 * (nx - 1)
    y = (torch.arange(ny, device=dev, dtype=torch.float32) - 0.5 * (ny - 1))[:, None]
    u = torch.empty(nt, ny, nx, device=dev, dtype=_dtype(case))
    es = _ellipses(case, seed)
    for t in range(nt):
        f = 0.05 * torch.cos(x * (3.0 / nx)) * torch.cos(y * (2.0 / ny))
        for e in es:
            cx, cy, a, b, phi, rho = _at(e, t)
            c, s = math.cos(phi), math.sin(phi)
            dx, dy = x - cx, y - cy
            r = torch.sqrt(((c * dx + s * dy) / a) ** 2 + ((c * dy - s * dx) / b) ** 2)
            f = f + rho * torch.clamp((1.0 - r) * (0.5 * (a + b)) + 0.5, 0.0, 1.0)
        u[t] = f
    return u.reshape(-1)


def _rays(case):
    """Per ray of every view: a point and a direction, FP64, each (views, nb)."""
    n, ang = _geometry(case)
    th = torch.tensor(ang, device="cuda")[:, None]
    sg = ((torch.arange(case["nb"], device="cuda", dtype=torch.float64) - 0.5 * (case["nb"] - 1)) * case.get("db", 1.0))[None, :]
    c, s = torch.cos(th), torch.sin(th)
    far = _distances(case)
    if far is None:
        px, py, vx, vy = sg * c, sg * s, -s + 0 * sg, c + 0 * sg
    else:
        rs, rd = far
        px, py = rs * s + 0 * sg, -rs * c + 0 * sg
        vx, vy = -rd * s + sg * c - px, rd * c + sg * s - py
    return n, px, py, vx, vy


def _data(case, seed):
    """Analytic line integrals of the phantom's ellipses along every ray, plus 1 % noise; its norm."""
    n, px, py, vx, vy = _rays(case)
    ln = torch.sqrt(vx * vx + vy * vy)
    nrx, nry = vy / ln, -vx / ln
    off = px * nrx + py * nry
    b = torch.zeros_like(off)
    a0 = 0
    for t, k in enumerate(n):
        sl = slice(a0, a0 + int(k))
        for e in _ellipses(case, seed):
            cx, cy, a, bb, phi, rho = _at(e, t)
            th = torch.atan2(nry[sl], nrx[sl])
            q0 = (a * torch.cos(th - phi)) ** 2 + (bb * torch.sin(th - phi)) ** 2
            q = q0 - (off[sl] - cx * nrx[sl] - cy * nry[sl]) ** 2
            b[sl] += rho * 2 * a * bb * torch.sqrt(torch.clamp(q, min=0)) / q0
        a0 += int(k)
    g = torch.Generator(device="cuda").manual_seed(seed + 17)
    e = torch.randn(b.shape, generator=g, device="cuda", dtype=torch.float64) * (0.01 * b.square().mean().sqrt())
    return (b + e).reshape(-1).to(_dtype(case)), float(e.norm())


def _velocity(case, seed):
    """A smooth field of up to about 3 px per frame with the small roughness of an estimated one,
    and a reverse field as the reverse flow leaves it: opposite, with holes of zero."""
    nx, ny, P, dev = case["nx"], case["ny"], case["nt"] - 1, "cuda"
    rng = np.random.default_rng(seed + 5)
    g = torch.Generator(device=dev).manual_seed(seed + 31)
    x = torch.arange(nx, device=dev, dtype=torch.float32) / nx
    y = (torch.arange(ny, device=dev, dtype=torch.float32) / ny)[:, None]
    s = torch.empty(P, 2, ny, nx, device=dev, dtype=_dtype(case))
    for p in range(P):
        for c in range(2):
            kx, ky = rng.uniform(1, 7, 2)
            f = rng.uniform(0.5, 2.6) * torch.sin(kx * x + rng.uniform(0, 6)) * torch.cos(ky * y + rng.uniform(0, 6))
            s[p, c] = f + 0.05 * torch.randn(ny, nx, generator=g, device=dev)
    keep = torch.rand(P, 1, ny, nx, generator=g, device=dev) > 0.03
    return s.reshape(-1), (-s * keep).reshape(-1).contiguous()


def _noise(case, seed, n):
    g = torch.Generator(device="cuda").manual_seed(seed + 57)
    return torch.randn(n, generator=g, device="cuda", dtype=_dtype(case))


def prepare(case, seed):
    k, dt = case["kind"], _dtype(case)
    if k == "batch":
        return dict(case=case, parts=[prepare(c, seed + 1000 * i) for i, c in enumerate(members(case))])
    p = _problem(case)
    st = dict(case=case, p=p)
    ns = case["nx"] * case["ny"]

    def new(n):
        return torch.empty(n, device="cuda", dtype=dt)

    if k == "solve":
        st["b"], delta = _data(case, seed)
        st["prm"] = api.mof_default_params(noise_norm=delta, temporal_tv=1 if case.get("tv") else 0, of_scale=case.get("scale", 1))
        st["u"], st["out"] = new(p.n), new(p.nv)
        return st
    st["u"] = _frames(case, seed)
    if k in ("tomo", "gradstep"):
        st["d"] = _data(case, seed)[0]
    if k in ("gradstep", "reg", "motion"):
        st["s"], st["sr"] = _velocity(case, seed)
    if k == "tomo":
        st["d"] += 0.1 * _noise(case, seed, p.m)  # a residual's signs on a sinogram's scale
        st["b"], st["g"] = new(p.m), new(p.n)
    elif k == "gradstep":
        st["dr"] = _noise(case, seed, 2 * (p.nt - 1) * ns)
    elif k == "reg":
        st["x"] = st["u"] + 0.05 * _noise(case, seed, p.n)
        st["y"] = new(p.n)
    elif k == "motion":
        for name in ("ux", "uy", "ut", "r"):
            st[name] = new((p.nt - 1) * ns)
        st["out"] = new(p.nv)
    else:
        st["out"] = new(p.nv)
        st["prm"] = api.mof_default_params(of_iters=case["of_iters"])
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    case = st["case"]
    k = case["kind"]
    if k == "batch":
        ps = st["parts"]
        api.mof_solve_batch([q["p"] for q in ps], [q["prm"] for q in ps], case["outer"], [q["b"] for q in ps],
                            [q["u"] for q in ps], [q["out"] for q in ps])
        return [{"u": q["u"], "s": q["out"]} for q in ps]
    p = st["p"]
    if k == "tomo":
        api.mof_apply_A(p, st["u"], st["b"])
        api.mof_apply_AT(p, st["d"], st["g"])
        return {"b": st["b"], "g": st["g"]}
    if k == "gradstep":  # H u with the gradient of ||H u - d||^2 / 2, and a cotangent of the flow residual
        u, s, sr = (st[n].detach().requires_grad_(True) for n in ("u", "s", "sr"))
        b, r = autograd.project(p, u), autograd.flow_residual(p, u, s, sr)
        torch.autograd.backward([b, r], [b.detach() - st["d"], st["dr"]])
        return {"b": b.detach(), "r": r.detach(), "gu": u.grad, "gs": s.grad, "gsr": sr.grad}
    if k == "reg":
        api.mof_apply_reg_normal(p, st["x"], st["u"], st["s"], st["sr"], 1e-3, st["y"])
        return st["y"]
    if k == "motion":
        api.mof_of_fields(p, st["u"], case["dr"], st["ux"], st["uy"], st["ut"])
        api.mof_apply_flow_lin(p, st["ux"], st["uy"], st["ut"], st["s"], st["r"])
        api.mof_reverse_flow(p, st["s"], st["out"])
        return {n: st[n] for n in ("ux", "uy", "ut", "r", "out")}
    if k == "solve_of":
        api.mof_solve_of(p, st["prm"], st["u"], st["out"])
        return st["out"]
    rep = api.mof_solve(p, st["prm"], case["outer"], st["b"], st["u"], st["out"])
    return {"u": st["u"], "s": st["out"], "resid": [r["resid"] for r in rep], "basis": [r["basis"] for r in rep]}


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    k, es = case["kind"], 8 if case["fp64"] else 4
    if k == "batch":
        parts = [work(c) for c in members(case)]
        return {m: sum(w[m] for w in parts) for m in ("bytes", "flops")}
    nx, ny, nt = case["nx"], case["ny"], case["nt"]
    ns, P = nx * ny, nt - 1
    n = ns * nt
    if "na" in case:
        m = int(_geometry(case)[0].sum()) * case["nb"]
        taps = 2.0 * m * max(nx, ny) * 0.7  # two taps per step over the part of a ray inside the frame
    if k == "tomo":
        return {"bytes": es * (2 * n + 2 * m), "flops": 2 * 2 * taps}
    if k == "gradstep":
        return {"bytes": es * (2 * n + 2 * m + 12 * P * ns), "flops": 2 * 2 * taps + 80.0 * P * ns}
    if k == "reg":
        return {"bytes": es * (3 * n + 4 * P * ns), "flops": 100.0 * n}
    if k == "motion":
        return {"bytes": es * (n + 8 * P * ns), "flops": 40.0 * P * ns}
    ell, its = 10, case.get("of_iters", 20)
    # Solve-OF: the Krylov basis of each pair read once per step, each vector written once
    of = es * 2 * P * (ns / case.get("scale", 1) ** 2) * (sum(range(ell)) + sum(ell + i for i in range(its)) + 2 * (ell + its))
    if k == "solve_of":
        return {"bytes": of, "flops": of}
    outer = case["outer"]
    img = es * (n + m) * (sum(range(ell)) + sum(ell + i for i in range(outer)) + 2 * (ell + outer))
    return {"bytes": outer * of + img, "flops": outer * of + 2 * taps * 2 * (ell + outer)}


# ------------------------------------------------------------------ the same in 64 bits
def _march(case, t0, nviews, px, py, vx, vy):
    """Joseph's rule for the rays of one frame's views: yields (rays, flat padded index of the first
    tap, weight of the second, length per step, frame stored by columns)."""
    nx, ny = case["nx"], case["ny"]
    sl = slice(t0, t0 + nviews)
    ln = torch.sqrt(vx[sl] ** 2 + vy[sl] ** 2)
    rows = vy[sl].abs() >= vx[sl].abs()
    for by_rows in (True, False):
        rays = torch.nonzero((rows == by_rows).reshape(-1)).reshape(-1)
        if not len(rays):
            continue
        ax, ay, bx, by, nf, nst = (px, py, vx, vy, nx, ny) if by_rows else (py, px, vy, vx, ny, nx)
        ax, ay, bx, by = (v[sl].reshape(-1)[rays][:, None] for v in (ax, ay, bx, by))
        j = (torch.arange(nst, device="cuda", dtype=torch.float64) - 0.5 * (nst - 1)) * H
        f = (ax + (j[None, :] - ay) * (bx / by)) / H + 0.5 * (nf - 1)
        fl = torch.floor(f)
        i0 = torch.clamp(fl, -2, nf).long() + 2
        yield rays, i0 + torch.arange(nst, device="cuda")[None, :] * (nf + 4), f - fl, (H * ln.reshape(-1)[rays][:, None] / by.abs()), not by_rows


def _pad(img):
    return torch.nn.functional.pad(img, (2, 2)).reshape(-1)


def _project64(case, u):
    n, px, py, vx, vy = _rays(case)
    u = u.double().reshape(case["nt"], case["ny"], case["nx"])
    out, a0 = torch.empty(px.shape, device="cuda", dtype=torch.float64), 0
    for t, k in enumerate(int(v) for v in n):
        for v0 in range(0, k, 16):
            kk = min(16, k - v0)
            o = torch.empty(kk * case["nb"], device="cuda", dtype=torch.float64)
            for rays, q, w, ln, turned in _march(case, a0 + v0, kk, px, py, vx, vy):
                f = _pad(u[t].t().contiguous() if turned else u[t])
                o[rays] = (((1 - w) * f[q] + w * f[q + 1]) * ln).sum(1)
            out[a0 + v0:a0 + v0 + kk] = o.reshape(kk, -1)
        a0 += k
    return out.reshape(-1)


def _backproject64(case, b):
    nx, ny, nb, db = case["nx"], case["ny"], case["nb"], case.get("db", 1.0)
    b = b.double().reshape(-1, nb)
    out, a0 = torch.zeros(case["nt"], ny, nx, device="cuda", dtype=torch.float64), 0
    n, ang = _geometry(case)
    if case.get("fan"):  # the transpose of the march itself
        _, px, py, vx, vy = _rays(case)
        for t, k in enumerate(int(v) for v in n):
            for rays, q, w, ln, turned in _march(case, a0, k, px, py, vx, vy):
                v = b[a0:a0 + k].reshape(-1)[rays][:, None] * ln
                nf, nst = (ny, nx) if turned else (nx, ny)
                acc = torch.zeros(nst * (nf + 4), device="cuda", dtype=torch.float64)
                acc.index_add_(0, q.reshape(-1), ((1 - w) * v).reshape(-1))
                acc.index_add_(0, (q + 1).reshape(-1), (w * v).reshape(-1))
                img = acc.reshape(nst, nf + 4)[:, 2:-2]
                out[t] += img.t() if turned else img
            a0 += k
        return out.reshape(-1)
    x = (torch.arange(nx, device="cuda", dtype=torch.float64) - 0.5 * (nx - 1)) * H
    y = ((torch.arange(ny, device="cuda", dtype=torch.float64) - 0.5 * (ny - 1)) * H)[:, None]
    for t, k in enumerate(int(v) for v in n):
        for a in range(a0, a0 + k):
            c, s = math.cos(ang[a]), math.sin(ang[a])
            mu = max(abs(c), abs(s))
            q = (x * c + y * s) / db + 0.5 * (nb - 1)
            fl, row = torch.floor(q), b[a]
            reach = math.ceil(mu * H / db)
            for m in range(1 - reach, reach + 1):
                kk = fl + m
                wt = (H / mu) * torch.clamp(1 - (q - kk).abs() * (db / (mu * H)), min=0) * ((kk >= 0) & (kk < nb))
                out[t] += wt * row[torch.clamp(kk, 0, nb - 1).long()]
        a0 += k
    return out.reshape(-1)


def _axis(case, v, horizontal):
    """First and second sample index and the weight of the second along one axis of M(s)."""
    n = case["nx"] if horizontal else case["ny"]
    i = torch.arange(n, device="cuda", dtype=torch.float64)
    v = v.double()
    pos = i if horizontal else i[:, None]
    if case.get("round"):
        i0 = torch.clamp(pos + torch.sign(v) * torch.floor(v.abs() + 0.5), 0, n - 1)
        return i0.long(), i0.long(), torch.zeros_like(i0)
    q = torch.clamp(pos + v, 0, n - 1)
    i0 = torch.floor(q)
    return i0.long(), torch.clamp(i0 + 1, max=n - 1).long(), q - i0


def _corners(case, v):
    """[(flat index, weight)] of M(v)'s four corners for one pair's field v (2, ny, nx)."""
    x0, x1, wx = _axis(case, v[0], True)
    y0, y1, wy = _axis(case, v[1], False)
    nx = case["nx"]
    return [(y0 * nx + x0, (1 - wx) * (1 - wy)), (y0 * nx + x1, wx * (1 - wy)), (y1 * nx + x0, (1 - wx) * wy), (y1 * nx + x1, wx * wy)]


def _warp(case, f, v):
    f = f.reshape(-1)
    return sum(w * f[q] for q, w in _corners(case, v))


def _warp_t(case, f, v):
    out = torch.zeros(f.numel(), device="cuda", dtype=torch.float64)
    for q, w in _corners(case, v):
        out.index_add_(0, q.reshape(-1), (w * f).reshape(-1))
    return out.reshape(f.shape)


def _slope(case, f, v):
    """Derivative of the bilinear sample along x and y, zero along an axis where it is clipped."""
    f = f.reshape(-1)
    a, b, c, d = (f[q] for q, _ in _corners(case, v))
    wx, wy = _axis(case, v[0], True)[2], _axis(case, v[1], False)[2]
    nx, ny = case["nx"], case["ny"]
    x = torch.arange(nx, device="cuda", dtype=torch.float64) + v[0].double()
    y = torch.arange(ny, device="cuda", dtype=torch.float64)[:, None] + v[1].double()
    mx, my = (x >= 0) & (x < nx - 1), (y >= 0) & (y < ny - 1)
    return mx * ((1 - wy) * (b - a) + wy * (d - c)), my * ((1 - wx) * (c - a) + wx * (d - b))


def _reflect(n, i):
    i = torch.remainder(i, 2 * n)
    return torch.where(i < n, i, 2 * n - 1 - i)


def exact(case, seed):
    k = case["kind"]
    if k in ("solve_of", "solve", "batch"):
        return None
    st = prepare(case, seed)
    nx, ny, nt = case["nx"], case["ny"], case["nt"]
    P = nt - 1
    u = st["u"].double().reshape(nt, ny, nx)
    if k == "tomo":
        return {"b": _project64(case, st["u"]), "g": _backproject64(case, st["d"])}
    s, sr = (st[n].reshape(P, 2, ny, nx) for n in ("s", "sr"))
    if k == "gradstep":
        b = _project64(case, st["u"])
        d = st["dr"].double().reshape(2, P, ny, nx)
        r, gu = torch.empty_like(d), _backproject64(case, b - st["d"].double()).reshape(nt, ny, nx)
        gs, gsr = torch.zeros(P, 2, ny, nx, device="cuda", dtype=torch.float64), torch.zeros(P, 2, ny, nx, device="cuda", dtype=torch.float64)
        for p in range(P):
            r[0, p] = u[p] - _warp(case, u[p + 1], s[p]).reshape(ny, nx)
            r[1, p] = u[p + 1] - _warp(case, u[p], sr[p]).reshape(ny, nx)
            gu[p] += d[0, p] - _warp_t(case, d[1, p], sr[p])
            gu[p + 1] += d[1, p] - _warp_t(case, d[0, p], s[p])
            if not case.get("round"):
                for out, f, v, c in ((gs, u[p + 1], s[p], d[0, p]), (gsr, u[p], sr[p], d[1, p])):
                    gx, gy = _slope(case, f, v)
                    out[p, 0], out[p, 1] = -c * gx, -c * gy
        return {"b": b, "r": r.reshape(-1), "gu": gu.reshape(-1), "gs": gs.reshape(-1), "gsr": gsr.reshape(-1)}
    if k == "reg":
        x, y = st["x"].double().reshape(nt, ny, nx), torch.zeros_like(u)

        def weigh(a, b):
            return a / torch.sqrt(b * b + 1e-6)

        for t in range(nt):
            g = weigh(x[t][:, 1:] - x[t][:, :-1], u[t][:, 1:] - u[t][:, :-1])
            y[t][:, 1:] += g
            y[t][:, :-1] -= g
            g = weigh(x[t][1:] - x[t][:-1], u[t][1:] - u[t][:-1])
            y[t][1:] += g
            y[t][:-1] -= g
        for p in range(P):
            for a, c, v in ((p, p + 1, s[p]), (p + 1, p, sr[p])):
                q = weigh(x[a] - _warp(case, x[c], v).reshape(ny, nx), u[a] - _warp(case, u[c], v).reshape(ny, nx))
                y[a] += q
                y[c] -= _warp_t(case, q, v)
        return y.reshape(-1)
    dr = case["dr"]
    ux, uy, ut = (torch.zeros(P, ny, nx, device="cuda", dtype=torch.float64) for _ in range(3))
    xs = [_reflect(nx, torch.arange(nx, device="cuda") + j) for j in range(-dr, dr + 1)]
    ys = [_reflect(ny, torch.arange(ny, device="cuda") + j) for j in range(-dr, dr + 1)]
    out = torch.zeros(P, 2, ny, nx, device="cuda", dtype=torch.float64)
    for p in range(P):
        a, box = u[p], 2 * dr + 1
        for j in range(box):
            ux[p] += (a[ys[j]][:, xs[-1]] - a[ys[j]][:, xs[0]]) / (2 * dr * box)
            uy[p] += (a[ys[-1]][:, xs[j]] - a[ys[0]][:, xs[j]]) / (2 * dr * box)
            for i in range(box):
                ut[p] += (u[p + 1] - a)[ys[j]][:, xs[i]] / (box * box)
        q = _axis_dest(case, s[p])
        cnt = torch.zeros(ny * nx, device="cuda", dtype=torch.float64).index_add_(0, q, torch.ones_like(q, dtype=torch.float64))
        for c in range(2):
            acc = torch.zeros(ny * nx, device="cuda", dtype=torch.float64).index_add_(0, q, -s[p, c].double().reshape(-1))
            out[p, c] = (acc / torch.clamp(cnt, min=1)).reshape(ny, nx)
    r = ux * s[:, 0].double() + uy * s[:, 1].double() + ut
    return {n: v.reshape(-1) for n, v in (("ux", ux), ("uy", uy), ("ut", ut), ("r", r), ("out", out))}


def _axis_dest(case, v):
    """Flat destination of every pixel under the reverse flow: x + s rounded half away from zero, clipped."""
    nx, ny = case["nx"], case["ny"]
    x = torch.arange(nx, device="cuda", dtype=torch.float64) + v[0].double()
    y = torch.arange(ny, device="cuda", dtype=torch.float64)[:, None] + v[1].double()
    x, y = (torch.sign(q) * torch.floor(q.abs() + 0.5) for q in (x, y))
    return (torch.clamp(y, 0, ny - 1) * nx + torch.clamp(x, 0, nx - 1)).long().reshape(-1)
