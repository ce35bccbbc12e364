"""The calls whose time this library is judged by, from the smallest to the largest a program makes.

Inputs follow the recipe of the repository's workloads: Burden loops (512 nodes each, length
log-uniform in 0.01-0.1, wavenumbers 1-5, at distance 0.3-0.5) and random-walk long strings
(step 1e-3 in a 0.2 cube), drawn here from the seed alone.  Cases that start from light-cone
samples get them from this file's own solve.

FP32-compensated results ("f32c") come back in float64 storage but carry single precision; a
program that asks for them keeps them as float32 (the default of HEALPix map files, and the type
of an optimiser's state), so those cases end with that conversion.
"""
import math

import numpy as np
import torch

import paper_1204_5041_gb300 as isw

NODES = 512          # nodes per loop
DEV = "cuda"
F = torch.float64


def listed():
    return [
        # one box of loops moved to the light cone: the smallest call, launch latency
        {"name": "solve_10k", "op": "solve", "loops": 20},
        # a quick look at one box: low-resolution map, both precisions
        {"name": "map32_n64_10k", "op": "map", "prec": "f32c", "nside": 64, "loops": 20, "nodes": 0, "pix": 0},
        {"name": "map64_n64_10k", "op": "map", "prec": "f64", "nside": 64, "loops": 20, "nodes": 0, "pix": 0},
        # the FP64 check of a map a level finer, loops and a long string, an odd sample count
        {"name": "map64_n128_25k", "op": "map", "prec": "f64", "nside": 128, "loops": 40, "nodes": 4607, "pix": 0},
        # the benchmark workload: 234 loops and 8 strings through the light-cone solve into one map
        {"name": "shells32_n512_200k", "op": "shells", "nside": 512, "loops": 234, "nodes": 80192, "shells": 1, "graph": False},
        # a stack of uneven shells at the next resolution, as one captured launch
        {"name": "shells32_n1024_100k", "op": "shells", "nside": 1024, "loops": 117, "nodes": 40096, "shells": 16, "graph": True},
        # scattered lines of sight of the paper's resolution (checks, small fields)
        {"name": "pixels32_n4096_100k", "op": "map", "prec": "f32c", "nside": 4096, "loops": 117, "nodes": 40096, "pix": 50001},
        # the gradient of a map's loss for every node of 98 loops
        {"name": "adjoint32_n256_50k", "op": "adjoint", "prec": "f32c", "nside": 256, "loops": 98, "ngrad": 6},
        # one training step on loop parameters: solve, FP64 map, and both adjoints
        {"name": "train64_n64_5k", "op": "train", "prec": "f64", "nside": 64, "loops": 10},
        # a 7.2 degree field at 512 x 512, full sky and flat sky
        {"name": "patch32_512_100k", "op": "patch", "prec": "f32c", "flat": False, "M": 512, "width": 0.1256, "loops": 117, "nodes": 40096},
        {"name": "flat32_1024_200k", "op": "patch", "prec": "f32c", "flat": True, "M": 1024, "width": 0.1256, "loops": 234, "nodes": 80192},
        # the power spectrum of the benchmark map
        {"name": "cl_n512_1536", "op": "cl", "nside": 512, "lmax": 1536},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["solve", "map", "map", "map", "shells", "shells", "adjoint", "train", "patch", "patch", "cl"])
    prec = rng.choice(["f32c", "f64"])
    if op == "solve":
        return {"op": op, "loops": _log(rng, 1, 400)}
    if op == "cl":
        nside = _log(rng, 8, 512)
        return {"op": op, "nside": nside, "lmax": rng.randint(nside, 3 * nside)}
    if op == "shells":
        nside, loops = _log(rng, 16, 700), _log(rng, 2, 234)
        return {"op": op, "nside": nside, "loops": loops, "nodes": _log(rng, 100, 80192), "shells": _log(rng, 1, 24),
                "graph": rng.random() < 0.5}
    if op == "patch":
        m = 60 if prec == "f64" else 1024
        return {"op": op, "prec": prec, "flat": rng.random() < 0.5, "M": _log(rng, 16, m), "width": rng.uniform(0.05, 0.3),
                "loops": _log(rng, 2, 234), "nodes": _log(rng, 100, 80192)}
    if op == "map" and rng.random() < 0.3:
        return {"op": op, "prec": prec, "nside": _log(rng, 64, 4096), "loops": _log(rng, 2, 117), "nodes": _log(rng, 100, 40096),
                "pix": _log(rng, 100, 10000 if prec == "f64" else 100000)}
    if op == "train":
        return {"op": op, "prec": prec, "nside": _log(rng, 8, 64), "loops": _log(rng, 1, 10)}
    hi = 100 if prec == "f64" else 256
    nside, loops = _log(rng, 8, hi), _log(rng, 1, 80 if prec == "f32c" else 40)
    if op == "adjoint":
        return {"op": op, "prec": prec, "nside": nside if prec == "f32c" else min(nside, 64), "loops": loops,
                "ngrad": rng.choice([6, 9, 10])}
    return {"op": op, "prec": prec, "nside": nside, "loops": loops, "nodes": _log(rng, 100, 9000), "pix": 0}


# ----------------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------------
def _units(rng, k):
    v = rng.standard_normal((k, 3))
    return v / np.linalg.norm(v, axis=1, keepdims=True)


def _loop_params(rng, centres):
    k = len(centres)
    q = rng.standard_normal((k, 4))
    w, x, y, z = (q / np.linalg.norm(q, axis=1, keepdims=True)).T
    R = [1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w), 2 * (x * y + z * w), 1 - 2 * (x * x + z * z),
         2 * (y * z - x * w), 2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)]
    P = np.empty((17, k))
    P[0:3], P[3:12] = centres.T, np.stack(R)
    P[12] = 10.0 ** rng.uniform(-2.0, -1.0, k)
    P[13], P[14] = rng.integers(1, 6, k), rng.integers(1, 6, k)
    P[15], P[16] = rng.uniform(0.0, math.pi, k), rng.uniform(0.0, 1.0, k) * P[12]
    return P


def _loop_nodes(P, first, count):
    ids = np.repeat(np.arange(first, first + count), NODES)
    nodes = np.zeros((10, ids.size))
    nodes[0], nodes[9] = ids, P[12, ids] / NODES
    nodes[1] = np.tile(np.arange(NODES), count) * nodes[9]
    return nodes


def _string_nodes(rng, count, centre, side):
    """Random walks of at most 10,024 nodes, velocities normal to the tangent, |Xdot|^2 + |X'|^2 = 1."""
    out = []
    while count > 0:
        k = min(count, 10024)
        k = k if count - k != 1 else k - 1
        count -= k
        if k < 2:
            break
        while True:
            X = centre + rng.uniform(-0.5, 0.5, 3) * side + np.vstack([np.zeros(3), np.cumsum(_units(rng, k - 1) * 1e-3, axis=0)])
            if np.min(np.linalg.norm(X, axis=1)) >= 0.02:
                break
        tang = np.gradient(X, axis=0)
        tang /= np.linalg.norm(tang, axis=1, keepdims=True) + 1e-300
        e1 = np.cross(tang, np.where(np.abs(tang[:, :1]) < 0.9, [[1.0, 0.0, 0.0]], [[0.0, 1.0, 0.0]]))
        e1 /= np.linalg.norm(e1, axis=1, keepdims=True)
        az, v = rng.uniform(0.0, 2 * math.pi, k), rng.uniform(0.3, 0.85, k)
        share = np.full(k, 1e-3)
        share[0] = share[-1] = 0.5e-3
        nodes = np.empty((10, k))
        nodes[0:3] = X.T
        nodes[3:6] = (v[:, None] * (np.cos(az)[:, None] * e1 + np.sin(az)[:, None] * np.cross(tang, e1))).T
        nodes[6:9], nodes[9] = (np.sqrt(1 - v * v)[:, None] * tang).T, share / np.sqrt(1 - v * v)
        out.append(nodes)
    return np.concatenate(out, axis=1) if out else np.zeros((10, 0))


def _network(case, seed):
    """(nodes, loop parameters, shell offsets, box times, modes): loops on the sky and strings in one
    cube, or the same counts dealt to cube shells between 0.05 and 0.95 of the horizon."""
    rng = np.random.default_rng(seed)
    loops, count, shells = case["loops"], case.get("nodes", 0), case.get("shells", 1)
    share = np.diff(np.round(np.concatenate([[0.0], np.cumsum(rng.dirichlet(np.ones(shells)))]) * loops).astype(int))
    nodes, params, t_box, mode, first = [], [], [], [], 0
    for k in range(shells):
        d = 0.4 if shells == 1 else rng.uniform(0.05, 0.95)
        centre, side = _units(rng, 1)[0] * d, 0.2 if shells == 1 else 0.1
        if share[k] > 0:
            c = _units(rng, share[k]) * rng.uniform(0.3, 0.5, share[k])[:, None] if shells == 1 \
                else centre + rng.uniform(-0.5, 0.5, (share[k], 3)) * side
            params.append(_loop_params(rng, c))
            nodes.append(_loop_nodes(np.concatenate(params, axis=1), first, share[k]))
            t_box.append(0.0)
            mode.append(isw.BURDEN)
            first += share[k]
        s = _string_nodes(rng, count // shells + (k < count % shells), centre, side)
        if s.shape[1]:
            nodes.append(s)
            t_box.append(1.0 - d)
            mode.append(isw.LINEAR)
    off = np.concatenate([[0], np.cumsum([a.shape[1] for a in nodes])]).astype(np.int64)
    return np.concatenate(nodes, axis=1), np.concatenate(params, axis=1), off, np.array(t_box), np.array(mode, dtype=np.int32)


def _gpu(a, dtype=F):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV, dtype)


def _worldsheet(P, sigma, t):
    """X, Xdot, X' [3, n] of the Burden loops P [17, n] at (sigma, t)."""
    L, m, n, psi, dt = P[12], P[13], P[14], P[15], t - P[16]
    a, b = 2 * math.pi * m * (sigma - dt) / L, 2 * math.pi * n * (sigma + dt) / L
    ra, rb = L / (2 * math.pi * m), L / (2 * math.pi * n)
    sa, ca, sb, cb, sp, cp = torch.sin(a), torch.cos(a), torch.sin(b), torch.cos(b), torch.sin(psi), torch.cos(psi)
    A, B = torch.stack([ra * sa, -ra * ca, 0 * sa]), torch.stack([rb * sb, -rb * cp * cb, -rb * sp * cb])
    Ap, Bp = torch.stack([ca, sa, 0 * sa]), torch.stack([cb, cp * sb, sp * sb])
    R = P[3:12].reshape(3, 3, -1)
    turn = lambda v: (R * v[None]).sum(1)  # noqa: E731
    return P[0:3] + turn(0.5 * (A + B)), turn(0.5 * (Bp - Ap)), turn(0.5 * (Ap + Bp))


def _solve_loops(nodes, P):
    """The crossing times |X(sigma, t)| = 1 - t: Newton steps kept inside a bracket."""
    Q = P[:, nodes[0].long()]
    d, half = Q[0:3].norm(dim=0), 0.5 * Q[12]
    lo, hi, t = 1 - d - half, 1 - d + half, 1 - d
    best, t_best = torch.full_like(t, math.inf), t
    for it in range(80):
        X, Xd, _ = _worldsheet(Q, nodes[1], t)
        r = X.norm(dim=0)
        f = r - (1 - t)
        t_best, best = torch.where(f.abs() < best, t, t_best), torch.minimum(best, f.abs())
        if it % 8 == 7 and bool((best <= 9e-16).all()):
            break
        lo, hi = torch.where(f < 0, t, lo), torch.where(f < 0, hi, t)
        tn = t - f / (1 + (X * Xd).sum(0) / r)
        t = torch.where((tn > lo) & (tn < hi) & (torch.tensor(it % 8 < 6, device=DEV)), tn, 0.5 * (lo + hi))
    return t_best


def _samples(nodes, P, off, t_box, mode, grad_tau=False):
    """Light-cone samples [10, n] and crossing times of every node, differentiable in nodes and P."""
    out, taus = [], []
    for k in range(len(t_box)):
        a = nodes[:, off[k]:off[k + 1]]
        if mode[k] == isw.BURDEN:
            with torch.no_grad():
                t = _solve_loops(a, P)
            Q = P[:, a[0].detach().long()]
            if grad_tau:   # one more Newton step carries the implicit derivative
                X, Xd, _ = _worldsheet(Q, a[1], t)
                fp = (1 + (X * Xd).sum(0) / X.norm(dim=0)).detach()
                t = t - (X.norm(dim=0) - (1 - t)) / fp
            X, Xd, Xp = _worldsheet(Q, a[1], t)
        else:
            T, X, Xd, Xp = 1 - t_box[k], a[0:3], a[3:6], a[6:9]
            R, v2 = X.norm(dim=0), (Xd * Xd).sum(0)
            c, bh = (R - T) * (R + T), (X * Xd).sum(0) + T
            D = -c / (bh + torch.sqrt(bh * bh + (1 - v2) * c))
            t, X = t_box[k] + D, X + Xd * D
        out.append(torch.cat([X, Xd, Xp, a[9:10]]))
        taus.append(t)
    return torch.cat(out, dim=1), torch.cat(taus)


def _frame(seed):
    q, _ = np.linalg.qr(np.random.default_rng(seed + 7).standard_normal((3, 3)))
    q = q.T * np.sign(np.linalg.det(q))
    return q


def prepare(case, seed):
    op = case["op"]
    if op == "cl":
        g = torch.Generator(DEV).manual_seed(seed)
        return {"case": case, "theta": torch.randn(12 * case["nside"] ** 2, dtype=F, device=DEV, generator=g)}
    nodes, P, off, t_box, mode = _network(case, seed)
    s = {"case": case, "nodes": _gpu(nodes), "P": _gpu(P), "off": off, "t_box": t_box, "mode": mode}
    if op in ("map", "adjoint", "patch"):
        s["samples"] = _samples(s["nodes"], s["P"], off, t_box, mode)[0].contiguous()
    g = torch.Generator(DEV).manual_seed(seed)
    if op == "solve":
        s["out"], s["tau"] = torch.empty_like(s["nodes"]), torch.empty(nodes.shape[1], dtype=F, device=DEV)
    if op in ("adjoint", "train"):
        s["g"] = torch.randn(12 * case["nside"] ** 2, dtype=F, device=DEV, generator=g)
    if op == "map":
        s["pix"] = None
        if case["pix"]:
            s["pix"] = torch.randint(12 * case["nside"] ** 2, (case["pix"],), device=DEV, generator=g)
    if op == "patch":
        s["frame"] = _frame(seed)
        if off[-1] > off[-2] and mode[-1] == isw.LINEAR:   # a field on the strings
            e3 = s["samples"][0:3, int(off[-2])].cpu().numpy()
            e3 = e3 / np.linalg.norm(e3)
            e1 = np.cross(e3, s["frame"][0])
            e1 = e1 / np.linalg.norm(e1)
            s["frame"] = np.stack([e1, np.cross(e3, e1), e3])
    return s


def run(s):
    case = s["case"]
    op, prec = case["op"], case.get("prec", "f32c")
    keep = (lambda x: x.float()) if prec == "f32c" else (lambda x: x)
    if op == "solve":
        isw.lightcone_intersect(isw.BURDEN, s["nodes"], s["P"], out=s["out"], tau=s["tau"])
        return s["out"], s["tau"]
    if op == "cl":
        return isw.isw_map_cl(case["nside"], s["theta"], case["lmax"])
    if op == "map":
        return keep(isw.isw_map(case["nside"], s["samples"], pix=s["pix"], prec=prec))
    if op == "shells":
        flags = isw.AUTOTUNE | (isw.GRAPH if case["graph"] else 0)
        return keep(isw.isw_map_batched(case["nside"], s["nodes"], s["off"], s["t_box"], s["mode"], s["P"], flags=flags))
    if op == "adjoint":
        return keep(isw.isw_map_adjoint(case["nside"], s["samples"], s["g"], prec=prec, ngrad=case["ngrad"]))
    if op == "patch":
        return keep(isw.isw_map_patch(s["frame"], case["M"], case["width"], s["samples"], prec=prec,
                                      approx=isw.FLATSKY if case["flat"] else isw.FULLSKY))
    nodes, P = s["nodes"].detach().requires_grad_(), s["P"].detach().requires_grad_()
    theta = isw.ISWLightconeMap.apply(nodes, P, case["nside"], isw.BURDEN, 0.0, None, None, 1.0, 1.0, prec)
    gn, gp = torch.autograd.grad(theta, (nodes, P), s["g"])
    return keep(theta.detach()), keep(gn), keep(gp)


def _counts(case):
    n = case["loops"] * NODES + case.get("nodes", 0)
    npix = case["M"] ** 2 if case["op"] == "patch" else case.get("pix") or 12 * case.get("nside", 0) ** 2
    return n, npix


def work(case):
    """Each input read once, each output written once.  The sum over samples and pixels has no
    operation count that every method must spend beyond one pair term (36 flops, 66 with its
    derivatives) for each sample and each pixel; the power spectrum has one Legendre value and its
    product with the ring's coefficient (8 flops) per ring pair, l and m."""
    op = case["op"]
    if op == "cl":
        n, l = case["nside"], case["lmax"]
        return {"bytes": 96.0 * n * n + 8.0 * l, "flops": 2.0 * n * 0.5 * (l + 1) * (l + 2) * 8}
    n, npix = _counts(case)
    size = 4 if case.get("prec", "f32c") == "f32c" else 8
    if op == "solve":
        return {"bytes": n * (80.0 + 88.0), "flops": 100.0 * n}
    if op == "adjoint":
        return {"bytes": 8.0 * npix + n * (80.0 + size * case["ngrad"]), "flops": 66.0 * (n + npix)}
    if op == "train":
        return {"bytes": npix * (8.0 + size) + n * (80.0 + 10 * size), "flops": (100 + 36 + 66.0) * (n + npix)}
    return {"bytes": 80.0 * n + size * npix + (8.0 * npix if case.get("pix") else 0.0), "flops": 36.0 * (n + npix)}


# ----------------------------------------------------------------------------------------
# the same in 64 bits, as plain torch gives it
# ----------------------------------------------------------------------------------------
def _sky(N, p):
    """RING pixel centres [3, len(p)]."""
    cap, npix = 2 * N * (N - 1), 12 * N * N
    q = torch.where(p < cap, p, npix - 1 - p)                    # cap pixels, counted from their pole
    i = ((1 + torch.sqrt((1 + 2 * q).double())) / 2).floor().long()
    i = torch.where(2 * i * (i - 1) > q, i - 1, i)
    i = torch.where(2 * (i + 1) * i <= q, i + 1, i).clamp(min=1)
    j = q - 2 * i * (i - 1)
    j = torch.where(p < cap, j, 4 * i - 1 - j)
    iv = i.double()
    ib, jb = (p - cap) // (4 * N) + N, (p - cap) % (4 * N)
    belt = (p >= cap) & (p < npix - cap)
    st = torch.where(belt, torch.sqrt(((2 * ib - N) * (7 * N - 2 * ib)).clamp(min=0).double()) / (3 * N),
                     iv * torch.sqrt((6 * N * N - i * i).clamp(min=0).double()) / (3 * N * N))
    z = torch.where(belt, (4 * N - 2 * ib).double() / (3 * N),
                    (3 * N * N - i * i).double() / (3 * N * N) * torch.where(p < cap, 1.0, -1.0).double())
    phi = torch.where(belt, (jb + 1).double() - torch.where((ib + N) % 2 == 1, 1.0, 0.5).double(), j.double() + 0.5) \
        * (0.5 * math.pi) / torch.where(belt, torch.full_like(iv, N), iv)
    return torch.stack([st * torch.cos(phi), st * torch.sin(phi), z])


def _terms(n, S):
    """theta [np] of directions n [3, np] summed over the samples S [10, ns] of one chunk."""
    X = S[0:3].norm(dim=0)
    xh, Xd, Xp = S[0:3] / X, S[3:6], S[6:9]
    c = -4 * torch.sqrt((Xp * Xp).sum(0) / (1 - (Xd * Xd).sum(0))) * S[9] / X
    Q = Pd = Qd = 0
    for k in range(3):
        d = n[k][:, None] - xh[k][None]
        Q, Pd, Qd = Q + d * d, Pd + Xd[k] * d, Qd + Xp[k] * d
    A, B = n.T @ Xp, 1 + n.T @ Xd
    return torch.where(Q > 0, (B * Pd - A * Qd) / (B * torch.where(Q > 0, Q, 1.0)), 0.0) @ c


def _theta(n, S, cells=1 << 22):
    ns = min(S.shape[1], 2048)
    step = max(1, cells // ns)
    out = torch.zeros(n.shape[1], dtype=F, device=DEV)
    for a in range(0, n.shape[1], step):
        for b in range(0, S.shape[1], ns):
            out[a:a + step] += _terms(n[:, a:a + step], S[:, b:b + ns])
    return out


def _grad(n, S, g, cells=1 << 22):
    ns = min(S.shape[1], 2048)
    step = max(1, cells // ns)
    out = torch.zeros_like(S)
    for b in range(0, S.shape[1], ns):
        for a in range(0, n.shape[1], step):
            with torch.enable_grad():
                s = S[:, b:b + ns].detach().requires_grad_()
                out[:, b:b + ns] += torch.autograd.grad(_terms(n[:, a:a + step], s), s, g[a:a + step])[0]
    return out


def _flat(case, s):
    fr, h = _gpu(s["frame"]), case["width"] / case["M"]
    S = s["samples"]
    r, Xd, Xp = fr @ S[0:3], fr @ S[3:6], fr @ S[6:9]
    w = -4 * torch.sqrt((Xp * Xp).sum(0) / (1 - (Xd * Xd).sum(0))) * S[9] / r[2]
    w = torch.where(r[2] > 0, w, 0.0) * (Xd[0:2] - Xp[2] * Xp[0:2] / (1 + Xd[2]))
    p = torch.where(r[2] > 0, r[0:2] / r[2], 1e3)
    x = (torch.arange(case["M"], device=DEV, dtype=F) + 0.5 - 0.5 * case["M"]) * h
    out = torch.empty((case["M"], case["M"]), dtype=F, device=DEV)
    for j in range(case["M"]):
        acc = torch.zeros_like(x)
        for b in range(0, p.shape[1], 4096):
            q, v = p[:, b:b + 4096], w[:, b:b + 4096]
            dx, dy = x[:, None] - q[0], x[j] - q[1]
            Q = dx * dx + dy * dy
            acc += torch.where(Q > 0, (v[0] * dx + v[1] * dy) / torch.where(Q > 0, Q, 1.0), 0.0).sum(1)
        out[j] = acc
    return out


def _cl(N, theta, lmax):
    """C_l from the definition: ring Fourier sums, then the normalised Legendre recursion in l for
    every m and ring pair, values kept with a separate power of two."""
    m = torch.arange(lmax + 1, device=DEV)
    mf = m.to(F)
    north, south, z, first = [], [], [], 0
    F_ring = []
    for i in range(1, 4 * N):
        k = min(i, N, 4 * N - i)
        t0 = 0.5 if k < N or (i + N) % 2 == 0 else 0.0
        row = torch.fft.fft(theta[first:first + 4 * k])
        F_ring.append(row[m % (4 * k)] * torch.exp(-2j * math.pi * (mf * (t0 / (4 * k)))))
        first += 4 * k
    Fr = torch.stack(F_ring)
    north, south = Fr[:2 * N], Fr[2 * N - 1:].flip(0)     # ring i with ring 4N - i; the equator alone
    south = torch.cat([south[:-1], torch.zeros_like(south[-1:])])
    ii = torch.arange(1, 2 * N + 1, device=DEV, dtype=F)
    z = torch.where(ii < N, 1 - ii * ii / (3.0 * N * N), (4.0 * N - 2 * ii) / (3.0 * N))
    even, odd = north + south, north - south
    logs = 0.5 * torch.log2(1 - z * z)                    # log2 sin(theta)
    k = torch.arange(1, lmax + 1, device=DEV, dtype=F)
    cm = torch.cat([torch.zeros(1, dtype=F, device=DEV), torch.cumsum(0.5 * torch.log2((2 * k - 1) / (2 * k)), 0)])
    e = cm + 0.5 * torch.log2((2.0 * mf + 1) / (4 * math.pi)) + mf * logs[:, None]     # log2 |lambda_mm|
    sc = torch.clamp(torch.ceil(e / 512), max=0)
    cur = torch.exp2(e - 512 * sc) * torch.where(m % 2 == 1, -1.0, 1.0).to(F)
    prev, start = torch.zeros_like(cur), cur
    cl = torch.zeros(lmax + 1, dtype=F, device=DEV)
    cur, zc = torch.zeros_like(cur), z[:, None]
    for l in range(lmax + 1):
        ok = mf < l
        a = torch.sqrt(torch.where(ok, (4.0 * l * l - 1) / (l * l - mf * mf), 0.0))
        b = torch.sqrt(torch.where(ok & (mf < l - 1), (2.0 * l + 1) * (l + mf - 1) * (l - mf - 1) / ((2.0 * l - 3) * (l * l - mf * mf)), 0.0))
        cur, prev = torch.where(m == l, start, zc * a * cur - b * prev), cur
        if l % 8 == 7:     # a value that grew past 1 takes its power back
            up = (sc < 0) & (cur.abs() > 1)
            f = torch.where(up, 2.0 ** -512, 1.0).to(F)
            cur, prev, sc = cur * f, prev * f, sc + up
        lam = torch.where(sc == 0, cur, 0.0)[:, :l + 1]
        par = (l + m[:l + 1]) % 2 == 0
        alm = (lam * torch.where(par, even[:, :l + 1], odd[:, :l + 1])).sum(0) * (4 * math.pi / (12.0 * N * N))
        p = alm.real ** 2 + alm.imag ** 2
        cl[l] = (2 * p.sum() - p[0]) / (2 * l + 1)
    return cl


def exact(case, seed):
    op = case["op"]
    if op == "cl":
        return _cl(case["nside"], prepare(case, seed)["theta"], case["lmax"]) if case["nside"] * case["lmax"] <= 8e5 else None
    n, npix = _counts(case)
    if n * npix > {"adjoint": 1.5e10, "train": 1.5e10}.get(op, 4e10):
        return None
    s = prepare(case, seed)
    with torch.no_grad():
        if op == "patch" and case["flat"]:
            return _flat(case, s)
        S, tau = (s["samples"], None) if "samples" in s else _samples(s["nodes"], s["P"], s["off"], s["t_box"], s["mode"])
        if op == "solve":
            return S, tau
        if op == "patch":
            x = (torch.arange(case["M"], device=DEV, dtype=F) + 0.5 - 0.5 * case["M"]) * (case["width"] / case["M"])
            eta, xi = torch.meshgrid(x, x, indexing="ij")
            v = _gpu(s["frame"]).T @ torch.stack([xi.reshape(-1), eta.reshape(-1), torch.ones(npix, dtype=F, device=DEV)])
            return _theta(v / v.norm(dim=0), S).reshape(case["M"], case["M"])
        pix = s.get("pix")
        v = _sky(case["nside"], torch.arange(npix, device=DEV) if pix is None else pix)
        if op in ("map", "shells"):
            return _theta(v, S)
        gs = _grad(v, S, s["g"])
        if op == "adjoint":
            return gs[:case["ngrad"]]
        theta = _theta(v, S)
    nodes, P = s["nodes"].detach().requires_grad_(), s["P"].detach().requires_grad_()
    S, _ = _samples(nodes, P, s["off"], s["t_box"], s["mode"], grad_tau=True)
    gn, gp = torch.autograd.grad(S, (nodes, P), gs)
    gp[13:15] = 0     # the wavenumbers are integers
    return theta, gn, gp
