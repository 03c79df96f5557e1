"""Performance cases of the gDC library: what its users run, through the public Python binding.

Two kinds of case.  The ``step_*`` cases are whole gDC steps (restore a state, advance one
step, read the frame back).  The others are single building blocks, each the call a program
makes that needs only that part: a mobility product, a mobility solve, a Brownian velocity,
the pair forces, the fluctuating-FCM operators.

Lengths are in blob radii, a = eta = kT = 1.  Bodies are placed by random sequential addition
(no two blobs of different bodies closer than 2a) at the volume fractions of the benchmark
configurations.  Results of the FP32-mixed mode and of the FP32 FCM grid, and trajectory
frames, are returned in float32: they carry single precision (the library states 2e-6 for
the FP32 products, 2e-5 for FCM), and that is how such a program keeps them.  Results of FP64
products, of FP64 forces and of FP64 Brownian velocities come back in float64.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

import paper_2106_00449_gb300 as gdc

SIGMA = 1.0 / math.sqrt(math.pi)      # FCM envelope width that gives the RPY self-mobility
R_T = 3.0                             # its truncation radius
SIGMA_OVER_H = 2.0631977647078092     # grid resolution of the 512^3 benchmark leg
REPULSION = dict(rep_A=4.0, rep_b=0.1)


# ---- the cases -----------------------------------------------------------------------------

def listed():
    return [
        # the smallest suspension of the benchmark configurations (4 icosahedral shells, 48
        # blobs), plain FP64: a step is a chain of small launches, so latency is what counts
        {"name": "step_icosahedra_4", "kind": "step", "shape": "icosahedra", "bodies": 4, "susp": 1,
         "precision": "fp64"},
        # 36 independent 15-blob boomerangs above a no-slip wall in FP64: the ensembles that the
        # paper's wall experiments step
        {"name": "step_boomerangs_36", "kind": "step", "shape": "wall", "bodies": 1, "susp": 36, "precision": "fp64"},
        # the headline: one FP32-mixed step of 2,520 mixed bodies (65,520 blobs)
        {"name": "step_mixed_65520", "kind": "step", "shape": "mixed", "bodies": 2520, "susp": 1, "precision": "mixed"},
        # mobility of 256 settling rods (2,560 blobs), FP32-mixed to 1e-6: a deterministic
        # sedimentation program calls this every step
        {"name": "solve_rods_256", "kind": "solve", "shape": "rods", "bodies": 256, "susp": 1, "precision": "mixed"},
        # the same solve for 48 uneven suspensions batched in one context, with a Brownian slip
        {"name": "solve_batch_48", "kind": "solve", "shape": "batch", "bodies": 0, "susp": 48, "precision": "mixed"},
        # Brownian velocities of 60 mixed bodies in FP64 (block-preconditioned Lanczos)
        {"name": "slip_mixed_60", "kind": "slip", "shape": "mixed", "bodies": 60, "susp": 1, "precision": "fp64"},
        # FP64 mobility product, an odd number of bodies (the default precision of the library)
        {"name": "product64_mixed_351", "kind": "product", "shape": "mixed", "bodies": 351, "susp": 1,
         "precision": "fp64"},
        # FP32 mobility product of a mid-size suspension, an odd number of bodies
        {"name": "product32_mixed_777", "kind": "product", "shape": "mixed", "bodies": 777, "susp": 1,
         "precision": "mixed"},
        # the allocation-free product of free blobs, from a program that owns all device memory
        {"name": "noalloc_3001", "kind": "noalloc", "blobs": 3001},
        # soft repulsion of 16,384 rods (327,680 blobs): the pair forces of the largest configuration
        {"name": "forces_rods_16384", "kind": "forces", "shape": "long_rods", "bodies": 16384, "susp": 1,
         "precision": "mixed", "potential": 0},
        # deterministic FCM mobility at the benchmark's size: 512^3 grid, 65,520 blobs
        {"name": "fcm_apply_512", "kind": "fcm_apply", "grid": 512, "blobs": 65520},
        # fluctuating FCM velocity (draw, solve, average) at 256^3
        {"name": "fcm_brownian_256", "kind": "fcm_brownian", "grid": 256, "blobs": 8190},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    k = rng.randrange(12)
    mode = rng.choice(["fp64", "mixed"])
    if k == 0:
        return {"kind": "step", "shape": "icosahedra", "bodies": _log_int(rng, 2, 40), "susp": 1, "precision": mode}
    if k == 1:
        return {"kind": "step", "shape": "wall", "bodies": rng.randint(1, 2), "susp": rng.randint(4, 64),
                "precision": mode}
    if k == 2:
        return {"kind": "step", "shape": "mixed", "bodies": _log_int(rng, 40, 2520), "susp": 1, "precision": "mixed"}
    if k == 3:
        return {"kind": "solve", "shape": "rods", "bodies": _log_int(rng, 16, 400), "susp": 1, "precision": mode}
    if k == 4:
        return {"kind": "solve", "shape": "batch", "bodies": 0, "susp": _log_int(rng, 6, 64), "precision": "mixed"}
    if k == 5:
        return {"kind": "slip", "shape": "mixed", "bodies": _log_int(rng, 6, 64), "susp": 1, "precision": "fp64"}
    if k == 6:
        return {"kind": "product", "shape": "mixed", "bodies": _log_int(rng, 12, 700), "susp": 1, "precision": "fp64"}
    if k == 7:
        return {"kind": "product", "shape": "mixed", "bodies": _log_int(rng, 12, 2520), "susp": 1,
                "precision": "mixed"}
    if k == 8:
        return {"kind": "noalloc", "blobs": _log_int(rng, 40, 16384)}
    if k == 9:
        wells = rng.randrange(3)
        return {"kind": "forces", "shape": "long_rods", "bodies": _log_int(rng, 60, 2500 if wells else 16384), "susp": 1,
                "precision": mode, "potential": wells}
    grid = rng.choice([64, 128, 256, 512])
    full = 65520 * (grid / 512.0) ** 3      # blobs at 10% volume fraction
    return {"kind": "fcm_apply" if k == 10 else "fcm_brownian", "grid": grid,
            "blobs": _log_int(rng, max(8, 0.05 * full), max(16, full))}


# ---- shapes and placement -------------------------------------------------------------------

def _icosahedron():
    phi = (1.0 + math.sqrt(5.0)) / 2.0
    v = []
    for s, t in itertools.product((-1.0, 1.0), repeat=2):
        v += [(0.0, s, t * phi), (s, t * phi, 0.0), (t * phi, 0.0, s)]
    v = np.array(v)
    return v / np.linalg.norm(v[0])


def _icosphere42():
    v = _icosahedron()
    d = np.linalg.norm(v[:, None] - v[None], axis=-1)
    edge = d[d > 0].min()
    mid = [(v[i] + v[j]) / np.linalg.norm(v[i] + v[j]) for i in range(12) for j in range(i + 1, 12)
           if d[i, j] < 1.001 * edge]
    p = np.vstack([v, np.array(mid)])
    d = np.linalg.norm(p[:, None] - p[None], axis=-1)
    return p * (2.0 / d[d > 0].min())


def _rod(n):
    return np.stack([np.zeros(n), np.zeros(n), 2.0 * np.arange(n)], axis=1)


def _boomerang(arm):
    k = np.arange(1.0, arm)
    o = np.zeros_like(k)
    return np.vstack([np.zeros((1, 3)), np.stack([k, o, o], 1), np.stack([o, k, o], 1)])


def _centred(t):
    return t - t.mean(axis=0)


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _rotations(q):
    """Rotation matrices of unit quaternions, scalar first (n, 3, 3)."""
    a, b, c, d = q.unbind(-1)
    return torch.stack([1 - 2 * (c * c + d * d), 2 * (b * c - d * a), 2 * (b * d + c * a),
                        2 * (b * c + d * a), 1 - 2 * (b * b + d * d), 2 * (c * d - b * a),
                        2 * (b * d - c * a), 2 * (c * d + b * a), 1 - 2 * (b * b + c * c)], -1).reshape(-1, 3, 3)


def _close_pairs(x, group, radius, y=None, group_y=None):
    """Index pairs (i of x, j of y) of points of one group that may lie within `radius`:
    those in the 27 cells of that size around i.  y = None: among x, the pair (i, i) included."""
    same = y is None
    y, group_y = (x, group) if same else (y, group_y)
    if len(x) == 0 or len(y) == 0:
        e = torch.zeros(0, dtype=torch.int64, device=x.device)
        return e, e
    cx, cy = (torch.floor(p / radius).to(torch.int64) for p in (x, y))
    low = torch.minimum(cx.amin(0), cy.amin(0)) - 1
    size = (torch.maximum(cx.amax(0), cy.amax(0)) - low + 2).tolist()

    def key(c, g):
        c = c - low
        return ((g * size[0] + c[:, 0]) * size[1] + c[:, 1]) * size[2] + c[:, 2]

    ky, order = torch.sort(key(cy, group_y))
    ii, jj = [], []
    # the three cells of a row are neighbours in the key: one range per row
    for dx, dy in itertools.product((-1, 0, 1), repeat=2):
        k0 = key(cx + torch.tensor([dx, dy, 0], device=x.device), group)
        lo, hi = torch.searchsorted(ky, k0 - 1), torch.searchsorted(ky, k0 + 1, right=True)
        n = hi - lo
        i = torch.repeat_interleave(torch.arange(len(x), device=x.device), n)
        first = torch.cumsum(n, 0) - n
        j = order[torch.arange(len(i), device=x.device) - first[i] + lo[i]]
        ii.append(i)
        jj.append(j)
    return torch.cat(ii), torch.cat(jj)


def _place(gen, templates, tmpl, susp, box):
    """Random sequential addition: uniform centres in each suspension's cube, uniform
    orientations, no two blobs of different bodies closer than 2a.  Proposals are made for
    many bodies at once and taken when no placed body and no earlier proposal is in the way."""
    dev = _device()
    n = len(tmpl)
    most = max(len(t) for t in templates)
    pad = torch.zeros(len(templates), most, 3, dtype=torch.float64, device=dev)
    live = torch.zeros(len(templates), most, dtype=torch.bool, device=dev)
    for k, t in enumerate(templates):
        pad[k, :len(t)] = torch.as_tensor(_centred(t))
        live[k, :len(t)] = True
    tmpl, susp, box = (torch.as_tensor(v, device=dev) for v in (tmpl, susp, box))
    Y = torch.zeros(n, 3, dtype=torch.float64, device=dev)
    q = torch.zeros(n, 4, dtype=torch.float64, device=dev)
    todo = torch.arange(n, device=dev)
    placed, placed_susp = torch.zeros(0, 3, dtype=torch.float64, device=dev), torch.zeros(0, dtype=torch.int64, device=dev)
    for _ in range(2000):
        if len(todo) == 0:
            break
        pool = todo.repeat(-(-min(max(len(todo), 2048), 8192) // len(todo)))[:8192]
        m = len(pool)
        y = torch.rand(m, 3, generator=gen, dtype=torch.float64, device=dev) * box[susp[pool]][:, None]
        p = torch.randn(m, 4, generator=gen, dtype=torch.float64, device=dev)
        p = p / p.norm(dim=1, keepdim=True)
        t = tmpl[pool]
        pts = y[:, None] + torch.einsum("nij,nbj->nbi", _rotations(p), pad[t])
        own = torch.arange(m, device=dev)[:, None].expand(m, most)[live[t]]
        x = pts[live[t]]
        g = susp[pool][own]
        bad = torch.zeros(m, dtype=torch.bool, device=dev)
        i, j = _close_pairs(x, g, 2.0, placed, placed_susp)
        hit = ((x[i] - placed[j]).square().sum(1) < 4.0) & (g[i] == placed_susp[j])
        bad[own[i[hit]]] = True
        keep = ~bad[own]
        x, own, g = x[keep], own[keep], g[keep]
        i, j = _close_pairs(x, g, 2.0)
        hit = ((x[i] - x[j]).square().sum(1) < 4.0) & (own[j] < own[i]) & (g[i] == g[j])
        bad[own[i[hit]]] = True
        first = torch.full((n,), m, dtype=torch.int64, device=dev)
        good = torch.nonzero(~bad)[:, 0]
        first.scatter_reduce_(0, pool[good], good, "amin")
        took = torch.nonzero(first < m)[:, 0]
        Y[took], q[took] = y[first[took]], p[first[took]]
        chosen = torch.zeros(m, dtype=torch.bool, device=dev)
        chosen[first[took]] = True
        placed = torch.cat([placed, x[chosen[own]]])
        placed_susp = torch.cat([placed_susp, g[chosen[own]]])
        todo = todo[first[todo] == m]
    else:
        raise RuntimeError("the bodies could not be placed")
    return Y.cpu().numpy(), q.cpu().numpy()


def _generator(seed, stream=0):
    g = torch.Generator(device=_device())
    g.manual_seed(1000003 * int(seed) + stream)
    return g


def _randn(seed, stream, *shape):
    return torch.randn(*shape, generator=_generator(seed, stream), dtype=torch.float64, device=_device())


def _suspension(case, seed):
    """Templates, body templates, suspension offsets, centres and quaternions of a case."""
    rng = np.random.default_rng([int(seed), 7])
    shape, bodies, S = case["shape"], case["bodies"], case["susp"]
    phi, box = None, None
    if shape == "icosahedra":           # 4 bodies in a 20a cube
        T, counts = [2.0 * _icosahedron()], [bodies]
        box = [20.0 * (bodies / 4.0) ** (1.0 / 3.0)]
    elif shape == "wall":
        T, counts = [_boomerang(8)], [bodies] * S
    elif shape == "rods":               # 256 rods in a 60a cube
        T, counts = [_rod(10)], [bodies]
        box = [60.0 * (bodies / 256.0) ** (1.0 / 3.0)]
    elif shape == "long_rods":
        T, counts, phi = [_rod(20)], [bodies], 0.08
    elif shape == "batch":              # uneven suspensions of 8 to 128 bodies
        T, phi = [2.0 * _icosahedron(), _rod(10), _icosphere42()], 0.05
        counts = np.random.default_rng([S, 11]).integers(8, 129, size=S).tolist()   # sizes belong to the case
    else:
        T, counts, phi = [_icosphere42(), _rod(15), _boomerang(11)], [bodies], 0.10
    n = int(sum(counts))
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    susp = np.repeat(np.arange(len(counts)), counts)
    tmpl = (np.arange(n) % len(T)).astype(np.int32)
    for s in range(len(counts)):        # each suspension has its own order of the shapes
        rng.shuffle(tmpl[off[s]:off[s + 1]])
    if shape == "wall":                 # every blob at least 0.5a above z = a; bodies of a suspension apart
        reach = np.linalg.norm(_centred(T[0]), axis=1).max()
        Y = np.stack([rng.uniform(0.0, 12.0, n), rng.uniform(0.0, 12.0, n), 1.5 + reach + rng.uniform(0.0, 2.0, n)], 1)
        Y[:, 0] += 32.0 * (np.arange(n) - off[susp])
        q = rng.standard_normal((n, 4))
        return T, tmpl, off, Y, q / np.linalg.norm(q, axis=1, keepdims=True)
    if box is None:
        nb = np.array([len(t) for t in T])[tmpl]
        vol = np.bincount(susp, weights=nb, minlength=len(counts)) * 4.0 / 3.0 * math.pi
        box = (vol / phi) ** (1.0 / 3.0)
    Y, q = _place(_generator(seed, 1), T, tmpl.astype(np.int64), susp.astype(np.int64), np.asarray(box, dtype=np.float64))
    return T, tmpl, off, Y, q


# ---- what a program has in hand -----------------------------------------------------------------

_PRECISION = {"fp64": gdc.FP64, "mixed": gdc.FP32_MIXED}


def _params(case, seed):
    shape = case["shape"]
    p = dict(precision=_PRECISION[case["precision"]], seed=int(seed) & 0x7FFFFFFF, gmres_tol=1e-6, lanczos_tol=1e-4,
             lanczos_max_iter=128, rfd_delta=1e-6 if case["precision"] == "fp64" else 1e-3)
    if shape == "icosahedra":
        p.update(dt=0.01)
    elif shape == "wall":               # Sec. 6.2: wall repulsion, weight, dt = 0.1 tau_D, tolerances 1e-4
        p.update(dt=0.6 * math.pi, gmres_tol=1e-4, wall=1, wall_V0=23.0, wall_b=0.5, body_weight=0.18)
    elif shape == "long_rods":          # kernels as they are by default: tuning takes seconds at this size
        p.update(dt=0.002, shear_rate=1.0, autotune=0, lanczos_max_iter=32, **REPULSION)
    else:
        p.update(dt=0.005, **REPULSION)
    if case.get("potential"):           # Sec. 6.3 soft sphere with the wells of Sec. 6.4
        p.update(rep_A=40.0, rep_b=0.5, potential=case["potential"], well_A=5.0, well_lambda=0.5)
    return p


def _blob_layout(T, tmpl):
    nb = np.array([len(t) for t in T])[tmpl]
    return nb, np.repeat(np.arange(len(tmpl)), nb)


def _blobs(T, tmpl, Y, q):
    """Blob positions (n, 3) in body order, and each blob's body."""
    dev = _device()
    nb, body = _blob_layout(T, tmpl)
    b = np.concatenate([_centred(T[t]) for t in tmpl])
    body = torch.as_tensor(body, device=dev)
    R = _rotations(torch.as_tensor(q, device=dev))
    r = torch.as_tensor(Y, device=dev)[body] + torch.einsum("nij,nj->ni", R[body], torch.as_tensor(b, device=dev))
    return r, body


def _loads(T, tmpl, Y, q, seed):
    """[force; torque] per body of random blob forces plus a weight along -z on every body."""
    r, body = _blobs(T, tmpl, Y, q)
    f = 0.3 * _randn(seed, 3, len(r), 3)
    arm = r - torch.as_tensor(Y, device=r.device)[body]
    FT = torch.zeros(len(tmpl), 6, dtype=torch.float64, device=r.device)
    FT.index_add_(0, body, torch.cat([f, torch.linalg.cross(arm, f)], 1))
    FT[:, 2] -= 1.0
    return FT


def _fcm_inputs(case, seed):
    L = case["grid"] * SIGMA / SIGMA_OVER_H
    r = torch.rand(case["blobs"], 3, generator=_generator(seed, 5), dtype=torch.float64, device=_device()) * L
    return L, r, _randn(seed, 6, case["blobs"], 3)


def _free_blobs(case, seed):
    n = case["blobs"]
    box = (n * 4.0 / 3.0 * math.pi / 0.05) ** (1.0 / 3.0)
    r = torch.rand(n, 3, generator=_generator(seed, 8), dtype=torch.float64, device=_device()) * box
    return r, _randn(seed, 9, n, 3)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "noalloc":
        r, lam = _free_blobs(case, seed)
        return {"case": case, "r": r, "lam": lam, "out": torch.empty_like(lam)}
    if kind.startswith("fcm"):
        L, r, lam = _fcm_inputs(case, seed)
        return {"case": case, "fcm": gdc.Fcm(case["grid"], L, SIGMA, R_T, max_blobs=case["blobs"]), "r": r, "lam": lam,
                "seed": int(seed) & 0x7FFFFFFF}
    T, tmpl, off, Y, q = _suspension(case, seed)
    st = {"case": case, "Y": Y, "q": q, "ctx": gdc.Context(gdc.Params(**_params(case, seed)), T, tmpl, off, Y, q)}
    n = st["ctx"].n_blobs
    if kind == "solve":
        st["FT"] = _loads(T, tmpl, Y, q, seed)
        # rods settle (no slip); the batch is driven by a Brownian slip as well
        st["slip"] = None if case["shape"] == "rods" else math.sqrt(2.0 / 0.005) * _randn(seed, 4, n, 3)
    elif kind in ("slip", "product"):
        st["x"] = _randn(seed, 4, n, 3)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    single = case.get("precision") == "mixed"
    if kind == "noalloc":
        return gdc.rpy_apply_noalloc(st["r"], st["lam"], out=st["out"]).float()
    if kind == "fcm_apply":
        return st["fcm"].apply(st["r"], st["lam"]).float()
    if kind == "fcm_brownian":
        return st["fcm"].brownian(st["r"], st["seed"], 0, 3, 1.0, 0.005).float()
    ctx = st["ctx"]
    if kind == "step":
        ctx.set_state(st["Y"], st["q"], 0)
        ctx.step(1)
        Y, q, _ = ctx.get_state()
        return {"Y": Y.astype(np.float32), "q": q.astype(np.float32)}
    if kind == "solve":
        V, lam, _ = ctx.mobility_solve(st["FT"], st["slip"], want_lambda=True)
        return {"V": V.float(), "lambda": lam.float()}
    if kind == "slip":
        return ctx.brownian_slip(st["x"])[0]
    out = ctx.forces() if kind == "forces" else ctx.rpy_apply(st["x"], ctx.params.precision)
    return out.float() if single else out


# ---- the work a pass cannot do without ----------------------------------------------------------

PAIR = 51.0         # flops of one unordered RPY pair with both sides' products
WALL_PAIR = 90.0    # flops of one ordered pair of the wall correction


def _counts(case):
    """(blobs per suspension, bodies) of a case, in expectation for a batch."""
    shape, S, b = case["shape"], case["susp"], case["bodies"]
    per = {"icosahedra": 12, "wall": 15, "rods": 10, "long_rods": 20, "mixed": 26}.get(shape)
    if shape == "batch":
        return 68 * 64.0 / 3.0, 68 * S
    return per * b, b * S


def work(case):
    kind = case["kind"]
    if kind == "noalloc":
        n = case["blobs"]
        return {"bytes": 72 * n, "flops": PAIR * n * (n - 1) / 2}
    if kind.startswith("fcm"):
        N, n = case["grid"], case["blobs"]
        box = 4.0 / 3.0 * math.pi * (R_T * SIGMA_OVER_H / SIGMA) ** 3     # grid points in an envelope
        fft = 2.5 * N ** 3 * 3.0 * math.log2(N)                           # one real 3-D transform
        if kind == "fcm_apply":
            return {"bytes": 72 * n, "flops": 6 * fft + 2 * 14.0 * box * n + 15.0 * N ** 3}
        return {"bytes": 48 * n, "flops": 9 * fft + 14.0 * box * n + 120.0 * N ** 3}
    ns, nb = _counts(case)
    n = ns * case["susp"]
    pairs = case["susp"] * ns * (ns - 1) / 2
    if case["shape"] == "wall":
        flops = PAIR * pairs + WALL_PAIR * case["susp"] * ns * ns
    else:
        flops = PAIR * pairs
    if kind == "forces":                # the pairs within the cutoff, 2a + 36 b or beyond the wells
        reach = 20.0 if case.get("potential") else 5.6
        near = min(ns, 0.08 * reach ** 3)
        return {"bytes": 56 * nb + 48 * nb, "flops": 10.0 * n * near + 20.0 * n}
    if kind == "product":
        return {"bytes": 56 * nb + 48 * n, "flops": flops}
    # Krylov products: a Brownian velocity takes about 6 + 2 log2(bodies) of them, a solve about
    # 8 + log2(bodies); a step takes three velocities and one solve
    lg = math.log2(max(2.0, nb / case["susp"]))
    slip, solve = 6 + 2 * lg, 8 + lg
    if case["shape"] == "wall":
        slip, solve = 1, 2
    if kind == "slip":
        return {"bytes": 56 * nb + 48 * n, "flops": flops * slip}
    if kind == "solve":
        return {"bytes": 56 * nb + 96 * nb + 48 * n, "flops": flops * solve}
    return {"bytes": 112 * nb, "flops": flops * (3 * slip + solve)}


# ---- the same results in 64 bits, by plain torch ------------------------------------------------

def _rpy_coefficients(r2):
    """A, B of the RPY tensor, u = (A lambda + B (d . lambda) d) / (8 pi eta), a = 1."""
    r = torch.sqrt(torch.clamp(r2, min=1e-300))
    far = r2 >= 4.0
    A = torch.where(far, 1.0 / r + 2.0 / (3.0 * r * r2.clamp(min=1.0)), 4.0 / 3.0 * (1.0 - 9.0 * r / 32.0))
    B = torch.where(far, (1.0 - 2.0 / r2.clamp(min=1.0)) / (r * r2.clamp(min=1.0)),
                    torch.where(r2 > 0, 1.0 / (8.0 * r), torch.zeros_like(r)))
    return A, B


def _rpy_product(r, lam):
    out = torch.empty_like(lam)
    rows = max(1, (1 << 25) // len(r))
    for i in range(0, len(r), rows):
        d = r[None] - r[i:i + rows, None]
        A, B = _rpy_coefficients(d.square().sum(-1))
        out[i:i + rows] = A @ lam + torch.einsum("ij,ijk->ik", B * (d * lam[None]).sum(-1), d)
    return out / (8.0 * math.pi)


def _rpy_matrix(r):
    d = r[None] - r[:, None]
    A, B = _rpy_coefficients(d.square().sum(-1))
    M = B[..., None, None] * d[..., :, None] * d[..., None, :]
    M += A[..., None, None] * torch.eye(3, dtype=r.dtype, device=r.device)
    return M.permute(0, 2, 1, 3).reshape(3 * len(r), 3 * len(r)) / (8.0 * math.pi)


def _rigid_matrix(r, Y, body, nb):
    """K: blob velocities of the bodies' [U; Omega], (3 n, 6 nb)."""
    n = len(r)
    arm = r - Y[body]
    K = torch.zeros(n, 3, nb, 6, dtype=r.dtype, device=r.device)
    i = torch.arange(n, device=r.device)
    for a in range(3):
        K[i, a, body, a] = 1.0
    for a, b, s in ((0, 4, 2), (1, 5, 0), (2, 3, 1)):        # Omega x arm
        K[i, a, body, b] = arm[:, s]
    for a, b, s in ((0, 5, 1), (1, 3, 2), (2, 4, 0)):
        K[i, a, body, b] = -arm[:, s]
    return K.reshape(3 * n, 6 * nb)


def _exact_solve(T, tmpl, off, Y, q, FT, slip):
    V, lam = [], []
    r, body = _blobs(T, tmpl, Y, q)
    Y = torch.as_tensor(Y, device=r.device)
    for s in range(len(off) - 1):
        lo, hi = int(off[s]), int(off[s + 1])
        sel = (body >= lo) & (body < hi)
        rs, bs = r[sel], body[sel] - lo
        C = torch.linalg.cholesky(_rpy_matrix(rs))
        K = _rigid_matrix(rs, Y[lo:hi], bs, hi - lo)
        v = torch.zeros_like(rs) if slip is None else slip[sel]
        X = torch.linalg.solve_triangular(C, torch.cat([K, v.reshape(-1, 1)], 1), upper=False)
        K1, v1 = X[:, :-1], X[:, -1]
        N = torch.linalg.pinv(K1.T @ K1, rtol=1e-10, hermitian=True)   # rods do not spin about their axis
        U = N @ (FT[lo:hi].reshape(-1) + K1.T @ v1)
        l = torch.linalg.solve_triangular(C.T, (K1 @ U - v1)[:, None], upper=True)[:, 0]
        V.append(U)
        lam.append(l)
    return {"V": torch.cat(V), "lambda": torch.cat(lam)}


def _exact_slip(T, tmpl, Y, q, W, dt):
    """sqrt(2 kT / dt) L (L^-1 M L^-T)^(1/2) W with L the bodies' Cholesky factors, each in its body's frame."""
    r, body = _blobs(T, tmpl, Y, q)
    M = _rpy_matrix(r)
    R = _rotations(torch.as_tensor(q, device=r.device))
    factor = [torch.linalg.cholesky(_rpy_matrix(torch.as_tensor(_centred(t), device=r.device))) for t in T]
    L = torch.block_diag(*[factor[t] for t in tmpl])
    turn = torch.block_diag(*[R[p] for p, t in enumerate(tmpl) for _ in range(len(T[t]))])
    A = torch.linalg.solve_triangular(L, turn.T @ M @ turn, upper=False)
    A = torch.linalg.solve_triangular(L, A.T.contiguous(), upper=False)
    w, Q = torch.linalg.eigh(0.5 * (A + A.T))
    root = Q @ (torch.sqrt(w.clamp(min=0.0)) * (Q.T @ W.reshape(-1)))
    return math.sqrt(2.0 / dt) * (turn @ (L @ root))


def _exact_forces(T, tmpl, Y, q, p):
    r, body = _blobs(T, tmpl, Y, q)
    f = torch.zeros_like(r)
    well = p.get("potential", 0)
    reach = max(2.0 + 36.0 * p["rep_b"], (3.5 if well == 2 else 3.0) + 6.0 * p["well_lambda"] if well else 0.0)
    order = torch.argsort(r[:, 0])
    zero = torch.zeros(len(r), dtype=torch.int64, device=r.device)
    for lo in range(0, len(r), 8192):       # slabs along x bound the number of candidate pairs
        mine = order[lo:lo + 8192]
        x0, x1 = r[mine[0], 0] - reach, r[mine[-1], 0] + reach
        others = torch.nonzero((r[:, 0] >= x0) & (r[:, 0] <= x1))[:, 0]
        i, j = _close_pairs(r[mine], zero[:len(mine)], reach, r[others], zero[:len(others)])
        i, j = mine[i], others[j]
        keep = body[i] != body[j]
        i, j = i[keep], j[keep]
        d = r[i] - r[j]
        dist = d.norm(dim=1)
        keep = (dist < reach) & (dist > 0)
        i, d, dist = i[keep], d[keep], dist[keep]
        x = dist.clamp(min=2.0)
        F = p["rep_A"] * torch.exp(-(x - 2.0) / p["rep_b"])
        if well:
            g = lambda c: 2.0 * p["well_A"] / p["well_lambda"] * ((x - c) / p["well_lambda"]) * torch.exp(   # noqa: E731
                -((x - c) / p["well_lambda"]) ** 2)
            F = F - g(3.0) + (g(3.5) if well == 2 else 0.0)
        f.index_add_(0, i, (F / dist)[:, None] * d)
    arm = r - torch.as_tensor(Y, device=r.device)[body]
    FT = torch.zeros(len(tmpl), 6, dtype=torch.float64, device=r.device)
    FT.index_add_(0, body, torch.cat([f, torch.linalg.cross(arm, f)], 1))
    return FT.reshape(-1)


def _envelopes(N, h, r):
    """Chunks (blobs, grid indices, weights) of the truncated Gaussian envelopes."""
    reach = int(math.ceil(R_T / h)) + 1
    o = torch.arange(-reach, reach + 1, device=r.device)
    step = max(1, (1 << 25) // len(o) ** 3)
    for lo in range(0, len(r), step):
        c = torch.floor(r[lo:lo + step] / h).to(torch.int64)[:, :, None] + o       # (b, 3, m)
        d2 = (c * h - r[lo:lo + step, :, None]).square()
        c = c % N
        dist = d2[:, 2, :, None, None] + d2[:, 1, None, :, None] + d2[:, 0, None, None, :]
        at = c[:, 0, None, None, :] + N * (c[:, 1, None, :, None] + N * c[:, 2, :, None, None])
        w = torch.where(dist <= R_T * R_T, torch.exp(-dist / (2.0 * SIGMA ** 2)), torch.zeros_like(dist))
        yield lo, at.flatten(1), w.flatten(1) * (2.0 * math.pi * SIGMA ** 2) ** -1.5


def _wave(N, L, device):
    k = torch.fft.fftfreq(N, 1.0 / N, dtype=torch.float64, device=device)
    keep = k.abs() != N // 2
    k = k * (2.0 * math.pi / L)
    half = N // 2 + 1
    kx, ky, kz = k[None, None, :half].abs(), k[None, :, None], k[:, None, None]
    keep = keep[None, None, :half] & keep[None, :, None] & keep[:, None, None]
    return kx, ky, kz, keep


def _stokes(fhat, N, L):
    """The velocity field (3, N^3) of a force density given by its real transforms."""
    kx, ky, kz, keep = _wave(N, L, fhat[0].device)
    k2 = kx * kx + ky * ky + kz * kz
    keep = keep & (k2 > 0)
    k2 = torch.where(k2 > 0, k2, torch.ones_like(k2))
    kf = (kx * fhat[0] + ky * fhat[1] + kz * fhat[2]) / k2
    out = []
    for f, k in zip(fhat, (kx, ky, kz)):
        u = torch.where(keep, (f - k * kf) / k2, torch.zeros_like(f))
        out.append(torch.fft.irfftn(u, s=(N, N, N)).reshape(-1))
    return out


def _averaged(N, L, r, u):
    h = L / N
    v = torch.empty_like(r)
    for lo, at, w in _envelopes(N, h, r):
        for c in range(3):
            v[lo:lo + len(at), c] = (u[c][at] * w).sum(1) * h ** 3
    return v


def _exact_fcm_apply(case, seed):
    L, r, lam = _fcm_inputs(case, seed)
    N = case["grid"]
    f = [torch.zeros(N ** 3, dtype=torch.float64, device=r.device) for _ in range(3)]
    for lo, at, w in _envelopes(N, L / N, r):
        for c in range(3):
            f[c].index_add_(0, at.reshape(-1), (w * lam[lo:lo + len(at), c, None]).reshape(-1))
    fhat = [torch.fft.rfftn(x.reshape(N, N, N)) for x in f]
    return _averaged(N, L, r, _stokes(fhat, N, L))


def _philox(j, owner, step, stream, seed):
    """Philox4x32-10 (Salmon et al. 2011) of the counters (j, owner, step, stream), as four words."""
    m = 0xFFFFFFFF

    def mul(a, x):                      # high and low words of a 32 x 32 bit product, in 64-bit integers
        lo, hi = a * (x & 0xFFFF), a * (x >> 16)
        s = lo + ((hi & 0xFFFF) << 16)
        return ((hi >> 16) + (s >> 32)) & m, s & m

    c = [j & m, torch.full_like(j, owner), torch.full_like(j, step), torch.full_like(j, stream)]
    k0, k1 = seed & m, seed >> 32 & m
    for rnd in range(10):
        if rnd:
            k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
    return c


def _exact_fcm_brownian(case, seed):
    L, r, _ = _fcm_inputs(case, seed)
    N = case["grid"]
    dv, dt = (L / N) ** 3, 0.005
    diag, cross = 2.0 * math.sqrt(1.0 / (dv * dt)), math.sqrt(2.0 / (dv * dt))
    kx, ky, kz, _ = _wave(N, L, r.device)
    k = (kx, ky, kz)
    fhat = [0.0, 0.0, 0.0]
    for pair in range(3):               # normals xx, yy | zz, xy | xz, yz of every point
        W = torch.empty(2, N ** 3, dtype=torch.float64, device=r.device)
        for lo in range(0, N ** 3, 1 << 24):
            g = torch.arange(lo, min(N ** 3, lo + (1 << 24)), dtype=torch.int64, device=r.device)
            x = _philox(3 * g + pair, 0, 3, 2, int(seed) & 0x7FFFFFFF)
            u = (x[0] >> 5).double() * 2.0 ** -27 + (x[1] >> 6).double() * 2.0 ** -53
            v = (x[2] >> 5).double() * 2.0 ** -27 + (x[3] >> 6).double() * 2.0 ** -53
            rad = torch.sqrt(-2.0 * torch.log1p(-u))
            W[0, lo:lo + len(g)] = rad * torch.cos(2.0 * math.pi * v)
            W[1, lo:lo + len(g)] = rad * torch.sin(2.0 * math.pi * v)
        for q, (a, b) in enumerate((((0, 0), (1, 1)), ((2, 2), (0, 1)), ((0, 2), (1, 2)))[pair]):
            w = torch.fft.rfftn(W[q].reshape(N, N, N)) * (1j * (diag if a == b else cross))
            fhat[a] = fhat[a] + k[b] * w
            if a != b:
                fhat[b] = fhat[b] + k[a] * w
        del W
    return _averaged(N, L, r, _stokes(fhat, N, L))


def exact(case, seed):
    kind = case["kind"]
    if kind == "noalloc":
        return _rpy_product(*_free_blobs(case, seed))
    if kind == "fcm_apply":
        return _exact_fcm_apply(case, seed)
    if kind == "fcm_brownian":
        return _exact_fcm_brownian(case, seed)
    if kind == "step":                  # a whole step ends its Krylov iterations by tolerances: no value of its own
        return None
    T, tmpl, off, Y, q = _suspension(case, seed)
    if kind == "forces":
        return _exact_forces(T, tmpl, Y, q, _params(case, seed))
    n = len(_blob_layout(T, tmpl)[1])
    if kind == "product":
        return _rpy_product(_blobs(T, tmpl, Y, q)[0], _randn(seed, 4, n, 3)).reshape(-1)
    if kind == "slip":
        return _exact_slip(T, tmpl, Y, q, _randn(seed, 4, n, 3), _params(case, seed)["dt"])
    slip = None if case["shape"] == "rods" else math.sqrt(2.0 / 0.005) * _randn(seed, 4, n, 3)
    return _exact_solve(T, tmpl, off, Y, q, _loads(T, tmpl, Y, q, seed), slip)
