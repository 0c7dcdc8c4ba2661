"""Timed cases of the library: what its users have it do, from one chain to a 262 144-box pile.

A pass is the loop of a program that owns the states (a controller, a trainer, a renderer): the
scene's state is written from page-locked host memory, the scene advances `steps` time steps and
the new state is read back, through the calls of ``paper_2609_02675_gb300.Scene``.  The
broad-phase case calls the allocation-free entry point on device buffers.

``exact`` restates the step in plain torch, in 64 bits; only the contact geometry stays in single
precision, operation by operation, as the method here is defined (the sides of a decision, such
as a box's reference face, are taken from it).
"""
import math

import numpy as np
import torch

import paper_2609_02675_gb300 as pabd
import scenes

_CASES = [
    # one articulated figure in an interactive loop: the smallest call, all latency and launches
    dict(name="chain_8", kind="chain", n=8, steps=1),
    # the paper's mass-ratio chain under augmented Lagrangian bonds (Table 2: 19 bodies)
    dict(name="al_chain_19", kind="al", n=18, steps=1),
    # the paper's 11 x 11 spring net: springs alone, no contacts
    dict(name="net_121", kind="net", n=11, steps=1),
    # a slab under 48 x 48 boxes: one body with thousands of contacts
    dict(name="slab_2305", kind="slab", n=48, steps=1),
    # a server's pool: 24 resident piles of very different sizes stepped together as groups
    dict(name="pool_24", kind="pool", n=8000, groups=24, steps=1),
    # the 4096-box pile at rest in its columns
    dict(name="pile_4096", kind="pile", n=4096, lbvh=False, steps=1),
    # a mid-size pile of a ragged count under the paper's broad phase, the linear BVH
    dict(name="pile_20011_lbvh", kind="pile", n=20011, lbvh=True, steps=1),
    # the largest pile: two steps between a program's reads
    dict(name="pile_262144", kind="pile", n=262144, lbvh=False, steps=2),
    # a small batch of articulated trees (evaluation of a controller)
    dict(name="trees_256", kind="trees", n=256, steps=2),
    # the training batch: 4096 trees, a control interval of two steps
    dict(name="trees_4096", kind="trees", n=4096, steps=2),
    # quadruped on a settled bed of 50 000 grains, with the flexible rod
    dict(name="quadruped_50k", kind="quadruped", n=100, layers=5, steps=1),
    # collision queries of a program that may not allocate: pairs alone, on device buffers
    dict(name="broadphase_16384", kind="broadphase", n=16384, steps=1),
]


def listed():
    return [dict(c) for c in _CASES]


def _between(rng, lo, hi):
    """A whole number spread over the logarithm of its range."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["chain", "net", "slab", "pool", "pile", "pile", "trees", "trees", "quadruped", "broadphase"])
    if kind == "chain":
        return dict(kind=kind, n=_between(rng, 3, 200), steps=rng.randint(1, 2))
    if kind == "net":
        return dict(kind=kind, n=_between(rng, 3, 60), steps=rng.randint(1, 2))
    if kind == "slab":
        return dict(kind=kind, n=_between(rng, 3, 90), steps=1)
    if kind == "pool":
        return dict(kind=kind, n=_between(rng, 400, 8000), groups=rng.randint(2, 32), steps=1)
    if kind == "pile":
        return dict(kind=kind, n=_between(rng, 30, 200000), lbvh=rng.random() < 0.25, steps=1)
    if kind == "trees":
        return dict(kind=kind, n=_between(rng, 1, 3500), steps=rng.randint(1, 2))
    if kind == "quadruped":
        return dict(kind=kind, n=_between(rng, 12, 100), layers=rng.randint(2, 5), steps=1)
    return dict(kind=kind, n=_between(rng, 100, 16384), steps=1)


# ---- inputs ----

def _turn(rng, quat, angle):
    """The orientations turned about random axes by normally distributed angles."""
    a = rng.normal(0.0, angle, (quat.shape[0], 3))
    th = np.linalg.norm(a, axis=1, keepdims=True) + 1e-300
    dq = np.concatenate([a * (np.sin(0.5 * th) / th), np.cos(0.5 * th)], axis=1)
    x, y, z, w = dq.T
    X, Y, Z, W = quat.T
    q = np.stack([w * X + x * W + y * Z - z * Y, w * Y - x * Z + y * W + z * X,
                  w * Z + x * Y - y * X + z * W, w * W - x * X - y * Y - z * Z], axis=1)
    return q / np.linalg.norm(q, axis=1, keepdims=True)


def _disturb(rng, sc, shift, angle, v, omega):
    """The scene's bodies as a running program holds them: displaced, turned and moving."""
    b, n, free = sc.bodies, sc.n_bodies, sc.bodies["pinned"] == 0
    b["c"][free] += rng.normal(0.0, shift, (n, 3))[free]
    b["quat"][free] = _turn(rng, b["quat"], angle)[free]
    b["v"][free] += rng.normal(0.0, v, (n, 3))[free]
    b["omega"][free] += rng.normal(0.0, omega, (n, 3))[free]
    return sc


def _pile(rng, n, seed):
    return _disturb(rng, scenes.box_pile_n(n, seed=seed, stacked=True), 0.0, 0.003, 0.1, 0.1)


def _pool(rng, n, groups, seed):
    """Piles of geometrically spread sizes, as the groups of one scene."""
    w = np.geomspace(1.0, 30.0, groups)
    sizes = np.maximum(10, (n * w / w.sum()).astype(int))
    parts = [_pile(rng, int(m), seed + 17 * k) for k, m in enumerate(sizes)]
    for k, p in enumerate(parts):
        p.bodies["group"] = k
    return scenes.Scene("pool", parts[0].params, np.concatenate([p.bodies for p in parts]), parts[0].bonds, 1)


def _trees(rng, n):
    """`n` trees of 4 to 64 boxes, half of them on the ground and half about to land: the sizes,
    joints and stiffnesses of ``scenes.batched_trees``, all boxes of a tree of one height, each child at a free
    side of its parent or on top of it, slightly out of joint and moving."""
    sizes = np.random.default_rng(n).integers(4, 65, n)
    base = np.concatenate([[0], np.cumsum(sizes)[:-1]])
    N = int(sizes.sum())
    b = np.zeros(N, dtype=scenes.BODY_DTYPE)
    b["he"] = rng.uniform(0.05, 0.25, (N, 3))
    b["he"][:, 1] = np.repeat(rng.uniform(0.05, 0.25, n), sizes)
    he = b["he"]
    b["mass"] = 8000.0 * he.prod(axis=1)
    b["group"] = np.repeat(np.arange(n), sizes)
    low = np.repeat(np.where(rng.random(n) < 0.5, 0.0003, 0.05), sizes)  # height of each box's underside
    c = np.zeros((N, 3))
    c[base, 1] = low[base] + he[base, 1]
    h, gap, bonds = 1.0 / 120.0, 0.02, []
    free = np.ones((N, 5), dtype=bool)  # faces +x, -x, +z, -z and +y without a child
    for i in range(1, 64):
        g = np.nonzero(sizes > i)[0]
        k = base[g] + i
        cand = base[g][:, None] + np.arange(i)
        p = base[g] + np.argmax(rng.random(cand.shape) * free[cand].any(axis=2), axis=1)
        face = np.argmax(rng.random((g.size, 5)) * free[p], axis=1)
        free[p, face] = False
        top = face == 4
        free[k[~top], face[~top] ^ 1] = False  # the face that looks back at the parent
        ax = np.where(top, 1, 2 * (face // 2))
        sg = np.where(top | (face % 2 == 0), 1.0, -1.0)
        r = np.arange(g.size)
        low[k] = np.where(top, low[p] + 2.0 * he[p, 1] + gap, low[p])
        c[k] = c[p]
        c[k, ax] += sg * (he[p, ax] + gap + he[k, ax])
        c[k, 1] = low[k] + he[k, 1]
        at = c[p].copy()  # the joint: the middle of the parent's face
        at[r, ax] += sg * he[p, ax]
        kind = np.array([scenes.SPHERICAL, scenes.REVOLUTE, scenes.ELASTIC_NL])[rng.integers(0, 3, g.size)]
        q = np.zeros(g.size, dtype=scenes.BOND_DTYPE)
        q["type"], q["i"], q["j"] = kind, p, k
        q["xi"], q["xj"] = at - c[p], at - c[k]
        soft = kind == scenes.ELASTIC_NL
        q["xj"][r[soft], ax[soft]] += (sg * gap)[soft]
        q["kappa"] = np.where(soft, 100.0, 1000.0) * np.minimum(b["mass"][p], b["mass"][k]) / h ** 2
        q["rest"] = np.where(soft, gap, 0.0)
        q["axis"][r, (ax + 1 + rng.integers(0, 2, g.size)) % 3] = 1.0
        q["arm"] = np.where(kind == scenes.REVOLUTE, 0.5 * he[k].min(axis=1), 0.0)
        bonds.append(q)
    b["c"], b["quat"][:, 3] = c, 1.0
    par = scenes.default_params(h=h, n_iter=10, mu=0.5, body_contacts=0)
    bo = np.concatenate(bonds)
    return scenes.Scene("trees", par, b, bo[np.argsort(bo["j"], kind="stable")], 1)


def _quadruped(rng, n, layers, seed):
    """``scenes.quadruped_bed_rod`` after the grains have settled: layers on each other, the
    quadruped's feet on the bed."""
    sc = scenes.quadruped_bed_rod(seed, bed=(n, layers, n))
    bed = slice(13, 13 + n * n * layers)
    c, k = sc.bodies["c"], np.arange(n * n * layers)
    drop = layers * (0.056 - 0.0302) + 0.02
    c[:13, 1] -= drop
    c[bed.stop:, 1] -= drop
    c[bed, 0] = (k % n - 0.5 * (n - 1)) * 0.034
    c[bed, 1] = 0.0151 + (k // (n * n)) * 0.0302
    c[bed, 2] = (k // n % n - 0.5 * (n - 1)) * 0.034
    c[bed] += rng.uniform(-1e-3, 1e-3, (k.size, 3)) * (1.0, 0.05, 1.0)
    yaw = rng.uniform(-0.3, 0.3, k.size)
    q = np.stack([0 * yaw, np.sin(0.5 * yaw), 0 * yaw, np.cos(0.5 * yaw)], axis=1)
    sc.bodies["quat"][bed] = _turn(rng, q, 0.01)
    sc.bodies["v"][bed] = rng.normal(0.0, 0.02, (k.size, 3))
    return sc


def _scene(case, seed):
    rng = np.random.default_rng([seed, case["n"]])
    kind, n = case["kind"], case["n"]
    if kind == "chain":
        sc = _disturb(rng, scenes.chain_pendulum(seed=seed, n_bodies=n), 1e-4, 1e-3, 0.3, 0.3)
    elif kind == "al":
        sc = _disturb(rng, scenes.mass_ratio_chain(n=n), 1e-3, 1e-3, 0.05, 0.05)
    elif kind == "net":
        sc = _disturb(rng, scenes.spring_net(n), 0.01, 0.02, 0.3, 0.3)
    elif kind == "slab":
        sc = _disturb(rng, scenes.slab_pile(n, seed=seed), 0.0, 0.002, 0.03, 0.03)
    elif kind == "pool":
        sc = _pool(rng, n, case["groups"], seed)
    elif kind == "trees":
        sc = _disturb(rng, _trees(rng, n), 2e-4, 0.002, 0.1, 0.2)
    elif kind == "quadruped":
        sc = _quadruped(rng, n, case["layers"], seed)
    elif kind == "broadphase":
        sc = _disturb(rng, scenes.box_pile_n(n, seed=seed, spacing=2.3), 0.2, 0.5, 1.0, 1.0)
    else:
        sc = _pile(rng, n, seed)
    b = sc.bodies
    for f in ("he", "mass", "c", "quat", "v", "omega"):
        b[f] = b[f].astype(np.float32)
    return sc


def _state(sc):
    """The state rows of ``Scene.write_state_f32``: (c, A), then Q, v and omega of every body."""
    b, n = sc.bodies, sc.n_bodies
    x, y, z, w = (b["quat"] / np.linalg.norm(b["quat"], axis=1, keepdims=True)).T
    A = np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                  2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                  2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], axis=1)
    pad = np.zeros((n, 1))
    rows = [np.concatenate([b["c"], A], axis=1), np.stack([x, y, z, w], axis=1),
            np.concatenate([b["v"], pad], axis=1), np.concatenate([b["omega"], pad], axis=1)]
    return np.concatenate([r.ravel() for r in rows]).astype(np.float32)


_streams = {}


def _stream():
    """One stream for all of a program's scenes."""
    dev = torch.cuda.current_device()
    if dev not in _streams:
        _streams[dev] = torch.cuda.Stream()
    return _streams[dev]


def prepare(case, seed):
    sc = _scene(case, seed)
    state, n = _state(sc), sc.n_bodies
    if case["kind"] == "broadphase":
        on = lambda a, t: torch.tensor(np.ascontiguousarray(a), dtype=t, device="cuda")  # noqa: E731
        return dict(n=n, par=sc.params, q=on(state[:12 * n], torch.float32), v=on(state[16 * n:20 * n], torch.float32),
                    he=on(np.pad(sc.bodies["he"], ((0, 0), (0, 1))), torch.float32),
                    group=on(sc.bodies["group"], torch.int32), flags=on(sc.bodies["pinned"], torch.int32),
                    pairs=torch.zeros((8 * n, 2), dtype=torch.int32, device="cuda"),
                    count=torch.zeros(1, dtype=torch.int32, device="cuda"))
    src = torch.from_numpy(state).pin_memory()
    g = pabd.Scene(sc, stream=_stream(), broadphase=1 if case.get("lbvh") else 0)
    g.write_state_f32(src.data_ptr())
    g.tune()
    return dict(g=g, src=src, dst=torch.empty_like(src).pin_memory(), steps=case["steps"])


def run(s):
    if "g" not in s:
        p = s["par"]
        pabd.pabd_broadphase_noalloc(s["q"].data_ptr(), s["v"].data_ptr(), s["he"].data_ptr(), s["group"].data_ptr(),
                                     s["flags"].data_ptr(), s["n"], p["h"], p["margin"], p["d_hat_rel"],
                                     s["pairs"].data_ptr(), s["pairs"].shape[0], s["count"].data_ptr(),
                                     torch.cuda.current_stream().cuda_stream)
        return dict(pairs=s["pairs"], count=s["count"])
    g = s["g"]
    g.write_state_f32(s["src"].data_ptr())
    g.step(s["steps"])
    g.read_state_f32(s["dst"].data_ptr())
    return dict(state=s["dst"])


def work(case):
    """State in and out and each body's and bond's description once; per sweep about 120
    operations a bond and 500 a body (assembly, 4 x 4 solve, rotation)."""
    n, steps = case["n"], case["steps"]
    bodies, ends, sweeps = {
        "chain": (n, n, 20), "al": (n + 1, n, 10), "net": (n * n, 2 * n * n, 20), "slab": (n * n + 1, 4 * n * n, 20),
        "pool": (n, 4 * n, 30), "pile": (n, 4 * n, 30), "trees": (34 * n, 75 * n, 10), "broadphase": (n, 2 * n, 0),
        "quadruped": (n * n * case.get("layers", 1) + 77, 4 * n * n * case.get("layers", 1), 20)}[case["kind"]]
    if case["kind"] == "broadphase":
        return {"bytes": 88 * bodies + 8 * ends, "flops": 60 * bodies + 12 * ends}
    return {"bytes": (2 * 96 + 48) * bodies + 64 * ends, "flops": steps * (sweeps * (500 * bodies + 120 * ends) + 400 * bodies)}


# ---- the step in 64 bits ----

def _dot(a, b):
    """Sum over three components in this order, each product and sum rounded."""
    return (a[..., 0] * b[..., 0] + a[..., 1] * b[..., 1]) + a[..., 2] * b[..., 2]


def _overlapping(lo, hi, group):
    """All i < j of one group whose boxes overlap: cells of the widest common box, and the few
    much wider boxes against all."""
    N, dev = lo.shape[0], lo.device
    width = (hi - lo).amax(dim=1)
    wide = width > 4.0 * width.median()
    found = []
    for i in torch.nonzero(wide).ravel().tolist():
        j = torch.nonzero((group == group[i]) & (lo <= hi[i]).all(1) & (lo[i] <= hi).all(1)).ravel()
        j = j[(j != i) & ~(wide[j] & (j < i))]
        i = torch.full_like(j, i)
        found.append(torch.stack([torch.minimum(i, j), torch.maximum(i, j)], 1))
    ids = torch.nonzero(~wide).ravel()
    cell = torch.floor(0.5 * (lo[ids] + hi[ids]).double() / (1.01 * float(width[ids].max()))).long()
    cell -= cell.amin(0) - 1
    dims = (cell.amax(0) + 2).tolist()
    key = ((group[ids].long() * dims[0] + cell[:, 0]) * dims[1] + cell[:, 1]) * dims[2] + cell[:, 2]
    key, order = torch.sort(key)
    ids = ids[order]
    for dx in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dz in (-1, 0, 1):
                to = key + (dx * dims[1] + dy) * dims[2] + dz
                a, b = torch.searchsorted(key, to), torch.searchsorted(key, to, right=True)
                i = torch.repeat_interleave(ids, b - a)
                at = torch.arange(i.numel(), device=dev) - torch.repeat_interleave((b - a).cumsum(0) - (b - a), b - a)
                j = ids[torch.repeat_interleave(a, b - a) + at]
                ok = (i < j) & (lo[i] <= hi[j]).all(1) & (lo[j] <= hi[i]).all(1)
                found.append(torch.stack([i[ok], j[ok]], 1))
    return torch.cat(found)


def _box_contacts(c, A, he, infl, ia, ib):
    """Contact points of the pairs (ia, ib): reference face by separation over the six face
    normals, the incident face clipped against its sides."""
    P, dev = ia.numel(), ia.device
    ca, cb, Aa, Ab, ha, hb = c[ia], c[ib], A[ia], A[ib], he[ia], he[ib]
    delta = infl[ia] + infl[ib]
    dv = ca - cb
    col = lambda M, k: M[:, :, k]  # noqa: E731
    best = ref_b = face = dsel = None
    for own, axis in [(1, 0), (1, 1), (1, 2), (0, 0), (0, 1), (0, 2)]:
        M, H, O, G, r = (Ab, hb, Aa, ha, dv) if own else (Aa, ha, Ab, hb, -dv)
        d = _dot(col(M, axis), r)
        R = torch.stack([_dot(col(Ab, axis), col(O, k)) if own else _dot(col(O, k), col(Aa, axis)) for k in range(3)], 1)
        sep = d.abs() - (H[:, axis] + _dot(R.abs(), G))
        if best is None:
            best, ref_b, face, dsel = sep, torch.ones_like(ia), torch.zeros_like(ia), d
        else:
            m = sep > best
            best, dsel = torch.where(m, sep, best), torch.where(m, d, dsel)
            ref_b, face = torch.where(m, own, ref_b), torch.where(m, axis, face)
    near = best <= delta
    ia, ib, delta, face, dsel = ia[near], ib[near], delta[near], face[near], dsel[near]
    rb = ref_b[near] == 1
    ir, ii = torch.where(rb, ib, ia), torch.where(rb, ia, ib)
    P = ia.numel()
    row = torch.arange(P, device=dev)
    cr, Ar, hr, ci, Ai, hi_ = c[ir], A[ir], he[ir], c[ii], A[ii], he[ii]
    sg = torch.where(dsel >= 0, 1.0, -1.0).float()
    N = sg[:, None] * Ar[row, :, face]
    dk = torch.stack([_dot(col(Ai, k), N) for k in range(3)], 1)
    ki = torch.zeros_like(face)
    for k in (1, 2):
        ki = torch.where(dk[:, k].abs() > dk[row, ki].abs(), k, ki)
    si = torch.where(dk[row, ki] > 0, -1.0, 1.0).float()
    poly = torch.zeros(P, 9, 6, dtype=torch.float32, device=dev)  # (u, x) of each corner; slot 8 takes what is dropped
    for v, (s1, s2) in enumerate([(1.0, 1.0), (-1.0, 1.0), (-1.0, -1.0), (1.0, -1.0)]):
        x = torch.zeros(P, 3, dtype=torch.float32, device=dev)
        x[row, ki] = si * hi_[row, ki]
        x[row, (ki + 1) % 3] = s1 * hi_[row, (ki + 1) % 3]
        x[row, (ki + 2) % 3] = s2 * hi_[row, (ki + 2) % 3]
        y = torch.stack([((ci[:, d] + Ai[:, d, 0] * x[:, 0]) + Ai[:, d, 1] * x[:, 1]) + Ai[:, d, 2] * x[:, 2] for d in range(3)], 1)
        poly[:, v, :3] = torch.stack([_dot(col(Ar, m), y - cr) for m in range(3)], 1)
        poly[:, v, 3:] = x
    count = torch.full((P,), 4, dtype=torch.long, device=dev)
    for plane in range(4):
        m = (face + 1 + plane // 2) % 3
        ps, lim = (1.0 if plane % 2 == 0 else -1.0), hr[row, m]
        out, nt = torch.zeros_like(poly), torch.zeros_like(count)
        for v in range(8):
            live = v < count
            p, q = poly[:, v], poly[row, (v + 1) % torch.clamp(count, min=1)]
            dp, dq = ps * p[row, m] - lim, ps * q[row, m] - lim
            keep = live & (dp <= 0)
            out[row, torch.where(keep, nt, 8)] = p
            nt = nt + keep
            cut = live & ((dp <= 0) != (dq <= 0))
            t = dp / torch.where(cut, dp - dq, 1.0)
            out[row, torch.where(cut, nt, 8)] = p + t[:, None] * (q - p)
            nt = nt + cut
        poly, count = out, nt
    xs = poly[:, :8, 3:]
    us = poly[:, :8, :3].clone()
    high = sg[:, None] * us[row, :, face] - hr[row, face][:, None]
    us[row, :, face] = (sg * hr[row, face])[:, None].expand(-1, 8)
    k, v = torch.nonzero((torch.arange(8, device=dev)[None] < count[:, None]) & (high < delta[:, None]), as_tuple=True)
    return ii[k], ir[k], xs[k, v], us[k, v], N[k]


def _contacts(sc, par, c, A, v, he, group, pinned):
    """This step's contacts, from the single-precision state: (i, j or -1, x_i, x_j, N)."""
    f = lambda x: float(np.float32(x))  # noqa: E731
    dev = c.device
    small = he.amin(1)
    infl = (f(par["d_hat_rel"]) * (2.0 * small) + f(par["h"]) * torch.sqrt(_dot(v, v))) + f(par["margin"])
    found = []
    if par["body_contacts"]:
        e = torch.stack([_dot(A[:, k].abs(), he) for k in range(3)], 1) + infl[:, None]
        pairs = _overlapping(c - e, c + e, group)
        pairs = pairs[~(pinned[pairs[:, 0]] & pinned[pairs[:, 1]])]
        if len(sc.bonds):
            bi, bj = (torch.tensor(sc.bonds[k].astype(np.int64), device=dev) for k in ("i", "j"))
            joined = torch.minimum(bi, bj) * c.shape[0] + torch.maximum(bi, bj)
            pairs = pairs[~torch.isin(pairs[:, 0] * c.shape[0] + pairs[:, 1], joined)]
        found.append(_box_contacts(c, A, he, infl, pairs[:, 0], pairs[:, 1]))
    if par["has_ground"]:
        ids = torch.nonzero(~pinned).ravel()
        n = torch.tensor(par["ground_n"], dtype=torch.float32, device=dev)
        for k in range(8):
            sgn = torch.tensor([1.0 if k & (1 << a) else -1.0 for a in range(3)], device=dev)
            x = sgn * he[ids]
            y = torch.stack([((c[ids, d] + A[ids, d, 0] * x[:, 0]) + A[ids, d, 1] * x[:, 1]) + A[ids, d, 2] * x[:, 2] for d in range(3)], 1)
            g = _dot(n.expand_as(y), y) - f(par["ground_d"])
            on = g < infl[ids]
            i = ids[on]
            found.append((i, torch.full_like(i, -1), x[on], y[on] - g[on][:, None] * n, n.expand(i.numel(), 3)))
    return [torch.cat(t) for t in zip(*found)] if found else None


def _rotation(X):
    """The rotation nearest to each matrix: Newton's iteration where the determinant is clearly
    positive, else the singular value decomposition."""
    def cof(X):
        return torch.stack([torch.linalg.cross(X[:, 1], X[:, 2]), torch.linalg.cross(X[:, 2], X[:, 0]),
                            torch.linalg.cross(X[:, 0], X[:, 1])], 1)
    C = cof(X)
    det = (X[:, 0] * C[:, 0]).sum(1)
    bad = ~(det > 1e-3 * X.square().sum((1, 2)) ** 1.5)
    Y = torch.where(bad[:, None, None], torch.eye(3, dtype=X.dtype, device=X.device), X)
    for _ in range(12):
        C = cof(Y)
        det = (Y[:, 0] * C[:, 0]).sum(1)[:, None, None]
        g = det.pow(-1.0 / 3.0)
        Y = 0.5 * (g * Y + C / (g * det))
    if bool(bad.any()):
        U, _, Vh = torch.linalg.svd(X[bad])
        U[:, :, 2] *= torch.sign(torch.linalg.det(U @ Vh))[:, None]
        Y[bad] = U @ Vh
    return Y


def _solve4(G, R):
    """G X = R for symmetric positive definite 4 x 4 matrices, by LDL^T."""
    n, L, D = 4, {}, []
    y = [R[:, k] for k in range(n)]
    for j in range(n):
        D.append(G[:, j, j] - sum((L[j, k] ** 2 * D[k] for k in range(j)), torch.zeros_like(G[:, 0, 0])))
        for i in range(j + 1, n):
            L[i, j] = (G[:, i, j] - sum((L[i, k] * L[j, k] * D[k] for k in range(j)), torch.zeros_like(D[0]))) / D[j]
    for i in range(n):
        for k in range(i):
            y[i] = y[i] - L[i, k][:, None] * y[k]
    x = [y[k] / D[k][:, None] for k in range(n)]
    for i in reversed(range(n)):
        for k in range(i + 1, n):
            x[i] = x[i] - L[k, i][:, None] * x[k]
    return torch.stack(x, 1)


def _user_bonds(sc):
    """The user's bonds as point bonds (rule, i, j, x_i, x_j, w, rest length), the zero-length
    ones of revolute joints and drives included, and what moves a drive's anchor."""
    b, h = sc.bonds, sc.params["h"]
    X, Y, Z, W = sc.bodies["quat"].T
    rot = lambda k: np.array(_matrix(X[k], Y[k], Z[k], W[k]))  # noqa: E731
    rows, moving = [], []
    for q in b:
        w = h * h * q["kappa"]
        if q["type"] in (scenes.REVOLUTE, scenes.DRIVE):
            u = q["axis"] / np.linalg.norm(q["axis"])
            to = rot(q["j"]).T @ rot(q["i"])
        if q["type"] == scenes.REVOLUTE:
            for s in (1.0, -1.0):
                rows.append((0, q["i"], q["j"], q["xi"] + s * q["arm"] * u, q["xj"] + s * q["arm"] * (to @ u), w, 0.0))
        elif q["type"] == scenes.DRIVE:
            r = np.cross(u, np.eye(3)[int(np.argmin(np.abs(u)))])
            r /= np.linalg.norm(r)
            moving.append((len(rows), q["xi"].copy(), q["arm"], r, np.cross(u, r), q["amp"], q["period"], q["phase"]))
            rows.append((0, q["i"], q["j"], q["xi"], q["xj"] + q["arm"] * (to @ r), w, 0.0))
        else:
            rule = {scenes.SPHERICAL: 0, scenes.SPRING: 1, scenes.ELASTIC_NL: 2, scenes.AL_DISTANCE: 3}[int(q["type"])]
            rows.append((rule, q["i"], q["j"], q["xi"], q["xj"], h * h if rule == 3 else w, q["rest"]))
    return rows, moving


def _matrix(x, y, z, w):
    return [[1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w)],
            [2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w)],
            [2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)]]


def exact(case, seed):
    if case["kind"] == "broadphase":
        return None  # whole numbers
    sc = _scene(case, seed)
    par, N = sc.params, sc.n_bodies
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    D = lambda a: torch.tensor(np.ascontiguousarray(a, dtype=np.float64), device=dev)  # noqa: E731
    st = D(_state(sc))
    c, A = st[:12 * N].view(N, 12)[:, :3].clone(), st[:12 * N].view(N, 12)[:, 3:].reshape(N, 3, 3).clone()
    Q, v, w = (st[k * N:(k + 4) * N].view(N, 4).clone() for k in (12, 16, 20))
    v, w = v[:, :3].clone(), w[:, :3].clone()
    he, m = D(sc.bodies["he"]), D(sc.bodies["mass"])
    mass = torch.cat([m[:, None], m[:, None] * he.square() / 3.0], 1)
    pinned = torch.tensor(sc.bodies["pinned"] != 0, device=dev)
    group = torch.tensor(sc.bodies["group"].astype(np.int64), device=dev)
    dhat = par["d_hat_rel"] * 2.0 * he.amin(1)
    rows, moving = _user_bonds(sc)
    I = lambda a: torch.tensor(np.array(a, dtype=np.int64), device=dev)  # noqa: E731
    nb = len(rows)
    rule = I([r[0] for r in rows])
    bi, bj = I([r[1] for r in rows]), I([r[2] for r in rows])
    bxi, bxj = (D([r[k] for r in rows]).view(nb, 3) for k in (3, 4))
    bw, bl = D([r[5] for r in rows]), D([r[6] for r in rows])
    al = rule == 3
    kap0 = D(sc.bonds["kappa"])[al] if bool(al.any()) else None
    beta, alpha, gamma = (D(sc.bonds[k])[al] for k in ("beta", "alpha", "gamma")) if kap0 is not None else (None,) * 3
    kap, lam = (kap0, torch.zeros_like(kap0)) if kap0 is not None else (None, None)
    h, gr = par["h"], D(par["gravity"])
    for step in range(case["steps"]):
        for k, x0, arm, r, ur, amp, period, phase in moving:
            th = amp * math.sin(2.0 * math.pi * (step + 1) * h / period + phase)
            bxi[k] = D(x0 + arm * (math.cos(th) * r + math.sin(th) * ur))
        F = lambda a: a.float()  # noqa: E731
        found = _contacts(sc, par, F(c), F(A), F(v), F(he), group, pinned)
        if found is None:
            ki = kj = I([])
            kxi = kxj = kn = D(np.zeros((0, 3)))
        else:
            ki, kj = found[0], found[1]
            kxi, kxj, kn = (t.double() for t in found[2:])
        kjj = torch.where(kj < 0, ki, kj)
        big = torch.full_like(m, math.inf)
        mm = torch.where(pinned, big, m)
        kw = par["c_kappa"] * torch.minimum(mm[ki], mm[kjj])
        kd = torch.minimum(dhat[ki], dhat[kjj])
        # the predictor
        vs = v + h * gr
        cs = c + h * vs
        wx, wy, wz = w.unbind(1)
        qx, qy, qz, qw = Q.unbind(1)
        dq = torch.stack([wx * qw + wy * qz - wz * qy, wy * qw + wz * qx - wx * qz, wz * qw + wx * qy - wy * qx,
                          -(wx * qx + wy * qy + wz * qz)], 1)
        Qs = Q + 0.5 * h * dq
        Qs = Qs / Qs.norm(dim=1, keepdim=True)
        As = torch.stack([torch.stack(r, 1) for r in _matrix(*Qs.unbind(1))], 1)
        cs, As = torch.where(pinned[:, None], c, cs), torch.where(pinned[:, None, None], A, As)
        ck, Ak = cs.clone(), As.clone()
        if kap is not None:
            kap, lam = torch.maximum(gamma * kap, kap0), alpha * gamma * lam
        ti, tj = torch.cat([bi, ki]), torch.cat([bj, kj])
        txi, txj = torch.cat([bxi, kxi]), torch.cat([bxj, kxj])
        world = tj < 0
        tjj = torch.where(world, 0, tj)

        def gap(ck, Ak):
            yi = ck[ti] + (Ak[ti] @ txi[:, :, None])[:, :, 0]
            yj = torch.where(world[:, None], txj, ck[tjj] + (Ak[tjj] @ txj[:, :, None])[:, :, 0])
            return yj - yi

        def updated(r, kap, lam):
            C = r[:nb][al].norm(dim=1) - bl[al]
            return kap + beta * C.abs(), kap * C + lam

        for it in range(par["n_iter"]):
            r = gap(ck, Ak)
            if kap is not None and it > 0:
                kap, lam = updated(r, kap, lam)
            rb = r[:nb]
            d = rb.norm(dim=1)
            n = torch.where((d > 0)[:, None], rb / d[:, None], D([0.0, 1.0, 0.0]))
            f, W = bw[:, None] * rb, bw.clone()
            s = rule == 1
            f[s] = (bw * (d - bl))[s][:, None] * n[s]
            s = rule == 2
            l = bl[s]
            f[s] = (bw[s] / 3.0 * (d[s] - l) * (d[s] ** 2 + d[s] * l + l * l) / (l * l))[:, None] * n[s]
            W[s] = bw[s] * d[s] ** 2 / (l * l)
            if kap is not None:
                cst = lam - kap * bl[al]
                W[al] = h * h * (kap + cst.clamp(min=0) / d[al].clamp(min=1e-9))
                f[al] = W[al][:, None] * rb[al] + (h * h * cst.clamp(max=0))[:, None] * n[al]
            rr = -r[nb:]
            g = (kn * rr).sum(1)
            t = rr - g[:, None] * kn
            tn, tau = t.norm(dim=1), par["mu"] * (kd - g)
            keep = torch.where(tn > tau, 1.0 - tau / tn, torch.zeros_like(tn))
            on = (g < kd).double()
            kf = (kw * on)[:, None] * (kd[:, None] * kn + keep[:, None] * t - rr)
            f, W = torch.cat([f, kf]), torch.cat([W, kw * on])
            one = torch.ones_like(W)[:, None]
            G = torch.diag_embed(mass)
            R = mass[:, :, None] * torch.cat([(cs - ck)[:, None], (As - Ak).transpose(1, 2)], 1)
            for ids, x, sgn, live in ((ti, txi, 1.0, None), (tjj, txj, -1.0, ~world)):
                x1 = torch.cat([one, x], 1)
                gx, rx = W[:, None, None] * x1[:, :, None] * x1[:, None], sgn * x1[:, :, None] * f[:, None]
                if live is not None:
                    gx, rx, ids = gx[live], rx[live], ids[live]
                G.index_add_(0, ids, gx)
                R.index_add_(0, ids, rx)
            X = _solve4(G, R)
            cn, An = ck + X[:, 0], Ak + X[:, 1:].transpose(1, 2)
            if par["project"]:
                An = _rotation(An)
            ck = torch.where(pinned[:, None], c, cn)
            Ak = torch.where(pinned[:, None, None], A, An)
        if kap is not None:
            kap, lam = updated(gap(ck, Ak), kap, lam)
        # velocities and the quaternion of the new rotation
        Wk = (Ak - A) @ A.transpose(1, 2) / h
        free = ~pinned
        v = torch.where(free[:, None], (ck - c) / h, v)
        w = torch.where(free[:, None], 0.5 * torch.stack([Wk[:, 2, 1] - Wk[:, 1, 2], Wk[:, 0, 2] - Wk[:, 2, 0], Wk[:, 1, 0] - Wk[:, 0, 1]], 1), w)
        tr = Ak[:, 0, 0] + Ak[:, 1, 1] + Ak[:, 2, 2]
        quad = torch.stack([1 + 2 * Ak[:, k, k] - tr for k in range(3)] + [1 + tr], 1).clamp(min=0)
        lead = quad.argmax(1)
        o = lambda a, b, s: Ak[:, a, b] + s * Ak[:, b, a]  # noqa: E731
        K = torch.stack([torch.stack([quad[:, 0], o(1, 0, 1), o(2, 0, 1), o(2, 1, -1)], 1),
                         torch.stack([o(1, 0, 1), quad[:, 1], o(2, 1, 1), o(0, 2, -1)], 1),
                         torch.stack([o(2, 0, 1), o(2, 1, 1), quad[:, 2], o(1, 0, -1)], 1),
                         torch.stack([o(2, 1, -1), o(0, 2, -1), o(1, 0, -1), quad[:, 3]], 1)], 1)
        q = K[torch.arange(N, device=dev), lead]
        q = q / q.norm(dim=1, keepdim=True)
        q = torch.where(((q * Q).sum(1) < 0)[:, None], -q, q)
        Q = torch.where(free[:, None], q, Q)
        c, A = ck, Ak
    zero = torch.zeros(N, 1, dtype=torch.float64, device=dev)
    parts = [torch.cat([c, A.reshape(N, 9)], 1), Q, torch.cat([v, zero], 1), torch.cat([w, zero], 1)]
    return dict(state=torch.cat([p.reshape(-1) for p in parts]).cpu().numpy())
