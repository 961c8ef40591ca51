"""Performance cases: the calls a solver built on this library makes, over the sizes it makes them at.

Most cases are one whole contact pass (contact_build, contact_filter, barrier_eval, ccd_step: what every
Newton iteration runs) and the first product with its Hessian, on one of the scene families of paper_2510_10256_gb300.scenes, from a patch of a few
hundred vertices, where launches and host waits count, to a 256 x 256 pleated sheet, a 200,000-triangle graded
disk and a batch of 64 yarn scenes.  The others are the calls a Newton solver makes around the pass: the
line search's energy, the products of its conjugate-gradient solve with and without lagged friction, and the
step bound of a caller's own stencil list.

A case is a dict of plain values: "call" names the entry points, "scene" the family, "size" its scale (vertices
per side, yarns per direction, triangles, loops or scenes) and "mollifier" IPC's edge-edge mollifier.  Sheets
keep the edge 0.5 mm, thickness 1 mm and dhat 0.05 mm of the repository's pleated sheet, yarns the parameters
of its woven patch, rod batch and loop chain.
"""
import math

import numpy as np
import torch

from paper_2510_10256_gb300 import contact, scenes

DEV = torch.device("cuda", 0) if torch.cuda.is_available() else torch.device("cpu")
MU, EPS = 0.4, 1e-3   # friction coefficient and sliding tolerance (mm) of the friction case
SHIFT = 4.0           # 1 / h^2 of the Newton system's inertia term


def listed():
    return [
        # the smallest pass: two layers of a 12 x 12 grid pressed together (a unit test, a button, a hem)
        dict(name="pass_layers_12", call="pass", scene="layers", size=12, mollifier=False),
        # the woven rod patch of the benchmark: 16 yarns of 257 vertices, every crossing at the thickness
        dict(name="pass_woven_8", call="pass", scene="woven", size=8, mollifier=False),
        # a sheet of an odd size in the middle of the range
        dict(name="pass_pleated_97", call="pass", scene="pleated", size=97, mollifier=False),
        # the benchmark's default workload
        dict(name="pass_pleated_256", call="pass", scene="pleated", size=256, mollifier=False),
        # few active pairs among many candidates: a graded sheet, 0.1 to 4 mm edges
        dict(name="pass_graded_200k", call="pass", scene="graded", size=200_000, mollifier=False),
        # many scenes in one launch sequence: 64 weaves and knits of 1k to 64k vertices
        dict(name="pass_batch_64", call="pass", scene="batch", size=64, mollifier=False),
        # closed yarn loops, 2,000 interlocked rings
        dict(name="pass_chain_2000", call="pass", scene="chain", size=2000, mollifier=False),
        # the pass with IPC's edge-edge mollifier
        dict(name="pass_mollified_128", call="pass", scene="pleated", size=128, mollifier=True),
        # a line-search trial: candidates and energy at x + alpha p, no derivatives
        dict(name="energy_pleated_181", call="energy", scene="pleated", size=181, mollifier=False),
        # one product of the conjugate-gradient solve with the assembled Hessian
        dict(name="product_pleated_256", call="product", scene="pleated", size=256, mollifier=False),
        # lagged friction: energy, gradient and one conjugate-gradient product with the friction Hessian
        dict(name="friction_pleated_200", call="friction", scene="pleated", size=200, mollifier=False),
        # the step bound of a caller's stencil list that may not allocate
        dict(name="stencils_pleated_52", call="stencils", scene="pleated", size=52, mollifier=False),
    ]


# per call and family: the sizes a drawn case takes (spread over their logarithm)
_RANGES = [
    ("pass", "layers", 6, 40), ("pass", "woven", 2, 24), ("pass", "pleated", 20, 256), ("pass", "graded", 4_000, 200_000),
    ("pass", "batch", 3, 40), ("pass", "chain", 20, 2000), ("energy", "pleated", 20, 256), ("energy", "woven", 2, 24),
    ("product", "pleated", 40, 256), ("product", "woven", 3, 24), ("friction", "pleated", 40, 256),
    ("stencils", "pleated", 12, 56),
]


def draw(rng):
    call, scene, lo, hi = rng.choice(_RANGES)
    size = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    moll = call == "pass" and scene in ("layers", "woven", "pleated") and size <= 128 and rng.random() < 0.2
    return dict(call=call, scene=scene, size=size, mollifier=moll)


# ------------------------------------------------------------------ inputs

def _scenes(case, seed):
    """The members (one scene but for a batch) of a case, from the seed alone."""
    n, fam, s = case["size"], case["scene"], 1_000 * int(seed)
    if fam == "layers":
        return [scenes.tiny_shell(s + 1, nx=n)]
    if fam == "woven":
        return [scenes.woven_patch(seed=s + 2, n_warp=n, n_weft=n, nseg=256 if n >= 8 else 32 * n)]
    if fam == "pleated":
        return [scenes.pleated_sheet(seed=s + 3, nx=n)]
    if fam == "graded":
        return [scenes.graded_disk(seed=s + 4, target_tris=n)]
    if fam == "chain":
        return [scenes.ring_chain(seed=s + 5, n_rings=n, m=96)]
    if fam == "batch":
        return _rod_batch(n, s + 6)
    raise ValueError(fam)


def _rod_batch(count, seed):
    """Weaves and knits in turn with the sizes and yarns of the repository's rod batch (1k to 64k vertices,
    log-uniform; radius 0.05 to 0.3, segment 0.2 to 1 radius).  Sizes and yarns follow from the count, the
    jitter, the loops' gaps and the directions from the seed."""
    rng, out = np.random.default_rng(scenes.BASE_SEED + 4), []
    for k in range(count):
        n = int(round(math.exp(rng.uniform(math.log(1e3), math.log(6.4e4)))))
        r = float(rng.uniform(0.05, 0.3))
        seg = float(rng.uniform(0.2 * r, r))
        make = scenes.knit_rows if k % 2 else scenes.weave_sized
        out.append(make(seed + 1000 + k, n, r, seg, 0.1 * r, sigma=0.2 * r))
    return out


def _trial(sc):
    """The line search's trial point: a tenth of the way along p."""
    return sc.x + 0.1 * sc.p


def _slid(sc, seed):
    """Positions a sliding tolerance away from the lagged ones."""
    return sc.x + np.random.default_rng(7_000_000 + int(seed)).normal(0.0, EPS, size=sc.x.shape)


def _vector(n, seed):
    """A vector to multiply."""
    return np.random.default_rng(8_000_000 + int(seed)).normal(size=(3, n))


class State:
    pass


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def prepare(case, seed):
    st = State()
    st.case = dict(case)
    scs = _scenes(case, seed)
    members = [contact.ContactScene.from_scene(sc, mollifier=bool(case["mollifier"])) for sc in scs]
    if case["scene"] == "batch":
        st.cs = contact.ContactBatch(members)
        for m in members:
            m.close()
    else:
        st.cs = members[0]
    st.x = _dev(np.concatenate([sc.x for sc in scs], axis=1))
    st.p = _dev(np.concatenate([sc.p for sc in scs], axis=1))
    st.energy = torch.zeros(len(scs), dtype=torch.float64, device=DEV)
    st.alpha = torch.zeros(len(scs), dtype=torch.float64, device=DEV)
    st.grad = torch.zeros(3, st.cs.n, dtype=torch.float64, device=DEV)
    call = case["call"]
    if call == "energy":
        st.x = _dev(_trial(scs[0]))
    st.v, st.y = _dev(_vector(st.cs.n, seed)), torch.zeros_like(st.x)
    if call in ("product", "friction"):
        st.cs.contact_build(st.x)
        st.cs.contact_filter()
        st.cs.barrier_eval(st.x, st.energy, st.grad)
        if call == "friction":
            st.x1 = _dev(_slid(scs[0], seed))
            st.cs.friction_lag(st.x, MU, EPS)
    if call == "stencils":
        st.cs.contact_build(st.x)
        st.cs.contact_filter()
        st.cs.ccd_step(st.x, st.p, st.alpha)
        got = st.cs.ccd()
        st.list = _stencil_list(scs[0], got["keys"], got["klass"])
        st.flags = torch.zeros(1, dtype=torch.int32, device=DEV)
        st.cs.close()
    return st


def _stencil_list(sc, keys, klass):
    """A caller's list: vertex ids, kind and offset of each pair."""
    lo = np.uint64(0x7FFFFFFF)
    i, j = ((keys >> np.uint64(31)) & lo).astype(np.int64), (keys & lo).astype(np.int64)
    pt = (keys >> np.uint64(62)) == 1
    t, e = np.asarray(sc.tris, np.int64), _edges_of(sc)
    ids = np.empty((keys.size, 4), np.int32)
    ids[pt, 0], ids[pt, 1:] = i[pt], t[:, j[pt]].T
    ids[~pt, :2], ids[~pt, 2:] = e[i[~pt]], e[j[~pt]]
    off = np.where((klass & 0x7F) == 0, sc.thickness, 0.0)
    return _dev(ids), _dev((~pt).astype(np.uint8)), _dev(off)


def run(st):
    cs, call = st.cs, st.case["call"]
    if call == "pass":
        cs.run_pass(st.x, st.p, st.energy, st.grad, st.alpha)
        cs.bsr_spmv(st.v, st.y, SHIFT)
        return dict(energy=st.energy, grad=st.grad, alpha=st.alpha, y=st.y)
    if call == "energy":
        cs.contact_build(st.x)
        cs.contact_filter()
        cs.barrier_energy(st.x, st.energy)
        return dict(energy=st.energy)
    if call == "product":
        cs.bsr_spmv(st.v, st.y, SHIFT)
        return dict(y=st.y)
    if call == "friction":
        st.energy.zero_()
        st.grad.zero_()
        cs.friction_eval(st.x1, st.x, st.energy, st.grad)
        cs.bsr_spmv(st.v, st.y, SHIFT)
        cs.friction_spmv(st.v, st.y)
        return dict(energy=st.energy, grad=st.grad, y=st.y)
    ids, ee, off = st.list
    contact.ccd_step_noalloc(st.x, st.p, ids, ee, off, st.alpha, st.flags)
    return dict(alpha=st.alpha, flags=st.flags)


# Per vertex (pass on a sheet or yarns of the family): broad-phase candidates, active pairs, blocks of the
# Hessian, pairs of the swept broad phase; per vertex topology bytes.  Mean counts of the listed
# sizes.
_PER_VERTEX = {
    "layers": (170.0, 34.0, 36.0, 167.0, 44), "woven": (5.5, 0.5, 2.0, 5.5, 8), "pleated": (235.0, 15.0, 28.0, 240.0, 48),
    "graded": (260.0, 0.0004, 0.0035, 278.0, 48), "batch": (6.6, 0.9, 4.6, 7.1, 8), "chain": (7.0, 0.76, 6.3, 10.3, 8),
}
# FP64 operations a pair cannot do without: its exact distance, barrier and derivatives with the projection; an
# FP32 bound settles each other candidate and swept pair.
_FLOP_ACTIVE, _FLOP_BOUND = 900.0, 60.0


def _vertices(case):
    n, fam = case["size"], case["scene"]
    return {"layers": 2 * n * n, "woven": 2 * n * ((256 if n >= 8 else 32 * n) + 1), "pleated": n * n, "graded": n // 2,
            "chain": 96 * n, "batch": 17_000 * n}[fam]


def work(case):
    """Bytes: positions (and p) in, topology, results out, each once; flops: the pairs' arithmetic."""
    n = _vertices(case)
    cand, act, nnzb, ccd, topo = _PER_VERTEX[case["scene"]]
    call = case["call"]
    if call == "pass":
        return dict(bytes=n * (120.0 + topo + 76.0 * nnzb + 4.0), flops=n * (_FLOP_ACTIVE * act + _FLOP_BOUND * (cand + ccd)))
    if call == "energy":
        return dict(bytes=n * (24.0 + topo) + 8.0, flops=n * (60.0 * act + _FLOP_BOUND * cand))
    if call == "product":
        return dict(bytes=n * (52.0 + 76.0 * nnzb), flops=n * 18.0 * nnzb)
    if call == "friction":
        return dict(bytes=n * (148.0 + 76.0 * nnzb + 128.0 * act), flops=n * (18.0 * nnzb + 200.0 * act))
    return dict(bytes=n * 48.0 + n * ccd * 25.0, flops=n * ccd * 150.0)


# ------------------------------------------------------------------ the same results in 64 bits
# Plain torch, from the definitions: every pair whose inflated boxes overlap, typed distances, the offset
# barrier with autograd derivatives, eigenvalues clamped per pair, additive CCD pair by pair.

_INF = float("inf")


def _edges_of(sc):
    if sc.kind == "rod":
        out = []
        closed = sc.rod_closed if sc.rod_closed is not None else np.zeros(len(sc.rod_ptr) - 1, np.uint8)
        for a, b, c in zip(sc.rod_ptr[:-1], sc.rod_ptr[1:], closed):
            v = np.arange(a, b - 1, dtype=np.int64)
            out.append(np.stack([v, v + 1], axis=1))
            if c:
                out.append(np.array([[b - 1, a]], np.int64))
        return np.concatenate(out)
    t = np.asarray(sc.tris, np.int64)
    e = np.concatenate([np.sort(np.stack([t[a], t[b]], 1), axis=1) for a, b in ((0, 1), (1, 2), (0, 2))])
    return np.unique(e, axis=0)


def _labels(sc, edges):
    """Component of each vertex: the polyline, or the connected part of a mesh."""
    n = sc.rest.shape[1]
    if sc.kind == "rod":
        return _dev(np.repeat(np.arange(len(sc.rod_ptr) - 1, dtype=np.int64), np.diff(sc.rod_ptr)))
    lab, e = torch.arange(n, device=DEV), _dev(edges)
    while True:
        m = torch.minimum(lab[e[:, 0]], lab[e[:, 1]])
        new = lab.clone().scatter_reduce_(0, e[:, 0], m, "amin").scatter_reduce_(0, e[:, 1], m, "amin")
        new = new[new]
        if bool((new == lab).all()):
            return lab
        lab = new


def _boxes(ids, x, p, h):
    pts = x[ids]                                        # [m][verts][3]
    lo, hi = pts.amin(1), pts.amax(1)
    if p is not None:
        end = (x + p)[ids]
        lo, hi = torch.minimum(lo, end.amin(1)), torch.maximum(hi, end.amax(1))
    return lo - h, hi + h


def _ranges(start, stop, most=1 << 24):
    """(i, j) for every j in [start[i], stop[i]), in pieces."""
    cnt = (stop - start).clamp(min=0)
    cum = torch.cumsum(cnt, 0)
    total, at, k = int(cum[-1]) if cum.numel() else 0, 0, 0
    while at < total:
        k2 = max(k + 1, int(torch.searchsorted(cum, at + most, right=True)))
        c = cnt[k:k2]
        i = torch.repeat_interleave(torch.arange(k, min(k2, cnt.numel()), device=DEV), c)
        first = torch.cumsum(c, 0) - c
        yield i, start[i] + torch.arange(i.numel(), device=DEV) - first[i - k]
        at, k = int(cum[min(k2, cnt.numel()) - 1]), k2


def _overlap(A, B, i, j):
    return ((A[0][i] <= B[1][j]) & (B[0][j] <= A[1][i])).all(1)


def _pairs(sc, edges, x, p, h):
    """Stencils (vertex ids, [m][4]) and kinds of every pair whose boxes overlap and share no vertex."""
    e = _dev(edges)
    out = []
    E = _boxes(e, x, p, h)
    ax = int((E[1] - E[0]).mean(0).div(E[1].amax(0) - E[0].amin(0) + 1e-300).argmin())
    o = torch.argsort(E[0][:, ax])
    Es, es = (E[0][o], E[1][o]), e[o]
    stop = torch.searchsorted(Es[0][:, ax].contiguous(), Es[1][:, ax].contiguous(), right=True)
    for i, j in _ranges(torch.arange(1, e.shape[0] + 1, device=DEV), stop):
        k = _overlap(Es, Es, i, j)
        a, b = o[i[k]], o[j[k]]
        a, b = torch.minimum(a, b), torch.maximum(a, b)
        s = torch.cat([e[a], e[b]], 1)
        s = s[(s[:, 0:1] != s[:, 2:]).all(1) & (s[:, 1:2] != s[:, 2:]).all(1)]
        out.append((s, True))
    if sc.kind == "shell":
        t = _dev(np.asarray(sc.tris, np.int64).T)
        v = torch.arange(x.shape[0], device=DEV)
        P, T = _boxes(v[:, None], x, p, h), _boxes(t, x, p, h)
        op, ot = torch.argsort(P[0][:, ax]), torch.argsort(T[0][:, ax])
        Ps, Ts = (P[0][op], P[1][op]), (T[0][ot], T[1][ot])
        pl, tl = Ps[0][:, ax].contiguous(), Ts[0][:, ax].contiguous()
        # the later of the two starts inside the other: a triangle starting in [lo, hi] of the point, or a
        # point starting in (lo, hi] of the triangle
        for i, j in _ranges(torch.searchsorted(tl, pl), torch.searchsorted(tl, Ps[1][:, ax].contiguous(), right=True)):
            k = _overlap(Ps, Ts, i, j)
            out.append((torch.cat([op[i[k]][:, None], t[ot[j[k]]]], 1), False))
        for j, i in _ranges(torch.searchsorted(pl, tl, right=True), torch.searchsorted(pl, Ts[1][:, ax].contiguous(), right=True)):
            k = _overlap(Ps, Ts, i, j)
            out.append((torch.cat([op[i[k]][:, None], t[ot[j[k]]]], 1), False))
    got = []
    for ee in (False, True):
        parts = [s for s, f in out if f == ee]
        s = torch.cat(parts) if parts else torch.zeros((0, 4), dtype=torch.int64, device=DEV)
        got.append(s if ee else s[(s[:, :1] != s[:, 1:]).all(1)])
    return got                                          # point-triangle, edge-edge


def _dot(a, b):
    return a[:, 0] * b[:, 0] + a[:, 1] * b[:, 1] + a[:, 2] * b[:, 2]


def _cross(a, b):
    return torch.stack([a[:, 1] * b[:, 2] - a[:, 2] * b[:, 1], a[:, 2] * b[:, 0] - a[:, 0] * b[:, 2],
                        a[:, 0] * b[:, 1] - a[:, 1] * b[:, 0]], 1)


def _segment(q, e0, e1):
    """Squared distance of points to segments and where: 0 at e0, 1 at e1, 2 inside."""
    u, w = e1 - e0, q - e0
    lam, uu = _dot(w, u), _dot(u, u)
    r = torch.where(lam <= 0, 0, torch.where(lam >= uu, 1, 2))
    c, d0, d1 = _cross(w, u), e0 - q, e1 - q
    return torch.where(r == 2, _dot(c, c) / uu, torch.where(r == 0, _dot(d0, d0), _dot(d1, d1))), r


# types of both kinds as rows (w, u, v) over the four points: the distance is |w|, the distance of w from the
# line along u, or from the plane along u and v
_PT = [((-1, 1, 0, 0),), ((-1, 0, 1, 0),), ((-1, 0, 0, 1),), ((1, -1, 0, 0), (0, -1, 1, 0)), ((1, 0, -1, 0), (0, 0, -1, 1)),
       ((1, 0, 0, -1), (0, 1, 0, -1)), ((1, -1, 0, 0), (0, -1, 1, 0), (0, -1, 0, 1))]
_EE = [((-1, 0, 1, 0),), ((-1, 0, 0, 1),), ((0, -1, 1, 0),), ((0, -1, 0, 1),), ((1, 0, -1, 0), (0, 0, -1, 1)),
       ((0, 1, -1, 0), (0, 0, -1, 1)), ((-1, 0, 1, 0), (-1, 1, 0, 0)), ((-1, 0, 0, 1), (-1, 1, 0, 0)),
       ((-1, 0, 1, 0), (-1, 1, 0, 0), (0, 0, -1, 1))]


def _typed(X, ee):
    """Distance and type of stencils given relative to their first point."""
    a, b, c, d = X
    if ee:
        u, v, w = b - a, d - c, a - c
        n = _cross(u, v)
        cc, uu, vv = _dot(n, n), _dot(u, u), _dot(v, v)
        B, D, E = _dot(u, v), _dot(u, w), _dot(v, w)
        s, t = B * E - vv * D, uu * E - B * D
        inside = (cc > 1e-20 * uu * vv) & (s > 0) & (s < cc) & (t > 0) & (t < cc)
        g = _dot(c - a, n)
        segs = [(a, c, d, (0, 1, 4)), (b, c, d, (2, 3, 5)), (c, a, b, (0, 2, 6)), (d, a, b, (1, 3, 7))]
        face = 8
    else:
        n = _cross(c - b, d - b)
        cc = _dot(n, n)
        inside = (cc > 0) & (_dot(_cross(c, d), n) > 0) & (_dot(_cross(d, b), n) > 0) & (_dot(_cross(b, c), n) > 0)
        g = _dot(a - b, n)
        segs = [(a, b, c, (0, 1, 3)), (a, c, d, (1, 2, 4)), (a, d, b, (2, 0, 5))]
        face = 6
    best = torch.full_like(cc, _INF)
    ty = torch.full(cc.shape, 99, dtype=torch.int64, device=cc.device)
    for q, e0, e1, names in segs:
        s2, r = _segment(q, e0, e1)
        k = torch.tensor(names, device=cc.device)[r]
        take = (s2 < best) | ((s2 == best) & (k < ty))
        best, ty = torch.where(take, s2, best), torch.where(take, k, ty)
    best, ty = torch.where(inside, g * g / cc, best), torch.where(inside, face, ty)
    return torch.sqrt(best), ty


def _local(x, s):
    X = x[s]
    return [X[:, k] - X[:, 0] for k in range(4)]


def _distances(x, s, ee):
    d, ty = [], []
    for c in torch.split(s, 1 << 21):
        a, b = _typed(_local(x, c), ee)
        d.append(a)
        ty.append(b)
    return (torch.cat(d), torch.cat(ty)) if d else (x.new_zeros(0), s.new_zeros(0))


class _Rest:
    """Reference distances of a scene: which pairs are filtered, and the width of their barrier."""

    def __init__(self, sc):
        self.sc, self.edges, self.a = sc, _edges_of(sc), sc.thickness + sc.dhat
        self.comp, self.x = _labels(sc, self.edges), _dev(sc.rest.T)
        if sc.kind == "rod":
            S, L, first, last = np.zeros(sc.rest.shape[1]), [], [], []
            for k, (b, e) in enumerate(zip(sc.rod_ptr[:-1], sc.rod_ptr[1:])):
                seg = np.sqrt((np.diff(sc.rest[:, b:e], axis=1) ** 2).sum(0))
                S[b:e] = np.concatenate([[0.0], np.cumsum(seg)])
                closed = sc.rod_closed is not None and sc.rod_closed[k]
                L.append(S[e - 1] + np.sqrt(((sc.rest[:, b] - sc.rest[:, e - 1]) ** 2).sum()) if closed else _INF)
            self.S, self.L = _dev(S), _dev(np.array(L))
            # the closest non-incident edges of one polyline: two apart
            k = np.arange(self.edges.shape[0] - 2)
            s = _dev(np.concatenate([self.edges[k], self.edges[k + 2]], 1))
            s = [torch.zeros((0, 4), dtype=torch.int64, device=DEV), s]
            if any(math.isfinite(v) for v in L):        # and those on the other side of a loop's seam
                wrap = []
                for b, e, l in zip(sc.rod_ptr[:-1], sc.rod_ptr[1:], L):
                    if math.isfinite(l):
                        m = e - b
                        for i, j in ((0, m - 2), (1, m - 1)):
                            wrap.append([b + i, b + i + 1, b + j, b + (j + 1) % m])
                s[1] = torch.cat([s[1], _dev(np.array(wrap, np.int64))])
        else:
            s = _pairs(sc, self.edges, self.x, None, 0.5 * self.a)
        self.width = _INF
        for k, ee in enumerate((False, True)):
            f, d = self.filtered(s[k], ee)
            if bool(f.any()):
                self.width = min(self.width, float(d[f].min()))

    def filtered(self, s, ee):
        same = self.comp[s[:, 0]] == self.comp[s[:, 2]]
        if self.sc.kind == "rod":
            # arc-length gap between the edges, the shorter way round a loop; a closing edge spans (last, L)
            L = self.L[self.comp[s[:, 0]]]
            s0, e0 = self.S[s[:, 0]], torch.where(s[:, 1] > s[:, 0], self.S[s[:, 1]], L)
            s1, e1 = self.S[s[:, 2]], torch.where(s[:, 3] > s[:, 2], self.S[s[:, 3]], L)
            d = torch.minimum(s1 - e0, (L - e1) + s0)
        else:
            d, _ = _distances(self.x, s, ee)
        return same & (d < self.a), d


def _kappa_barrier(y, w):
    return -((y - w) ** 2) * torch.log(y / w)


def _energy(C, X, off, w, eps=None):
    """Barrier energy of one stencil ([4][3]) of the type with rows C; with eps times the mollifier."""
    z = C @ X
    if len(C) == 1:
        d = torch.sqrt((z[0] * z[0]).sum())
    elif len(C) == 2:
        c = torch.linalg.cross(z[0], z[1])
        d = torch.sqrt((c * c).sum() / (z[1] * z[1]).sum())
    else:
        n = torch.linalg.cross(z[1], z[2])
        d = torch.abs((z[0] * n).sum()) / torch.sqrt((n * n).sum())
    b = _kappa_barrier(d - off, w)
    if eps is None:
        return b
    n = torch.linalg.cross(X[1] - X[0], X[3] - X[2])
    c = (n * n).sum()
    return b * torch.where(c < eps, (2.0 - c / eps) * c / eps, 1.0)


def _active(sc, rest, x):
    """Active pairs of a scene at x: (stencils, kind, type, distance, offset, width) per kind."""
    out = []
    for s, ee in zip(_pairs(sc, rest.edges, x, None, 0.5 * rest.a), (False, True)):
        d, ty = _distances(x, s, ee)
        near = d < rest.a
        s, d, ty = s[near], d[near], ty[near]
        f, _ = rest.filtered(s, ee)
        core = ~f & (d <= sc.thickness)
        off = torch.where(f | core, 0.0, torch.full_like(d, sc.thickness))
        w = torch.where(f, rest.width, torch.where(core, rest.a, torch.full_like(d, sc.dhat)))
        k = d - off < w
        out.append((s[k], ee, ty[k], d[k], off[k], w[k]))
    return out


def _barrier(sc, rest, x, moll, full=True):
    """Energy, gradient [n][3] and the projected Hessian's blocks: sorted keys row * n + col and values [9]."""
    n = x.shape[0]
    e, g, keys, vals = x.new_zeros(()), x.new_zeros(n, 3), [], []
    grad, hess = torch.func.grad(_energy, argnums=1), torch.func.hessian(_energy, argnums=1)
    for s, ee, ty, d, off, w in _active(sc, rest, x):
        l2 = None
        if moll and ee:
            r = rest.x[s]
            l2 = 1e-3 * ((r[:, 1] - r[:, 0]) ** 2).sum(1) * ((r[:, 3] - r[:, 2]) ** 2).sum(1)
        for t, rows in enumerate(_EE if ee else _PT):
            sel = torch.nonzero(ty == t)[:, 0]
            for part in torch.split(sel, 1 << 15):
                if part.numel() == 0:
                    continue
                X = x[s[part]]
                X = X - X[:, :1]
                arg = (x.new_tensor(rows), X, off[part], w[part]) + ((l2[part],) if l2 is not None else ())
                dims = (None,) + (0,) * (len(arg) - 1)
                e = e + torch.func.vmap(_energy, dims)(*arg).sum()
                if not full:
                    continue
                g.index_add_(0, s[part].reshape(-1), torch.func.vmap(grad, dims)(*arg).reshape(-1, 3))
                H = torch.func.vmap(hess, dims)(*arg).reshape(-1, 12, 12)
                lam, V = torch.linalg.eigh(0.5 * (H + H.transpose(1, 2)))
                H = (V * lam.clamp(min=0)[:, None, :]) @ V.transpose(1, 2)
                H = H.reshape(-1, 4, 3, 4, 3).permute(0, 1, 3, 2, 4).reshape(-1, 9)
                key = (s[part][:, :, None] * n + s[part][:, None, :]).reshape(-1)
                uk, inv = torch.unique(key, return_inverse=True)
                acc = x.new_zeros(uk.numel(), 9).index_add_(0, inv, H)
                keys.append(uk)
                vals.append(acc)
    if not full:
        return e, None, None, None
    # every block of an active stencil is in the pattern, zero ones too
    if not keys:
        return e, g, torch.zeros(0, dtype=torch.int64, device=DEV), x.new_zeros(0, 9)
    uk, inv = torch.unique(torch.cat(keys), return_inverse=True)
    return e, g, uk, x.new_zeros(uk.numel(), 9).index_add_(0, inv, torch.cat(vals))


def _step_bound(sc, rest, x, p):
    """min(1, t) of additive CCD (s = 0.1, factor 0.9) over the pairs of the swept boxes."""
    best = 1.0
    for s, ee in zip(_pairs(sc, rest.edges, x, p, 0.5 * sc.thickness), (False, True)):
        lb, off = [], []
        for c in torch.split(s, 1 << 21):
            d, _ = _typed(_local(x, c), ee)
            f, _ = rest.filtered(c, ee)
            o = torch.where(f | (d <= sc.thickness), 0.0, torch.full_like(d, sc.thickness))
            lp, _ = _motion(p, c, ee)
            t = torch.where(lp == 0, 1.0, 0.9 * (d - o) / lp)
            lb.append(t.clamp(max=1.0))
            off.append(o)
        lb, off = torch.cat(lb), torch.cat(off)
        order = torch.argsort(lb)
        for part in torch.split(order, 1 << 16):
            if part.numel() == 0 or float(lb[part[0]]) >= best:
                break
            best = min(best, _accd(x, p, s[part], ee, off[part], best))
    return best


def _motion(p, s, ee):
    P = p[s]
    Q = P - (P[:, 0] + P[:, 1] + P[:, 2] + P[:, 3])[:, None] * 0.25
    l = [torch.sqrt(_dot(Q[:, k], Q[:, k])) for k in range(4)]
    lp = torch.maximum(l[0], l[1]) + torch.maximum(l[2], l[3]) if ee else \
        l[0] + torch.maximum(torch.maximum(l[1], l[2]), l[3])
    return lp, Q


def _accd(x, p, s, ee, off, best):
    lp, Q = _motion(p, s, ee)
    Y = torch.stack(_local(x, s), 1)
    keep = lp > 0
    Y, Q, lp, off = Y[keep], Q[keep], lp[keep], off[keep]
    g0 = _typed([Y[:, k] - Y[:, 0] for k in range(4)], ee)[0] - off
    if bool((g0 <= 0).any()):
        return 0.0
    g, t, tl = 0.1 * g0, torch.zeros_like(g0), (1.0 - 0.1) * g0 / lp
    for _ in range(10000):
        if t.numel() == 0:
            break
        Y = Y + tl[:, None, None] * Q
        d = _typed([Y[:, k] - Y[:, 0] for k in range(4)], ee)[0]
        end = (t > 0) & (d - off < g)
        if bool(end.any()):
            best = min(best, float(t[end].min()))
        t = t + tl
        go = ~end & (t < best) & (t <= 1.0)
        tl = 0.9 * (d - off) / lp
        Y, Q, lp, off, g, t, tl = Y[go], Q[go], lp[go], off[go], g[go], t[go], tl[go]
    return best


def exact(case, seed):
    call, moll = case["call"], bool(case["mollifier"])
    scs = _scenes(case, seed)
    if call == "stencils":
        sc = scs[0]
        return dict(alpha=torch.tensor([_step_bound(sc, _Rest(sc), _dev(sc.x.T), _dev(sc.p.T))], dtype=torch.float64), flags=None)
    if call == "energy":
        sc = scs[0]
        e = _barrier(sc, _Rest(sc), _dev(_trial(sc).T), moll, full=False)[0]
        return dict(energy=e.reshape(1))
    es, gs, als, keys, vals, n = [], [], [], [], [], sum(sc.rest.shape[1] for sc in scs)
    at = 0
    for sc in scs:
        rest, x = _Rest(sc), _dev(sc.x.T)
        e, g, uk, val = _barrier(sc, rest, x, moll)
        m = sc.rest.shape[1]
        keys.append((torch.div(uk, m, rounding_mode="floor") + at) * n + uk % m + at)
        es.append(e.reshape(1))
        gs.append(g)
        vals.append(val)
        if call == "pass":
            als.append(_step_bound(sc, rest, x, _dev(sc.p.T)))
        at += m
    key, val = torch.cat(keys), torch.cat(vals).reshape(-1, 3, 3)
    row, col = torch.div(key, n, rounding_mode="floor"), key % n
    v = _dev(_vector(n, seed).T)
    y = SHIFT * v
    y.index_add_(0, row, (val @ v[col][:, :, None])[:, :, 0])
    if call == "pass":
        return dict(energy=torch.cat(es), grad=torch.cat(gs).T.contiguous(), y=y.T.contiguous(),
                    alpha=torch.tensor(als, dtype=torch.float64))
    if call == "product":
        return dict(y=y.T.contiguous())
    x1 = _dev(_slid(scs[0], seed).T)
    fe, fg = x1.new_zeros(1), torch.zeros_like(x1)
    x = _dev(scs[0].x.T)
    for s, ee, ty, d, off, w in _active(scs[0], _Rest(scs[0]), x):
        yy = d - off
        lam = -(-2.0 * (yy - w) * torch.log(yy / w) - (yy - w) ** 2 / yy)
        beta = _weights(x, s, ee, ty)
        X = x[s]
        wv = (beta[:, :, None] * (X - X[:, :1])).sum(1)
        nrm = wv / torch.sqrt((wv * wv).sum(1, keepdim=True))
        u = (beta[:, :, None] * (x1[s] - X)).sum(1)
        u = u - (u * nrm).sum(1, keepdim=True) * nrm
        q = torch.sqrt((u * u).sum(1))
        c, stick = MU * lam, q < EPS
        f0 = torch.where(stick, -q ** 3 / (3 * EPS ** 2) + q ** 2 / EPS + EPS / 3, q)
        k1 = torch.where(stick, 2 / EPS - q / EPS ** 2, 1 / q)
        k2 = torch.where(q > 0, torch.where(stick, -1 / (EPS ** 2 * q), -1 / q ** 3), 0.0)
        fe += (c * f0).sum()
        fg.index_add_(0, s.reshape(-1), ((c * k1)[:, None, None] * beta[:, :, None] * u[:, None, :]).reshape(-1, 3))
        r = (beta[:, :, None] * v[s]).sum(1)
        r = c[:, None] * (k1[:, None] * (r - (r * nrm).sum(1, keepdim=True) * nrm) + k2[:, None] * (r * u).sum(1, keepdim=True) * u)
        y.index_add_(0, s.reshape(-1), (beta[:, :, None] * r[:, None, :]).reshape(-1, 3))
    return dict(energy=fe, grad=fg.T.contiguous(), y=y.T.contiguous())


def _weights(x, s, ee, ty):
    """Closest-point weights [m][4] of each pair's type (first primitive's point minus the second's)."""
    X = x[s]
    X = X - X[:, :1]
    out = x.new_zeros(s.shape[0], 4)
    for t, rows in enumerate(_EE if ee else _PT):
        k = ty == t
        if not bool(k.any()):
            continue
        C = x.new_tensor(rows)
        z = torch.einsum("rp,mpi->mri", C, X[k])
        if len(rows) > 1:                               # w minus its part along u (and v)
            A = z[:, 1:]
            G = A @ A.transpose(1, 2)
            co = torch.linalg.solve(G, A @ z[:, 0, :, None])[:, :, 0]
            w = C[0] - co @ C[1:]
        else:
            w = C[0].expand(z.shape[0], 4)
        # the rows of w run either way: first primitive minus second
        out[k] = w * torch.sign(w[:, :2].sum(1, keepdim=True) if ee else w[:, :1])
    return out
