"""Clusters and components: scenes of many components whose order, sizes or
rest places say little about where they lie -- shuffled fibres around a
cluster's 32 edges, instances of one sheet, confetti whose rest shapes lie
elsewhere -- against the oracle, and with memory (the list of overlapping
clusters is part of it) close to that of the same scene in good order."""
import numpy as np
import pytest

import oracle as O
from paper_2510_10256_gb300 import scenes as S
from tests.parity import compare, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_10256_gb300 import contact
    contact.build()
    contact.lib()


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


def _fibres(edges, box, seed, order="random", rest="own"):
    """Straight jittered polylines of edges[k] segments of 0.1 in a cube."""
    rng = np.random.default_rng(seed)
    m = len(edges)
    org, d = rng.uniform(0.0, box, (m, 3)), rng.normal(size=(m, 3))
    d /= np.linalg.norm(d, axis=1)[:, None]
    polys = [o + np.arange(e + 1)[:, None] * 0.1 * t + rng.normal(0.0, 0.01, (e + 1, 3)) for o, t, e in zip(org, d, edges)]
    if order == "slabs":  # by place: thin slabs, snaking through them
        cell = box / 12
        c = [np.floor(q.mean(0) / cell).astype(int) for q in polys]
        polys = [polys[k] for k in sorted(range(m), key=lambda k: (c[k][0], c[k][1] if c[k][0] % 2 else -c[k][1], polys[k].mean(0)[2]))]
    pos = np.ascontiguousarray(np.concatenate(polys).T)
    ptr = np.concatenate([[0], np.cumsum([len(q) for q in polys])]).astype(np.int32)
    if rest == "own":
        r = pos.copy()
    else:  # every rest shape straight from the origin
        r = np.zeros_like(pos)
        r[0] = np.concatenate([0.1 * np.arange(len(q)) for q in polys])
    p = rng.normal(0.0, 0.01, pos.shape)
    return S.Scene("rod", r, pos, p, 0.05, 0.01, rod_ptr=ptr, name="fibres")


def _confetti(m, side, box, seed, scramble):
    """Small square sheets at random places; scramble: their rest shapes at each other's places."""
    rng = np.random.default_rng(seed)
    r0, t0 = S.grid_mesh(side, side, 0.05)
    place = rng.uniform(0.0, box, (m, 3))
    other = place[rng.permutation(m)] if scramble else place
    rest = np.concatenate([r0 + o[:, None] for o in other], axis=1)
    x = np.concatenate([r0 + o[:, None] for o in place], axis=1)
    x += rng.normal(0.0, 0.004, x.shape)
    t = np.concatenate([t0 + k * r0.shape[1] for k in range(m)], axis=1).astype(np.int32)
    return S.Scene("shell", rest, x, rng.normal(0.0, 0.01, x.shape), 0.05, 0.01, tris=t, name="confetti")


def _bytes(sc, builds=1):
    from paper_2510_10256_gb300.contact import ContactScene
    cs = ContactScene.from_scene(sc)
    for _ in range(builds):
        cs.contact_build(_dev(sc.x))
    b, n = cs.stats()["device_bytes"], cs.stats()["n_candidates"]
    cs.close()
    return b, n


# ------------------------------------------------------------------- results

@pytest.mark.parametrize("edges", [(1,), (8,), (23,), (24,), (31,), (33,), (40,), (48,), (65,), (97,), (1, 40, 8, 129, 24)])
@pytest.mark.parametrize("rest", ["own", "shared"])
def test_fibres(edges, rest):
    m = 4000 // sum(edges) + 3
    sc = _fibres([edges[k % len(edges)] for k in range(m)], 2.5, sum(edges), rest=rest)
    rep = compare(sc, run_gpu(sc), O.contact_pass(sc))
    assert rep["C"] > 0


@pytest.mark.parametrize("rest", ["own", "shared"])
def test_many_short_fibres(rest):
    sc = _fibres([8] * 3000, 8.0, 3, rest=rest)   # 750 clusters: out of order nearly all meet
    rep = compare(sc, run_gpu(sc), O.contact_pass(sc))
    assert rep["active"] > 0


@pytest.mark.parametrize("scramble", [False, True])
def test_confetti(scramble):
    sc = _confetti(800, 3, 4.3, 11, scramble)     # classes by the masks of the clusters' new order
    rep = compare(sc, run_gpu(sc), O.contact_pass(sc))
    assert rep["F"] > 0 and rep["active"] > 0


def test_instances_of_one_sheet():
    one = S.pleated_sheet(seed=3, nx=9)
    n, off = one.n, 6.0 * np.arange(5)
    x = np.concatenate([one.x + np.array([[o], [0.0], [0.0]]) for o in off], axis=1)
    rest = np.concatenate([one.rest] * 5, axis=1)
    t = np.concatenate([np.asarray(one.tris) + n * k for k in range(5)], axis=1).astype(np.int32)
    sc = S.Scene("shell", rest, x, np.tile(one.p, (1, 5)), one.thickness, one.dhat, tris=t, name="instances")
    compare(sc, run_gpu(sc), O.contact_pass(sc))


@pytest.mark.parametrize("kind", ["rod", "shell"])
def test_batch_and_moves(kind):
    """Members of every kind of order; then a call with the components somewhere else entirely, and back."""
    from paper_2510_10256_gb300.contact import ContactBatch, ContactScene
    if kind == "rod":
        scs = [_fibres([8] * 900, 5.0, 1, rest="shared"), _fibres([33] * 20, 1.5, 2), _fibres([64, 1, 96], 1.0, 3)]
    else:
        scs = [_confetti(800, 3, 4.3, 1, True), S.tiny_shell(5, nx=7), _confetti(40, 2, 1.0, 2, False)]
    ms = [ContactScene.from_scene(sc) for sc in scs]
    ms[0].contact_build(_dev(scs[0].x))  # a member with an order of its own
    b = ContactBatch(ms)
    rng = np.random.default_rng(8)
    for turn in range(3):
        xs = []
        for sc in scs:
            x = sc.x.copy()
            if turn == 1:  # every component moved by itself
                c = O.topology(sc).comp
                x += rng.uniform(-3.0, 3.0, (3, int(c.max()) + 1))[:, c]
            xs.append(x)
        x, p = np.concatenate(xs, axis=1), np.concatenate([sc.p for sc in scs], axis=1)
        b.contact_build(_dev(x))
        b.contact_filter()
        b.ccd_step(_dev(x), _dev(p))
        keys, filt, ccd = b.pairs("candidate"), b.pairs("filtered"), b.pairs("ccd")
        for m, sc in enumerate(scs):
            topo = O.topology(sc)
            want = O.broad_phase(topo, xs[m], 0.5 * sc.activation)
            own = b.to_member_keys(keys[b.member_of_keys(keys) == m], m)
            assert np.array_equal(np.sort(own), want)
            swept = b.to_member_keys(ccd[b.member_of_keys(ccd) == m], m)
            assert np.array_equal(np.sort(swept), O.broad_phase(topo, xs[m], 0.5 * sc.thickness, sc.p))
            f = b.to_member_keys(filt[b.member_of_keys(filt) == m], m)
            if sc.kind == "shell":
                assert np.array_equal(np.sort(f), np.intersect1d(want, O.rest_filter(sc, topo, sc.activation)[0]))
    b.close()
    for m in ms:
        m.close()


# ------------------------------------------------------------ the list's size

@pytest.mark.parametrize("edges", [31, 8])
@pytest.mark.parametrize("rest", ["own", "shared"])
def test_shuffled_fibres_take_no_more_than_sorted_ones(edges, rest):
    m = 20_000
    box = 20.0 * (m * edges / 620_000) ** (1 / 3)
    good, n_good = _bytes(_fibres([edges] * m, box, 5, order="slabs"))
    bad, n_bad = _bytes(_fibres([edges] * m, box, 5, rest=rest))
    assert n_bad == n_good
    assert bad <= 1.25 * good, (bad, good)


def test_instances_take_no_more_than_sheets_of_their_own():
    """... in the swept broad phase: at rest they do lie in one place, and so do their clusters there."""
    from paper_2510_10256_gb300.contact import ContactScene
    one = S.pleated_sheet(seed=3, nx=20)
    n, off = one.n, 60.0 * np.arange(24)
    x = np.concatenate([one.x + np.array([[o], [0.0], [0.0]]) for o in off], axis=1)
    own = np.concatenate([one.rest + np.array([[o], [0.0], [0.0]]) for o in off], axis=1)
    t = np.concatenate([np.asarray(one.tris) + n * k for k in range(24)], axis=1).astype(np.int32)
    p = np.tile(one.p, (1, 24))
    grown, pairs = [], []
    for rest in (own, np.concatenate([one.rest] * 24, axis=1)):
        cs = ContactScene.from_scene(S.Scene("shell", rest, x, p, one.thickness, one.dhat, tris=t, name="instances"))
        before = cs.stats()["device_bytes"]
        cs.ccd_step(_dev(x), _dev(p))
        grown.append(cs.stats()["device_bytes"] - before)
        pairs.append(cs.stats()["n_ccd"])
        cs.close()
    assert pairs[0] == pairs[1]
    assert grown[1] <= 1.25 * grown[0], grown
