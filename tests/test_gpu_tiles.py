"""The cluster broad phase against the oracle's brute force at the sizes where
it can go wrong: primitive counts around a cluster of 32 and a supercluster of
1,024, positions that ignore the rest order the clusters come from (scattered,
all in one place, far apart), a thickness from none to everything overlapping,
members of very different sizes in one batch, and a pass after a far larger
one on the same scene (lists kept, lists grown)."""
import numpy as np
import pytest

import oracle as O
from paper_2510_10256_gb300 import scenes as S

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


def _rods(edges, seed):
    rng = np.random.default_rng(seed)
    n = edges + 1
    pos = np.cumsum(rng.normal(0.0, 0.1, (3, n)), axis=1)
    return S.Scene("rod", pos.copy(), pos.copy(), rng.normal(0.0, 0.02, pos.shape), 0.05, 0.01,
                   rod_ptr=np.array([0, n], np.int32), name=f"rod{edges}")


def _shell(tris, seed):
    rng = np.random.default_rng(seed)
    n = max(4, tris // 2 + 2)
    t = np.array([rng.choice(n, 3, replace=False) for _ in range(tris)], np.int32).T.copy()
    pos = rng.uniform(0.0, 1.0, (3, n))
    return S.Scene("shell", pos.copy(), pos.copy(), rng.normal(0.0, 0.05, pos.shape), 0.02, 0.01, tris=t, name=f"soup{tris}")


def _check(cs, sc, x, p):
    topo = O.topology(sc)
    cs.contact_build(_dev(x))
    cs.ccd_step(_dev(x), _dev(p))
    assert np.array_equal(cs.pairs("candidate"), O.broad_phase(topo, x, 0.5 * sc.activation))
    assert np.array_equal(cs.pairs("ccd"), O.broad_phase(topo, x, 0.5 * sc.thickness, p))


@pytest.mark.parametrize("edges", [1, 2, 31, 32, 33, 64, 65, 1023, 1024, 1025, 2100])
def test_rods(edges):
    from paper_2510_10256_gb300.contact import ContactScene
    sc = _rods(edges, edges)
    rng = np.random.default_rng(edges)
    cs = ContactScene.from_scene(sc)
    for x in (sc.x, rng.permuted(sc.x, axis=1), 1e-3 * sc.x, 50.0 * sc.x, sc.x):
        _check(cs, sc, x, sc.p)
    cs.close()


@pytest.mark.parametrize("tris", [1, 31, 32, 33, 97, 350, 700])
def test_shells(tris):
    from paper_2510_10256_gb300.contact import ContactScene
    sc = _shell(tris, tris)
    rng = np.random.default_rng(tris)
    cs = ContactScene.from_scene(sc, mode="off")   # a soup may hold stencils at zero reference distance
    for x in (sc.x, rng.permuted(sc.x, axis=1), 20.0 * sc.x, 0.05 * sc.x + 3.0, sc.x):
        _check(cs, sc, x, sc.p)
    cs.close()


def test_batch_members_of_all_sizes():
    from paper_2510_10256_gb300.contact import ContactBatch, ContactScene
    scs = [_rods(e, 7 + e) for e in (1, 33, 1100, 32, 5)]
    ms = [ContactScene.from_scene(sc) for sc in scs]
    b = ContactBatch(ms)
    x, p = (np.concatenate([getattr(sc, k) for sc in scs], axis=1) for k in ("x", "p"))
    b.contact_build(_dev(x))
    keys = b.pairs("candidate")
    for m, sc in enumerate(scs):
        own = b.to_member_keys(keys[b.member_of_keys(keys) == m], m)
        assert np.array_equal(np.sort(own), O.broad_phase(O.topology(sc), sc.x, 0.5 * sc.activation))
    assert p.shape == x.shape
    b.close()
    for m in ms:
        m.close()
