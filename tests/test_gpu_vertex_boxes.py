"""Primitive boxes formed from vertex boxes, as large scenes have them: primitive
counts on both sides of the change (1,216 clusters of 32 on 152 SMs), moves of
either sign, none and negative zero; the static and the swept candidate sets
against the oracle."""
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


def _rods(edges, rng):
    pos = np.cumsum(rng.normal(0.0, 0.1, (3, edges + 1)), axis=1) + np.array([[500.0], [-3.0], [0.0]])
    p = rng.normal(0.0, 0.02, pos.shape)
    p[:, ::3] = 0.0
    p[:, 1::9] = -0.0
    return S.Scene("rod", pos.copy(), pos, p, 0.05, 0.01, rod_ptr=np.array([0, edges + 1], np.int32), name="long_rod")


def _shell(tris, rng):
    c = rng.normal(0.0, 6.0, (tris, 1, 3))
    pos = np.ascontiguousarray((c + rng.normal(0.0, 0.2, (tris, 3, 3))).reshape(-1, 3).T)
    p = rng.normal(0.0, 0.05, pos.shape)
    p[:, ::3] = -0.0
    return S.Scene("shell", pos.copy(), pos, p, 0.05, 0.01, tris=np.arange(3 * tris, dtype=np.int32).reshape(-1, 3).T.copy(),
                   name="loose_triangles")


@pytest.mark.parametrize("kind,count", [("rod", 38880), ("rod", 38913), ("rod", 60001), ("shell", 5400), ("shell", 5600)])
def test_candidates_equal_the_oracle(kind, count):
    import torch
    from paper_2510_10256_gb300.contact import ContactScene
    sc = (_rods if kind == "rod" else _shell)(count, np.random.default_rng(count))
    o = O.contact_pass(sc)
    dev = torch.device("cuda:0")
    cs = ContactScene.from_scene(sc)
    x, p = torch.from_numpy(np.ascontiguousarray(sc.x)).to(dev), torch.from_numpy(np.ascontiguousarray(sc.p)).to(dev)
    alpha = torch.zeros(1, dtype=torch.float64, device=dev)
    cs.contact_build(x)
    cs.contact_filter()
    cs.ccd_step(x, p, alpha)
    assert np.array_equal(cs.pairs("candidate"), o.C)
    assert np.array_equal(np.sort(cs.ccd()["keys"]), np.sort(o.ccd_keys))
    assert float(alpha.item()) == o.alpha
    cs.close()
