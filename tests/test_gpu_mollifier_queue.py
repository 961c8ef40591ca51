"""The queue of mollified pairs among many more active ones: both forms of its
projection against the oracle, on either side of the length where they change,
and its memory, which follows the mollified pairs and not the active ones."""
import math

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


def _sticks(moll, plain):
    """Isolated crossings of two sticks: the first `moll` nearly parallel (below the threshold), the others not."""
    rng = np.random.default_rng(moll + 7 * plain)
    pts = []
    for k in range(moll + plain):
        th = rng.uniform(0.002, 0.025) if k < moll else rng.uniform(0.3, 1.5)
        c, s, sh = math.cos(th), math.sin(th), rng.uniform(-0.3, 0.3)
        o = np.array([4.0 * (k % 60), 4.0 * (k // 60 % 60), 4.0 * (k // 3600)])
        h = 0.31 + 0.03 * rng.random()
        pts += [o + [-0.5, 0, 0], o + [0.5, 0, 0], o + [-0.5 * c + sh, -0.5 * s, h], o + [0.5 * c + sh, 0.5 * s, h]]
    x = np.ascontiguousarray(np.array(pts).T)
    p = rng.normal(0.0, 0.01, x.shape)
    return S.Scene("rod", x.copy(), x, p, 0.3, 0.05, rod_ptr=np.arange(0, x.shape[1] + 1, 2, dtype=np.int32))


@pytest.mark.parametrize("moll,plain", [(0, 40), (1, 5000), (33, 5000), (300, 5000), (4095, 600), (4097, 600)])
def test_queue_among_many_active_pairs(moll, plain):
    sc = _sticks(moll, plain)
    g = run_gpu(sc, mollifier=True)
    rep = compare(sc, g, O.contact_pass(sc, mollifier=True))
    assert rep["active"] == moll + plain and g["stats"]["n_mollified"] == moll


def test_memory_follows_the_mollified_pairs():
    import torch
    from paper_2510_10256_gb300.contact import ContactScene
    sc = _sticks(50, 20_000)
    held = {}
    for on in (False, True):
        cs = ContactScene.from_scene(sc, mollifier=on)
        e = torch.zeros(1, dtype=torch.float64, device="cuda:0")
        g = torch.zeros(3, sc.n, dtype=torch.float64, device="cuda:0")
        x = torch.from_numpy(sc.x).to("cuda:0")
        cs.contact_build(x)
        cs.contact_filter()
        cs.barrier_eval(x, e, g)
        held[on] = cs.stats()["device_bytes"]
        n = cs.stats()["n_candidates"]
        cs.close()
    # the list of mollified candidates has room for every candidate, the matrices (360 bytes) for the listed ones
    assert held[True] - held[False] <= 5 * n + 450 * 50 + 1024
