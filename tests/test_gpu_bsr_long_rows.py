"""BSR rows with many columns, against the oracle: a hub edge crossing enough
needles that its vertices' buckets lie around a block's shared memory and well
past it (the columns of a run of 256 pairs are distinct, the hub's own repeat
in every run), several such hubs at once, and a sheet lying on two triangles."""
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


def _hubs(needles):
    """Hub k, at height k, crosses needles[k] needles in two rows above and below it."""
    rng = np.random.default_rng(sum(needles))
    polys = []
    for k, m in enumerate(needles):
        polys.append(np.array([[-1.0, 0.0, 2.0 * k], [0.25 * m + 1.0, 0.0, 2.0 * k]]))
        for j in range(m):
            x, t = 0.5 * (j // 2), (0.21 + 0.03 * rng.random()) * (-1) ** j
            polys.append(np.array([[x, -0.9, 2.0 * k + t], [x + 0.1 * rng.random(), 1.1, 2.0 * k + t]]))
    pos = np.ascontiguousarray(np.concatenate(polys).T)
    p = np.random.default_rng(9).normal(0.0, 0.001, pos.shape)
    rp = np.arange(0, pos.shape[1] + 1, 2, dtype=np.int32)
    return S.Scene("rod", pos.copy(), pos.copy(), p, 0.2, 0.05, rod_ptr=rp, name="hubs")


# a hub vertex's bucket: two entries a needle, and its edge's two in every run
@pytest.mark.parametrize("needles", [(4000,), (8100,), (8200,), (12000,), (300, 9000, 700, 9100, 8800)])
def test_hubs(needles):
    sc = _hubs(needles)
    rep = compare(sc, run_gpu(sc), O.contact_pass(sc))
    assert rep["active"] >= sum(needles) and rep["nnzb"] >= 8 * sum(needles)


def _sheet_on_two_triangles(nx):
    rng = np.random.default_rng(nx)
    r, t = S.grid_mesh(nx, nx, 0.5)
    r = r - r.min(axis=1, keepdims=True)
    w = r.max() + 1.0
    floor = np.array([[-1.0, w, -1.0, w], [-1.0, -1.0, w, w], [0.0] * 4])
    x = np.concatenate([floor, r + np.array([[0.0], [0.0], [0.22]])], axis=1)
    x[2, 4:] += rng.uniform(-0.015, 0.015, r.shape[1])
    tris = np.concatenate([np.array([[0, 1], [1, 3], [2, 2]]), t + 4], axis=1).astype(np.int32)
    p = rng.normal(0.0, 1e-4, x.shape)
    return S.Scene("shell", x.copy(), x, p, 0.2, 0.05, tris=tris, name="floor")


def test_sheet_on_two_triangles():
    sc = _sheet_on_two_triangles(140)  # 19,600 vertices over the floor's four
    rep = compare(sc, run_gpu(sc), O.contact_pass(sc))
    assert rep["active"] >= 19_600


def _pattern_ms(sc):
    """Barrier stage without its Hessian kernel, the middle of seven."""
    import torch
    from paper_2510_10256_gb300.contact import ContactScene
    cs = ContactScene.from_scene(sc)
    x = torch.from_numpy(np.ascontiguousarray(sc.x)).to("cuda:0")
    e = torch.zeros(1, dtype=torch.float64, device="cuda:0")
    g = torch.zeros(3, sc.n, dtype=torch.float64, device="cuda:0")
    cs.set_timing(True)
    ms = []
    for _ in range(7):
        cs.contact_build(x)
        cs.contact_filter()
        cs.barrier_eval(x, e, g)
        t = cs.stage_ms()
        ms.append(t[2] - t[4])
    assert cs.stats()["n_active"] == sc.n // 2 - sc.meta["hubs"]
    cs.close()
    return sorted(ms)[3]


def test_time_is_set_by_the_keys_not_by_the_longest_row():
    """The same 60,000 crossings on one hub and on 60.  (With each row sorted by one block it took 76 times as long
    on the one hub; the bound leaves room for a busy machine.)"""
    one, many = _hubs((60_000,)), _hubs((1_000,) * 60)
    one.meta["hubs"], many.meta["hubs"] = 1, 60
    assert _pattern_ms(one) <= 6.0 * _pattern_ms(many)
