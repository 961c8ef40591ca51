"""The BSR pattern at the edges of its stages, against the oracle: rows whose
buckets fit a warp's registers, its shared memory, or only global memory (one
edge crossing 3 to 700 needles), runs of active pairs that share no vertex at
all (isolated crossings, more than a run's local numbering holds), and counts
around a run of 256 pairs."""
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


def _rods(polys, xi=0.2, dhat=0.05):
    pos = np.ascontiguousarray(np.concatenate(polys, axis=0).T)
    p = np.random.default_rng(9).normal(0.0, 0.001, pos.shape)
    rp = np.concatenate([[0], np.cumsum([len(q) for q in polys])]).astype(np.int32)
    return S.Scene("rod", pos.copy(), pos.copy(), p, xi, dhat, rod_ptr=rp, name="rods")


@pytest.mark.parametrize("needles", [3, 8, 30, 120, 260, 700])
def test_one_edge_across_many(needles):
    hub = np.array([[-1.0, 0.0, 0.0], [0.5 * needles, 0.0, 0.0]])
    rng = np.random.default_rng(needles)
    polys = [hub]
    for k in range(needles):
        x, t = 0.5 * k, 0.21 + 0.03 * rng.random()
        polys.append(np.array([[x, -0.9, t], [x + 0.1 * rng.random(), 1.1, t]]))
    sc = _rods(polys)
    rep = compare(sc, run_gpu(sc), O.contact_pass(sc))
    assert rep["active"] >= needles and rep["nnzb"] >= 4 * needles


@pytest.mark.parametrize("crossings", [1, 128, 255, 256, 257, 300, 530])
def test_isolated_crossings(crossings):
    rng = np.random.default_rng(crossings)
    polys = []
    for k in range(crossings):
        c = np.array([3.0 * (k % 20), 3.0 * (k // 20), 0.0])
        h = np.array([0.0, 0.0, 0.21 + 0.03 * rng.random()])
        polys.append(c + np.array([[-0.5, 0.0, 0.0], [0.6, 0.1, 0.0]]))
        polys.append(c + h + np.array([[0.0, -0.6, 0.0], [0.1, 0.5, 0.0]]))
    sc = _rods(polys)
    rep = compare(sc, run_gpu(sc), O.contact_pass(sc))
    assert rep["active"] == crossings and rep["nnzb"] == 16 * crossings
