"""Primitives whose boxes reach from -inf to +inf on every axis (a solver that
has run away) against clusters with empty slots: the candidates are those of
the oracle's closed-interval test, and no empty slot is one of them."""
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


def _candidates(sc, x):
    import torch
    from paper_2510_10256_gb300.contact import ContactScene
    cs = ContactScene.from_scene(sc, mode="off")
    cs.contact_build(torch.from_numpy(np.ascontiguousarray(x)).to("cuda:0"))
    got = cs.pairs("candidate")
    cs.close()
    return got


@pytest.mark.parametrize("edges", [1, 3, 33, 70])
@pytest.mark.parametrize("at", [0, -1])
def test_rods(edges, at):
    rng = np.random.default_rng(edges)
    pos = np.cumsum(rng.normal(0.0, 0.1, (3, edges + 1)), axis=1)
    sc = S.Scene("rod", pos, pos, 0.0 * pos, 0.05, 0.01, rod_ptr=np.array([0, edges + 1], np.int32), name="runaway")
    x = pos.copy()
    k = at % edges
    x[:, k], x[:, k + 1] = -np.inf, np.inf
    assert np.array_equal(_candidates(sc, x), O.broad_phase(O.topology(sc), x, 0.5 * sc.activation))


@pytest.mark.parametrize("nx", [2, 5, 9])
def test_shells(nx):
    sc = S.flat_grid(nx=nx)
    x = sc.x.copy()
    t = np.asarray(sc.tris)[:, -1]
    x[:, t[0]], x[:, t[1]] = -np.inf, np.inf
    assert np.array_equal(_candidates(sc, x), O.broad_phase(O.topology(sc), x, 0.5 * sc.activation))
