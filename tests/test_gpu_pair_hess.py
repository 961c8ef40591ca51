"""The closed-form projected pair Hessians at their edge cases, against the
oracle: crossing edges whose 2x2 factor has equal or very different singular
values (perpendicular and equal, slanted, nearly parallel, of unequal length),
crossings at the edges' midpoints and triangles under their own centroid
(where rank-one coefficients vanish and the secular equation loses a pole),
gaps from nearly closed to nearly inactive, and points hovering over an edge
from far off its line to almost on it."""
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


def _rods(a, b, xi, dhat):
    pos = np.ascontiguousarray(np.concatenate([a, b], axis=0).T)
    p = np.random.default_rng(5).normal(0.0, 0.001, pos.shape)
    return S.Scene("rod", pos.copy(), pos.copy(), p, xi, dhat, rod_ptr=np.array([0, len(a), len(a) + len(b)], np.int32),
                   name="two_rods")


@pytest.mark.parametrize("gap", [1e-4, 0.02, 0.0499])
@pytest.mark.parametrize("at", [0.5, 0.37])
@pytest.mark.parametrize("degrees,ratio", [(90.0, 1.0), (90.0, 0.2), (60.0, 1.0), (7.0, 1.0), (3.0, 0.5)])
def test_crossing_edges(degrees, ratio, at, gap):
    c, s = math.cos(math.radians(degrees)), math.sin(math.radians(degrees))
    a = np.array([[-at, 0.0, 0.0], [1.0 - at, 0.0, 0.0]])
    b = ratio * np.array([[-at * c, -at * s, 0.0], [(1.0 - at) * c, (1.0 - at) * s, 0.0]]) + [0.0, 0.0, 0.2 + gap]
    sc = _rods(a, b, 0.2, 0.05)
    o = O.contact_pass(sc)
    assert (o.dtype[o.active] == 8).any()
    compare(sc, run_gpu(sc), o)


@pytest.mark.parametrize("gap", [1e-4, 0.02, 0.0499])
@pytest.mark.parametrize("foot", [(1 / 3, 1 / 3), (0.5, 0.25), (0.05, 0.9)])
@pytest.mark.parametrize("apex", [(0.5, math.sqrt(0.75)), (0.0, 1.0), (0.3, 0.1)])
def test_point_over_face(apex, foot, gap):
    t = np.array([[0.0, 0.0, 0.0], [1.0, 0.0, 0.0], [apex[0], apex[1], 0.0]])
    q = t[0] + foot[0] * (t[1] - t[0]) + foot[1] * (t[2] - t[0]) + [0.0, 0.0, 0.2 + gap]
    up = q + np.array([[0.0, 0.0, 0.0], [0.2, 0.1, 3.0], [-0.1, 0.2, 3.0]])
    pos = np.ascontiguousarray(np.concatenate([t, up]).T)
    p = np.random.default_rng(6).normal(0.0, 0.001, pos.shape)
    sc = S.Scene("shell", pos.copy(), pos.copy(), p, 0.2, 0.05, tris=np.array([[0, 3], [1, 4], [2, 5]], np.int32),
                 name="point_over_face")
    o = O.contact_pass(sc)
    assert (o.dtype[o.active] == 6).any()
    compare(sc, run_gpu(sc), o)


@pytest.mark.parametrize("height", [0.2499, 0.21, 0.05, 1e-3, 1e-5])
@pytest.mark.parametrize("at", [0.5, 0.02])
def test_point_over_edge(at, height):
    a = np.array([[0.0, 0.0, 0.0], [1.0, 0.0, 0.0]])
    b = np.array([[at, 0.0, height], [at, 1.0, height + 0.3]])
    sc = _rods(a, b, 0.2, 0.05)
    o = O.contact_pass(sc)
    assert np.isin(o.dtype[o.active], [4, 5, 6, 7]).any()
    compare(sc, run_gpu(sc), o)
