"""Distances whose type FP32 decides, against the oracle where it is hard to
decide: pairs of rods and of triangles on a small integer lattice (parallel
and crossing edges, ends over ends, points over vertices, edges and faces),
exactly tied, and shifted off the ties by amounts around FP32's and FP64's
resolution.  The pairs stand far apart, so every candidate is one pair's own;
distances and types must be the FP64 routine's, bit for bit."""
import numpy as np
import pytest

import oracle as O
from paper_2510_10256_gb300 import scenes as S
from tests.parity import run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_10256_gb300 import contact
    contact.build()
    contact.lib()


def _far_enough(x, verts):
    """No stencil of the two primitives is closer than 0.3 or further than 3."""
    a, b = x[:verts], x[verts:]
    edge = [(i, (i + 1) % verts) for i in range(verts if verts == 3 else 1)]
    st = [(True, np.concatenate([a[list(e)], b[list(f)]])) for e in edge for f in edge]
    if verts == 3:
        st += [(False, np.concatenate([p[i:i + 1], q])) for p, q in ((a, b), (b, a)) for i in range(3)]
    return all(0.3 < O.distance(ee, s.reshape(-1))[0] < 3.0 for ee, s in st)


def _lattice_pairs(rng, count, verts, shift):
    """count pairs of rods (verts 2) or triangles (verts 3), 40 apart."""
    out = []
    while len(out) < count:
        x = rng.integers(-2, 3, size=(2 * verts, 3)).astype(float)
        if verts == 3:
            n = [np.cross(t[1] - t[0], t[2] - t[0]) for t in (x[:3], x[3:])]
            if not all(np.any(v) for v in n):
                continue
        elif not all(np.any(e[1] - e[0]) for e in (x[:2], x[2:])):
            continue
        x += shift * rng.normal(size=x.shape)
        if _far_enough(x, verts):
            out.append(x + 40.0 * np.array([len(out) % 8, len(out) // 8 % 8, len(out) // 64]))
    return np.concatenate(out)


@pytest.mark.parametrize("shift", [0.0, 1e-13, 1e-8, 1e-7, 1e-6, 1e-4])
@pytest.mark.parametrize("verts,count", [(2, 1), (2, 300), (3, 1), (3, 200)])
def test_types_and_distances_equal_the_fp64_routine(verts, count, shift):
    pos = np.ascontiguousarray(_lattice_pairs(np.random.default_rng(40 * count + verts), count, verts, shift).T)
    p = np.zeros_like(pos)
    kw = dict(rod_ptr=np.arange(0, 4 * count + 1, 2, dtype=np.int32)) if verts == 2 else dict(
        tris=np.arange(6 * count, dtype=np.int32).reshape(-1, 3).T.copy())
    sc = S.Scene("rod" if verts == 2 else "shell", pos.copy(), pos.copy(), p, 0.2, 3.0, name="lattice_pairs", **kw)
    o = O.contact_pass(sc)
    g = run_gpu(sc)
    assert np.array_equal(g["C"], o.C)
    k = np.searchsorted(o.C, g["A"]["keys"])
    assert np.array_equal(np.sort(g["A"]["keys"]), np.sort(o.active_keys)) and g["A"]["keys"].size >= count
    assert np.array_equal(g["A"]["dtype"], o.dtype[k])
    assert np.array_equal(g["A"]["d"], o.d[k])
