"""The FP32 brackets of the additive-CCD times: the step bound must be the
FP64 iteration's own minimum, bit for bit, whatever the brackets drop.  Lists
of random stencils (gaps from a touch to far, head-on and grazing motions,
offsets from 0 to nearly the distance, edges nearly parallel, triangles nearly
flat, tiny and large scales), of lengths around the block and sample sizes,
against the oracle's iteration stencil by stencil."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_10256_gb300 import contact
    contact.build()
    contact.lib()


def _stencil(rng, ee, scale, thin):
    a, b = rng.normal(size=3), rng.normal(size=3)
    n = np.cross(a, b)
    n /= np.linalg.norm(n)
    if ee:
        b = a + thin * b if rng.random() < 0.5 else b   # nearly parallel
        s, t = rng.uniform(-0.3, 1.3, 2)
        x = np.array([np.zeros(3), a, s * a - t * b, s * a - t * b + b])
        x[2:] += 10.0 ** rng.uniform(-4, 0.5) * n
    else:
        b = a + thin * b if rng.random() < 0.5 else b   # nearly flat
        s, t = rng.uniform(-0.3, 1.0, 2)
        x = np.array([s * a + t * b + 10.0 ** rng.uniform(-4, 0.5) * n, np.zeros(3), a, b])
    p = rng.normal(size=(4, 3)) * 10.0 ** rng.uniform(-3, 1)
    if rng.random() < 0.4:   # head-on
        p = np.where(np.arange(4)[:, None] < (2 if ee else 1), 1.0, -1.0) * -n * (1 if ee else -1) * rng.uniform(0.1, 3) + 1e-3 * p
    shift = rng.normal(size=3) * rng.choice([0.0, 1.0, 300.0])
    return x * scale + shift * scale, p * scale


@pytest.mark.parametrize("scale", [1e-3, 1.0, 1e3])
@pytest.mark.parametrize("count", [1, 2, 15, 16, 17, 129, 700])
def test_step_bound_equals_the_full_iteration(count, scale):
    import torch
    from paper_2510_10256_gb300 import contact
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(1000 * count + int(1e3 * scale))
    for rep in range(12 if count < 100 else 4):
        xs, ps, ee, off, t = [], [], [], [], []
        while len(t) < count:
            e = bool(rng.random() < 0.5)
            x, p = _stencil(rng, e, scale, 10.0 ** rng.uniform(-6, -1))
            d = O.distance(e, x.reshape(-1))[0]
            o = 0.0 if rng.random() < 0.3 else d * (1.0 - 10.0 ** rng.uniform(-5, -0.05))
            r = O.accd(e, x.reshape(-1), p.reshape(-1), o)
            if r[1] != 0:
                continue   # penetrating, or at the iteration limit
            xs.append(x)
            ps.append(p)
            ee.append(e)
            off.append(o)
            t.append(r[0])
        x, p = np.concatenate(xs), np.concatenate(ps)
        ids = np.arange(4 * count, dtype=np.int32).reshape(-1, 4)
        alpha = torch.full((1,), -7.0, dtype=torch.float64, device=dev)
        flags = torch.full((1,), -1, dtype=torch.int32, device=dev)

        def on(a):
            return torch.from_numpy(np.ascontiguousarray(a)).to(dev)

        contact.ccd_step_noalloc(on(x.T), on(p.T), on(ids), on(np.array(ee, np.uint8)), on(np.array(off)), alpha, flags)
        assert int(flags.item()) == 0
        assert float(alpha.item()) == min(1.0, min(t)), (rep, float(alpha.item()), min(t))
