"""The step bound when many pairs tie for the minimum, so that the FP64
iteration's list is as long as the input: lengths around the change from half
a warp per pair to one lane per pair, through both entry points, against the
oracle's iteration of the one pair that is repeated."""
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


# dyadic coordinates: shifting them by whole numbers changes no difference
PAIR = {
    True: (np.array([[-1.0, 0.125, 0.0], [1.0, 0.0, 0.0], [0.25, -1.0, 1.5], [0.0, 1.0, 1.25]]),
           np.array([[1.0, 0.125, 1.0], [1.0, 0.5, 1.0], [0.0, -1.0, -0.75], [0.25, 0.0, -0.75]])),
    False: (np.array([[0.25, 0.125, 1.5], [-1.0, -1.0, 0.0], [1.0, -1.0, 0.25], [0.0, 1.5, 0.0]]),
            np.array([[0.5, 0.125, -1.0], [0.0, -1.5, 1.0], [0.0, 0.0, 0.75], [0.25, 0.0, 0.75]])),
}


@pytest.mark.parametrize("count", [4800, 4865, 40000])
@pytest.mark.parametrize("kinds", [(True,), (False,), (True, False)])
def test_tied_stencils(kinds, count):
    import torch
    from paper_2510_10256_gb300 import contact
    dev = torch.device("cuda:0")
    ee = np.array([kinds[i % len(kinds)] for i in range(count)])
    x = np.concatenate([PAIR[bool(e)][0] for e in ee])
    p = np.concatenate([PAIR[bool(e)][1] for e in ee])
    want = min(O.accd(e, PAIR[e][0].reshape(-1), PAIR[e][1].reshape(-1), 0.0625)[0] for e in kinds)
    assert 0.0 < want < 1.0
    ids = np.arange(4 * count, dtype=np.int32).reshape(-1, 4)
    alpha = torch.full((1,), -7.0, dtype=torch.float64, device=dev)
    flags = torch.full((1,), -1, dtype=torch.int32, device=dev)

    def on(a):
        return torch.from_numpy(np.ascontiguousarray(a)).to(dev)

    contact.ccd_step_noalloc(on(x.T), on(p.T), on(ids), on(ee.astype(np.uint8)), on(np.full(count, 0.0625)), alpha, flags)
    assert int(flags.item()) == 0
    assert float(alpha.item()) == want


@pytest.mark.parametrize("count", [4800, 12000])
def test_tied_rods(count):
    import torch
    from paper_2510_10256_gb300.contact import ContactScene
    dev = torch.device("cuda:0")
    at = 64.0 * np.stack([np.arange(count) % 32, np.arange(count) // 32 % 32, np.arange(count) // 1024], 1)
    pos = np.ascontiguousarray((PAIR[True][0][None] + at[:, None]).reshape(-1, 3).T)
    p = np.ascontiguousarray(np.tile(PAIR[True][1], (count, 1)).T)
    sc = S.Scene("rod", pos.copy(), pos.copy(), p, 0.0625, 0.125,
                 rod_ptr=np.arange(0, 4 * count + 1, 2, dtype=np.int32), name="tied_rods")
    one = S.Scene("rod", pos[:, :4].copy(), pos[:, :4].copy(), p[:, :4].copy(), 0.0625, 0.125,
                  rod_ptr=np.array([0, 2, 4], np.int32), name="tied_rods_one")
    want = O.contact_pass(one).alpha
    assert 0.0 < want < 1.0
    cs = ContactScene.from_scene(sc)
    alpha = torch.zeros(1, dtype=torch.float64, device=dev)
    x, pp = torch.from_numpy(pos).to(dev), torch.from_numpy(p).to(dev)
    cs.contact_build(x)
    cs.contact_filter()
    cs.ccd_step(x, pp, alpha)
    assert cs.sync_status() == 0
    assert float(alpha.item()) == want
    cs.close()
