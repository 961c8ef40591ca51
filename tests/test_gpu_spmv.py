"""The BSR product with its rows split over 4, 8, 16 and 32 lanes: row counts
on both sides of the changes (152 SMs) and around a block's edge, rows empty,
short and long, with and without the shift, against the scene's own matrix
multiplied on the CPU."""
import numpy as np
import pytest

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


def _bundles(n, rng):
    """n vertices in straight rods of two; every 50th group of 2 to 60 rods is a bundle in contact, the rest lie apart."""
    rods = n // 2
    start = np.zeros((rods, 3))
    i = group = 0
    while i < rods:
        m = min(rods - i, int(rng.integers(2, 61)) if group % 50 == 0 else 40)
        at = 100.0 * np.array([group % 64, group // 64 % 64, group // 4096])
        if group % 50 == 0:
            start[i:i + m] = at + np.stack([0 * np.arange(m), 0.22 * (np.arange(m) % 8), 0.22 * (np.arange(m) // 8)], 1)
        else:
            start[i:i + m] = at + np.stack([0 * np.arange(m), 2.0 * np.arange(m), 0 * np.arange(m)], 1)
        i += m
        group += 1
    pos = np.repeat(start, 2, 0)
    pos[1::2, 0] += 1.0 + 0.1 * rng.random(rods)
    return np.ascontiguousarray(pos.T)


@pytest.mark.parametrize("n", [4, 256, 9726, 9728, 19454, 19456, 38910, 38912, 38914])
@pytest.mark.parametrize("shift", [0.0, 4.0])
def test_product_equals_the_matrix(n, shift):
    import torch
    from paper_2510_10256_gb300.contact import ContactScene
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(n)
    pos = _bundles(n, rng)
    sc = S.Scene("rod", pos, pos.copy(), np.zeros_like(pos), 0.2, 0.05,
                 rod_ptr=np.arange(0, n + 1, 2, dtype=np.int32), name="bundles")
    cs = ContactScene.from_scene(sc)
    x = torch.from_numpy(pos).to(dev)
    energy, grad = torch.zeros(1, dtype=torch.float64, device=dev), torch.zeros(3, n, dtype=torch.float64, device=dev)
    cs.contact_build(x)
    cs.contact_filter()
    cs.barrier_eval(x, energy, grad)
    v = rng.normal(size=(3, n))
    y = torch.full((3, n), np.nan, dtype=torch.float64, device=dev)
    cs.bsr_spmv(torch.from_numpy(v).to(dev), y, shift)
    row, col, val = cs.bsr()
    assert col.size > n // 60
    val = val.reshape(-1, 3, 3)
    rows = np.repeat(np.arange(n), np.diff(row))
    want, mag = shift * v, np.abs(shift * v)
    for i in range(3):
        np.add.at(want[i], rows, np.einsum("kj,jk->k", val[:, i], v[:, col]))
        np.add.at(mag[i], rows, np.einsum("kj,jk->k", np.abs(val[:, i]), np.abs(v[:, col])))
    assert np.all(np.abs(y.cpu().numpy() - want) <= 1e-13 * mag)
    cs.close()
