"""Candidates are numbered in 32 bits: a call with more is refused, also when
the list an earlier call grew (25 % headroom) has room for them."""
import numpy as np
import pytest

from paper_2510_10256_gb300 import scenes as S

pytestmark = pytest.mark.gpu

TOO_LARGE = 8


def test_more_pairs_than_32_bits_number():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.mem_get_info()[0] < 90e9:
        pytest.skip("the list takes 48 GB")
    from paper_2510_10256_gb300 import contact
    contact.build()
    m, apart = 92_800, 400
    assert (m - apart) * (m - apart - 1) // 2 < 2**32 - 1 < m * (m - 1) // 2
    pos = np.random.default_rng(1).uniform(0.0, 1e-3, (3, 2 * m))
    far = pos.copy()
    far[0, :2 * apart] += np.repeat(10.0 + np.arange(apart), 2)
    sc = S.Scene("rod", pos, pos, 0.0 * pos, 0.05, 0.01, rod_ptr=np.arange(0, 2 * m + 1, 2, dtype=np.int32), name="heap")
    cs = contact.ContactScene.from_scene(sc)
    cs.contact_build(torch.from_numpy(far).to("cuda:0"))
    assert cs.stats()["n_candidates"] == (m - apart) * (m - apart - 1) // 2
    with pytest.raises(contact.ContactError) as e:
        cs.contact_build(torch.from_numpy(pos).to("cuda:0"))
    assert e.value.status == TOO_LARGE
    cs.close()
