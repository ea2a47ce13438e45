"""The whole generator order on both sides of the size up to which it is made
by counting, with ties in c^2, against numpy's stable sort: from a sweep of one
generator shard in a thousand, so that little else is done."""
import numpy as np
import pytest

from paper_1902_08154_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("norb", [20, 66])
@pytest.mark.parametrize("ndet", [8193, 12287, 12288, 12289, 20000])
def test_rank_of(ndet, norb):
    import paper_1902_08154_gb300 as qp

    h, eri = S.hamiltonian(norb, 2, 3)
    dets = S.excited_dets_fast(norb, 4, 4, ndet, 5)
    c = S.random_coefs(ndet, 6)
    c[::3] = c[0]           # ties in c^2, also with the sign flipped
    c[1::5] = -c[0]
    c[7::11] = 0.0
    pt2 = qp.PT2(norb, 4, 4, h, eri, shard_index=0, shard_count=ndet // 4)
    got = pt2.eval(dets, c, -60.0, 0, per_generator=True)
    pt2.close()
    want = np.empty(ndet, dtype=np.int32)
    want[np.argsort(-(c * c), kind="stable")] = np.arange(ndet)
    assert np.array_equal(got["rank_of"], want)
