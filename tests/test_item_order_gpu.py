"""Waves of 65,536 work items and more take the items by kind and a cells pass
per kind, smaller ones take them as they come with one cells pass: both give a
generator the same sums, just below and above the line (10 electrons, 55 items
per generator: 1,191 and 1,192 of them), for each number type and for open
shells."""
import numpy as np
import pytest

from paper_1902_08154_gb300 import synthetic as S
from tests.test_zz_no_alloc import _dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("norb,na,nb,ndet,precision", [
    (14, 5, 5, 1191, 0), (14, 5, 5, 1192, 0), (14, 5, 5, 1192, 1), (15, 6, 4, 1200, 0), (20, 9, 1, 1300, 0),
    (66, 5, 5, 1192, 0),
])
def test_generators_do_not_depend_on_the_order_of_items(norb, na, nb, ndet, precision):
    from paper_1902_08154_gb300 import build

    build.build()
    import paper_1902_08154_gb300 as qp

    h, eri = S.hamiltonian_fast(norb, 6, 601)
    dets = S.random_excited_dets(norb, na, nb, ndet, 602)
    c = S.random_coefs(len(dets), 603, decay=0.01)
    e0 = float(np.min(np.diag(h))) * (na + nb) - 50.0
    pt2 = qp.PT2(norb, na, nb, _dev(h), _dev(eri), precision=precision)
    full = pt2.eval(_dev(dets), _dev(c), e0, 200, per_generator=True)
    parts = [pt2.eval_generators(_dev(dets), _dev(c), e0, np.arange(i, min(i + 500, len(dets)))) for i in range(0, len(dets), 500)]
    pt2.close()
    n = len(dets)
    host = lambda x: np.asarray(x.cpu() if hasattr(x, "cpu") else x)[:n]
    # the items' sums are the same terms in the same fixed order
    assert np.array_equal(np.concatenate([g["eps"] for g in parts]), host(full["eps_by_rank"]))
    assert np.array_equal(np.concatenate([g["na"] for g in parts]), host(full["na_by_rank"]))
    assert np.array_equal(np.concatenate([g["ncon"] for g in parts]), host(full["ncon_by_rank"]))
    digest = np.zeros(2, dtype=np.uint64)
    for g in parts:
        digest[0] += np.uint64(g["digest"][0] & (2**64 - 1))
        digest[1] ^= np.uint64(g["digest"][1] & (2**64 - 1))
    assert [int(x) & (2**64 - 1) for x in full["digest"]] == [int(x) for x in digest]
