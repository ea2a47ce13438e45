"""Generator order and selection order by counting against numpy's stable
sort and the oracle: sizes around the blocks of 32 and 256 and across the
limit beyond which the radix sorts are used, ties in c^2, every error."""
import numpy as np
import pytest

from paper_1902_08154_gb300 import synthetic as S
from tests.parity_util import check_selection, check_totals

pytestmark = pytest.mark.gpu


def _dev(a):
    import torch

    return torch.from_numpy(np.ascontiguousarray(a.view(np.int64) if a.dtype == np.uint64 else a)).cuda()


@pytest.mark.parametrize("ndet,norb", [(1, 12), (31, 12), (32, 12), (33, 70), (256, 16), (257, 66), (2049, 16),
                                       (12288, 20), (12289, 20)])
def test_rank_order(ndet, norb):
    import paper_1902_08154_gb300 as qp

    na = nb = 2 if ndet < 40 else 4
    h, eri = S.hamiltonian(norb, 4, 3)
    dets = S.excited_dets_fast(norb, na, nb, ndet, 5)
    c = S.random_coefs(ndet, 6)
    c[::3] = c[0]           # ties in c^2, also with the sign flipped
    c[1::5] = -c[0]
    pt2 = qp.PT2(norb, na, nb, h, eri)
    rank = np.arange(min(ndet, 3), dtype=np.int32)  # few generators swept, the whole order made
    _, res = qp.qp_pt2_eval_gens(pt2.ctx, ndet, _dev(dets), _dev(c), -60.0, rank)
    if ndet <= 2049:
        got = pt2.eval(dets, c, -60.0, 0, per_generator=True)
        want = np.empty(ndet, dtype=np.int32)
        want[np.argsort(-(c * c), kind="stable")] = np.arange(ndet)
        assert np.array_equal(got["rank_of"], want)
    assert res.n_perturbers > 0
    pt2.close()


@pytest.mark.parametrize("k", [1, 31, 33, 700, 100000])
def test_selection_order(oracle_mod, k):
    import paper_1902_08154_gb300 as qp

    norb, na, nb = 14, 3, 3
    h, eri = S.hamiltonian(norb, 9, 3)
    ham = oracle_mod.Hamiltonian(norb, na, nb, h, eri)
    dets = S.random_excited_dets(norb, na, nb, 40, 5)
    c = S.random_coefs(40, 6, decay=0.05)
    e0 = min(ham.diag(d) for d in dets) - 1.0
    ref = ham.sweep(dets, c, e0, k=k)
    pt2 = qp.PT2(norb, na, nb, h, eri)
    for host in (True, False):
        got = pt2.eval(dets if host else _dev(dets), c if host else _dev(c), e0, k)
        check_totals(got, ref)
        check_selection(got["sel_dets"], got["sel_e"], ref["sel_dets"], ref["sel_e"])
    pt2.close()


def test_errors_before_the_sweep():
    import paper_1902_08154_gb300 as qp

    norb, na, nb, n = 14, 3, 3, 300
    h, eri = S.hamiltonian(norb, 9, 3)
    dets = S.random_excited_dets(norb, na, nb, n, 5)
    c = S.random_coefs(n, 6)
    pt2 = qp.PT2(norb, na, nb, h, eri)

    def code(d, cc):
        with pytest.raises(qp.QPError) as e:
            pt2.eval(np.ascontiguousarray(d), cc, -60.0, 5)
        return e.value.code

    d = dets.copy()
    d[299] = d[17]
    assert code(d, c) == qp.QP_EDUP
    d = dets.copy()
    d[40, 0, 0] |= np.uint64(1) << np.uint64(20)
    assert code(d, c) == qp.QP_EINVAL
    d = dets.copy()
    d[5, 1, 0] = 1
    assert code(d, c) == qp.QP_EINVAL
    cc = c.copy()
    cc[290] = np.inf
    assert code(dets, cc) == qp.QP_EINVAL
    assert pt2.eval(dets, c, -60.0, 5)["n_selected"] == 5
    pt2.close()
