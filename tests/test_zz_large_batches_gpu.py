"""The largest opposite-spin batches (124 to 128 orbitals, few electrons) in
every entry point that does not split them by itself: on both sides of the
size up to which one accumulator fits on an SM."""
import numpy as np
import pytest

from paper_1902_08154_gb300 import synthetic as S
from tests.parity_util import check_selection, check_totals

pytestmark = pytest.mark.gpu


def _dev(a):
    import torch

    return torch.from_numpy(np.ascontiguousarray(a.view(np.int64) if a.dtype == np.uint64 else a)).cuda()


# 121 x 121 cells fit in one tile, 122 x 122 (and all larger ones) do not
@pytest.mark.parametrize("norb,na,nb", [(124, 3, 3), (125, 3, 3), (128, 3, 3), (128, 1, 1)])
def test_unsplit_batches(oracle_mod, norb, na, nb):
    import torch

    import paper_1902_08154_gb300 as qp

    ndet, k = 3, 30
    h, eri = S.hamiltonian(norb, 2, 7)
    ham = oracle_mod.Hamiltonian(norb, na, nb, h, eri)
    dets = S.random_excited_dets(norb, na, nb, ndet, 8)
    c = S.random_coefs(ndet, 9, decay=0.05)
    e0 = min(ham.diag(d) for d in dets) - 1.0
    ref = ham.sweep(dets, c, e0, k=k)
    hd, ed, dd, cd = _dev(h), _dev(eri), _dev(dets), _dev(c)

    rc, res = qp.qp_pt2_eval_noalloc(norb, na, nb, hd, ed, ndet, dd, cd, e0, 0)
    assert rc == qp.QP_OK, qp.load().qp_pt2_last_error()
    check_totals(dict(res.as_dict(), n_selected=k), ref)

    pt2 = qp.PT2(norb, na, nb, hd, ed, tile=1)
    got = pt2.eval(dd, cd, e0, k)
    check_totals(got, ref)
    check_selection(got["sel_dets"], got["sel_e"], ref["sel_dets"], ref["sel_e"])

    batch = qp.Batch([dict(pt2=pt2, dets=dd, coefs=cd, e0=e0, k=k)], tile=1)
    out, _ = batch.run()
    check_totals(out[0], ref)
    check_selection(out[0]["sel_dets"], out[0]["sel_e"], ref["sel_dets"], ref["sel_e"])
    batch.close()
    pt2.close()
    torch.cuda.empty_cache()
