"""qp_pt2_eval_noalloc with three, two and one CTA per SM, as the selection
buffers of k + cells entries leave room in the fixed array, against
qp_pt2_eval: the same perturbers and selection, E_PT2 from the same items."""
import numpy as np
import pytest

from paper_1902_08154_gb300 import synthetic as S
from tests.parity_util import check_selection, check_totals
from tests.test_zz_no_alloc import _dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [0, 1, 300, 1100, 1700, 3000])
def test_launch_shapes_by_k(k):
    import torch

    from paper_1902_08154_gb300 import build

    build.build()
    import paper_1902_08154_gb300 as qp

    norb, na, nb = 28, 5, 4
    h, eri = S.hamiltonian(norb, 20, 501)
    dets = S.random_excited_dets(norb, na, nb, 150, 502)
    c = S.random_coefs(len(dets), 503, decay=0.05)
    hd, ed, dd, cd = _dev(h), _dev(eri), _dev(dets), _dev(c)
    e0 = float(np.min(np.diag(h))) * (na + nb) - 50.0
    pt2 = qp.PT2(norb, na, nb, hd, ed)
    ref = pt2.eval(dd, cd, e0, k)
    pt2.close()
    sel = torch.zeros((max(k, 1), 2, 1), dtype=torch.int64, device="cuda")
    sel_e = torch.zeros(max(k, 1), dtype=torch.float64, device="cuda")
    rc, res = qp.qp_pt2_eval_noalloc(norb, na, nb, hd, ed, len(dets), dd, cd, e0, k, sel, sel_e)
    torch.cuda.synchronize()
    assert rc == qp.QP_OK
    got = res.as_dict()
    check_totals(got, ref)
    m = got["n_selected"]
    assert m == min(k, got["n_perturbers"])
    if k:
        check_selection(sel[:m], sel_e[:m], ref["sel_dets"], ref["sel_e"])
