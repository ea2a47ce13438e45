"""One large entry of h or of the integrals (a level-shifted orbital) must not
cost the denominators that do not contain it any accuracy: every sweep against
the oracle at the bounds of ordinary integrals (1e-10 Eh; mixed 1e-6 Eh)."""
import numpy as np
import pytest

from paper_1902_08154_gb300 import synthetic as S
from tests.parity_util import E_TOL, check_selection, check_totals, cipsi_space

pytestmark = pytest.mark.gpu


def _dev(a):
    import torch

    return torch.from_numpy(np.ascontiguousarray(a.view(np.int64) if a.dtype == np.uint64 else a)).cuda()


def _case(oracle_mod, norb, na, nb, ndet, entry, size):
    """Psi0 leaves the last orbital empty; its own entry is `size`."""
    h, eri = S.hamiltonian(norb, 8, 5)
    if entry == "h":
        h[norb - 1, norb - 1] = size
    else:  # (rr|rr)
        eri[-1] = size
    ham = oracle_mod.Hamiltonian(norb, na, nb, h, eri)
    dets = S.random_excited_dets(norb - 1, na, nb, ndet, 3)
    c = S.random_coefs(ndet, 4, decay=0.05)
    return h, eri, ham, dets, c, min(ham.diag(d) for d in dets) - 1.0


SIZES = [(16, 4, 4, 30), (70, 2, 2, 12), (20, 1, 0, 3)]


# 1e2: some generators in fixed point and some in FP64; above: all in FP64
@pytest.mark.parametrize("norb,na,nb,ndet", SIZES)
@pytest.mark.parametrize("entry", ["h", "eri"])
@pytest.mark.parametrize("size", [1e2, 1e4, 1e6, 1e8, 1e12])
def test_sweep(oracle_mod, norb, na, nb, ndet, entry, size):
    import paper_1902_08154_gb300 as qp

    h, eri, ham, dets, c, e0 = _case(oracle_mod, norb, na, nb, ndet, entry, size)
    ref = ham.sweep(dets, c, e0, k=40)
    pt2 = qp.PT2(norb, na, nb, h, eri)
    got = pt2.eval(dets, c, e0, 40)
    check_totals(got, ref)
    check_selection(got["sel_dets"], got["sel_e"], ref["sel_dets"], ref["sel_e"])
    pt2.close()


# the mixed form states its bound for a unit-norm, variational Psi0
@pytest.mark.parametrize("norb,na,nb,ndet", [(16, 4, 4, 64), (70, 2, 2, 32)])
@pytest.mark.parametrize("size", [1e2, 1e6, 1e12])
def test_mixed_sweep(oracle_mod, norb, na, nb, ndet, size):
    import paper_1902_08154_gb300 as qp

    h, eri, ham, _, _, _ = _case(oracle_mod, norb, na, nb, 2, "h", size)
    dets, c, e0 = cipsi_space(oracle_mod, ham, norb, na, nb, ndet)
    ref = ham.sweep(dets, c, e0, k=0)
    pt2 = qp.PT2(norb, na, nb, h, eri, precision=qp.QP_MIXED)
    check_totals(pt2.eval(dets, c, e0, 0), ref, e_tol=1e-6)
    pt2.close()


@pytest.mark.parametrize("size", [1e2, 1e6, 1e8, 1e12])
def test_other_entry_points(oracle_mod, size):
    import torch

    import paper_1902_08154_gb300 as qp

    norb, na, nb, ndet = SIZES[0]
    h, eri, ham, dets, c, e0 = _case(oracle_mod, norb, na, nb, ndet, "h", size)
    ref = ham.sweep(dets, c, e0, k=40)
    hd, ed, dd, cd = _dev(h), _dev(eri), _dev(dets), _dev(c)
    pt2 = qp.PT2(norb, na, nb, hd, ed)

    sel, se = torch.zeros((40, 2, 1), dtype=torch.int64, device="cuda"), torch.zeros(40, dtype=torch.float64, device="cuda")
    rc, res = qp.qp_pt2_eval_noalloc(norb, na, nb, hd, ed, ndet, dd, cd, e0, 40, sel, se)
    assert rc == qp.QP_OK
    check_totals(res.as_dict(), ref)
    check_selection(sel, se, ref["sel_dets"], ref["sel_e"])

    batch = qp.Batch([dict(pt2=pt2, dets=dd, coefs=cd, e0=e0, k=40)])
    out, _ = batch.run()
    check_totals(out[0], ref)
    check_selection(out[0]["sel_dets"], out[0]["sel_e"], ref["sel_dets"], ref["sel_e"])
    batch.close()

    C = np.stack([c, S.random_coefs(ndet, 11, decay=0.03)])
    E0 = np.array([e0, e0 - 0.2])
    rs = ham.states(dets, C, E0, k=40)
    got = pt2.eval_states(dets, C, E0, 40)
    assert got["n_perturbers"] == rs["n_perturbers"]
    assert np.abs(got["e_pt2_states"] - rs["e_pt2_states"]).max() <= E_TOL
    assert np.all(np.abs(got["sum_e_over_d_states"] - rs["sum_e_over_d_states"])
                  <= E_TOL * np.maximum(1.0, np.abs(rs["sum_e_over_d_states"])))
    check_selection(got["sel_dets"], got["sel_crit"], rs["sel_dets"], rs["sel_crit"])

    dh, deri = torch.zeros_like(hd), torch.zeros_like(ed)
    de0, res = qp.qp_pt2_grad(pt2.ctx, ndet, dd, cd, e0, dh, deri)
    assert abs(res.e_pt2 - ref["e_pt2"]) <= E_TOL
    rg = ham.gradient(dets, c, e0)
    assert abs(de0 - rg["de0"]) <= 1e-9 * max(1.0, abs(rg["de0"]))
    for got, want in ((dh, rg["dh"]), (deri, rg["deri"])):
        got, want = got.cpu().numpy().reshape(-1), np.asarray(want).reshape(-1)
        assert np.abs(got - want).max() <= 1e-9 * max(1.0, np.abs(want).max())
    pt2.close()
