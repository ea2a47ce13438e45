"""One large entry of h or of the integrals (a level-shifted orbital) must not
cost the denominators that do not contain it any accuracy: every sweep against
the oracle at the bounds of ordinary integrals (1e-10 Eh; mixed 1e-6 Eh)."""
import numpy as np
import pytest

from paper_1902_08154_gb300 import synthetic as S
from tests.parity_util import E_TOL, check_per_generator, check_selection, check_totals, cipsi_space

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


# from 1e4 on every generator is in FP64
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


def _energy_sums(norb, h, eri, dets):
    """1/2 sum of |h_ii| and |F(i)| over each determinant's orbitals."""
    def tri(p, q):
        return max(p, q) * (max(p, q) + 1) // 2 + min(p, q)

    J = np.array([[eri[tri(tri(p, p), tri(q, q))] for q in range(norb)] for p in range(norb)])
    K = np.array([[eri[tri(tri(p, q), tri(p, q))] for q in range(norb)] for p in range(norb)])
    out = []
    for d in dets:
        occ = [[q for q in range(norb) if (int(d[s, q // 64]) >> (q % 64)) & 1] for s in range(2)]
        r = 0.0
        for s in range(2):
            for q in occ[s]:
                r += abs(h[q, q]) + abs(h[q, q] + J[q, occ[0]].sum() + J[q, occ[1]].sum() - K[q, occ[s]].sum())
        out.append(0.5 * r)
    return np.array(out)


# the unit, 2^-62 of a power of two below the bound, put between those that
# suit the generators of smallest and of largest energies, E0 near zero
@pytest.mark.parametrize("norb,na,nb,ndet", [(16, 4, 4, 60), (70, 2, 2, 30)])
def test_both_forms_in_one_sweep(oracle_mod, norb, na, nb, ndet):
    import torch

    import paper_1902_08154_gb300 as qp

    h, eri = S.hamiltonian(norb, 8, 5)
    h[np.arange(norb), np.arange(norb)] -= 0.15 * norb  # every h_pp negative
    dets = S.random_excited_dets(norb - 1, na, nb, ndet, 3)
    c = S.random_coefs(ndet, 4, decay=0.05)
    sums = _energy_sums(norb, h, eri, dets)
    f = 2.0 ** np.ceil(np.log2(128.0 * np.median(sums))) / (128.0 * np.median(sums))
    h, eri, sums = h * f, eri * f, sums * f
    unit = 128.0 * np.median(sums)
    n = na + nb + 2
    h[norb - 1, norb - 1] = (1.5 * unit - n * (n - 1) * np.abs(eri).max()) / n
    bound = n * np.abs(h).max() + n * (n - 1) * np.abs(eri).max()
    assert unit * 0.999 <= 2.0 ** np.floor(np.log2(bound)) <= unit * 1.001
    fixed = 128.0 * sums >= unit
    assert 5 < fixed.sum() < ndet - 5

    ham = oracle_mod.Hamiltonian(norb, na, nb, h, eri)
    e0 = 0.01  # above every H_aa but those with the last orbital
    pt2 = qp.PT2(norb, na, nb, h, eri)
    ref = ham.sweep(dets, c, e0, k=40)
    got = pt2.eval(dets, c, e0, 40, per_generator=True)
    check_totals(got, ref)
    check_per_generator(got, ref)
    check_selection(got["sel_dets"], got["sel_e"], ref["sel_dets"], ref["sel_e"])
    batch = qp.Batch([dict(pt2=pt2, dets=_dev(dets), coefs=_dev(c), e0=e0, k=40)])
    for _ in range(2):
        out, _ = batch.run()
        assert out[0]["e_pt2"] == got["e_pt2"] and out[0]["digest"] == got["digest"]
        check_selection(out[0]["sel_dets"], out[0]["sel_e"], ref["sel_dets"], ref["sel_e"])
    batch.close()
    E0 = np.array([e0, 0.02])
    C = np.stack([c, S.random_coefs(ndet, 11, decay=0.03)])
    rs, gs = ham.states(dets, C, E0, k=40), pt2.eval_states(dets, C, E0, 40)
    assert np.abs(gs["e_pt2_states"] - rs["e_pt2_states"]).max() <= E_TOL
    check_selection(gs["sel_dets"], gs["sel_crit"], rs["sel_dets"], rs["sel_crit"])
    pt2.close()
    torch.cuda.synchronize()
