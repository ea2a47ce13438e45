"""The fixed-point denominators and integer quotients of the cells pass
against the oracle: integrals scaled by powers of two, E0 far below, far away
and among the diagonal energies (denominators of both signs), one electron,
and integrals that are not finite."""
import numpy as np
import pytest

from paper_1902_08154_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


def _run(norb, na, nb, h, eri, dets, c, e0):
    import torch

    import paper_1902_08154_gb300 as qp

    pt2 = qp.PT2(norb, na, nb, torch.from_numpy(h).cuda(), torch.from_numpy(eri).cuda())
    got = pt2.eval(torch.from_numpy(dets.view(np.int64)).cuda(), torch.from_numpy(c).cuda(), e0, 40, check=False)
    got["sel_e"] = got["sel_e"].cpu().numpy()
    pt2.close()
    return got


# every quantity is linear (energies) or invariant (s2) under the scale, so
# the bounds are those of the unscaled sweep: 1e-10 Eh times the scale on sums
# near 1 Eh, 1e-10 relative on each e_alpha and on the smallest denominator
@pytest.mark.parametrize("norb,na,nb,ndet", [(14, 3, 3, 40), (70, 2, 2, 20), (20, 1, 0, 3), (16, 1, 1, 6)])
@pytest.mark.parametrize("log2_scale,shift", [(0, -1.0), (0, -1.0e6), (-40, -0.5), (30, -2.0), (0, 4.03)])
def test_scaled_denominators(oracle_mod, norb, na, nb, ndet, log2_scale, shift):
    f = 2.0 ** log2_scale
    h, eri = S.hamiltonian(norb, 8, 5)
    h, eri = h * f, eri * f
    ham = oracle_mod.Hamiltonian(norb, na, nb, h, eri)
    dets = S.random_excited_dets(norb, na, nb, ndet, 3)
    c = S.random_coefs(ndet, 4, decay=0.05)
    e0 = min(ham.diag(d) for d in dets) + shift * f
    ref = ham.sweep(dets, c, e0, k=40)
    got = _run(norb, na, nb, h, eri, dets, c, e0)
    assert got["n_perturbers"] == ref["n_perturbers"] and tuple(got["digest"]) == tuple(int(x) for x in ref["digest"])
    near = ref["min_abs_den"] / f  # E0 among the energies: errors grow with 1 / |D|
    tol = 1e-10 * max(1.0, 1.0 / near) ** 2
    assert abs(got["e_pt2"] - ref["e_pt2"]) <= tol * f * max(1.0, abs(ref["e_pt2"]) / f)
    assert abs(got["sum_e_over_d"] - ref["sum_e_over_d"]) <= tol * max(1.0, ref["sum_e_over_d"])
    assert abs(got["min_abs_den"] - ref["min_abs_den"]) <= 1e-12 * abs(e0) + 1e-10 * ref["min_abs_den"]
    assert np.all(np.abs(got["sel_e"] - ref["sel_e"]) <= tol * np.abs(ref["sel_e"]) + 1e-12 * f)


def test_integrals_not_finite_give_nan():
    norb, na, nb = 12, 3, 3
    h, eri = S.hamiltonian(norb, 8, 5)
    eri[3] = np.nan
    dets = S.random_excited_dets(norb, na, nb, 20, 3)
    got = _run(norb, na, nb, h, eri, dets, S.random_coefs(20, 4), -50.0)
    assert np.isnan(got["e_pt2"])
