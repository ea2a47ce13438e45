"""The gradient's scatter by rows and pair tables against the oracle's, on
spaces whose particles crowd into a few orbitals at the edges of words and
lanes, and with more J reaching every cell than one group of pair tables and
more entries in a batch than one round takes."""
import numpy as np
import pytest

from paper_1902_08154_gb300 import synthetic as S
from tests.test_gradient_gpu import _gpu_grad, qp  # noqa: F401
from tests.test_rows_gpu import _crowded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("norb,na,nb,ndet", [
    (9, 4, 3, 60),     # few virtual orbitals
    (12, 4, 4, 900),   # several rounds and groups
    (33, 3, 3, 80),    # one lane in the second round of a row
    (64, 3, 2, 60),    # bit 63
    (66, 3, 3, 50),    # two words
    (34, 5, 0, 60),    # one spin only
    (40, 1, 1, 40),    # one-hole and one opposite-spin batch
])
def test_gradient_rows_match_oracle(qp, oracle_mod, norb, na, nb, ndet):  # noqa: F811
    h, eri = S.hamiltonian(norb, 6, norb)
    ham = oracle_mod.Hamiltonian(norb, na, nb, h, eri)
    dets = S.random_excited_dets(norb, na, nb, ndet, 8) if ndet > 500 else _crowded(norb, na, nb, ndet, 7)
    c = S.random_coefs(len(dets), 11, decay=0.03)
    e0 = min(ham.diag(d) for d in dets) - 1.0
    ref = ham.gradient(dets, c, e0)
    dh, deri, de0, res = _gpu_grad(qp, norb, na, nb, h, eri, dets, c, e0)
    # sums of at most 10^7 terms of |w| <= 1 in FP64, in different orders
    scale = max(1.0, np.abs(ref["deri"]).max(), np.abs(ref["dh"]).max())
    assert np.abs(dh - ref["dh"]).max() <= 1e-11 * scale
    assert np.abs(deri - ref["deri"]).max() <= 1e-11 * scale
    assert de0 == pytest.approx(ref["de0"], rel=1e-12, abs=1e-13)
