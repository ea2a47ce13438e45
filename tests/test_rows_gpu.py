"""The row pass of the batch kernel (phase masks, warp-wide single
substitutions, one-hole batches) against the oracle, on spaces whose
particles crowd into a few orbitals at the edges of words and lanes, so that
cells holding one, two and three particles of the same J are common."""
import numpy as np
import pytest

from paper_1902_08154_gb300 import synthetic as S
from tests.parity_util import check_per_generator, check_selection, check_totals

pytestmark = pytest.mark.gpu


def _crowded(norb, na, nb, ndet, seed):
    """Distinct determinants, up to 4 electrons moved into a few virtual orbitals."""
    rng = np.random.default_rng(seed)
    edge = [o for o in (30, 31, 32, 33, 62, 63, 64, 65, 95, 96, norb - 2, norb - 1) if max(na, nb) <= o < norb]
    few = sorted(set(edge[-7:] + list(range(max(na, nb), min(norb, max(na, nb) + 3)))))
    seen, out = set(), []
    for _ in range(100 * ndet):
        occ = [list(range(na)), list(range(nb))]
        for _ in range(int(rng.integers(0, 5))):
            s = int(rng.integers(0, 2))
            free = [o for o in few if o not in occ[s]]
            if occ[s] and free:
                occ[s].remove(occ[s][int(rng.integers(0, len(occ[s])))])
                occ[s].append(free[int(rng.integers(0, len(free)))])
        d = S.occ_to_det(sorted(occ[0]), sorted(occ[1]), norb)
        if d.tobytes() not in seen:
            seen.add(d.tobytes())
            out.append(d)
        if len(out) == ndet:
            break
    return np.ascontiguousarray(np.stack(out), dtype=np.uint64)


@pytest.mark.parametrize("norb,na,nb,ndet", [
    (9, 4, 3, 60),     # few virtual orbitals: most rows are flagged
    (33, 3, 3, 80),    # one lane in the second round of a row
    (64, 3, 2, 80),    # bit 63
    (65, 3, 3, 60),    # one bit in the second word
    (128, 3, 2, 50),   # bit 127
    (34, 5, 0, 60),    # one spin only
    (40, 1, 1, 40),    # one-hole and one opposite-spin batch
])
def test_rows_match_oracle(oracle_mod, norb, na, nb, ndet):
    import torch

    import paper_1902_08154_gb300 as qp

    h, eri = S.hamiltonian(norb, 6, norb)
    ham = oracle_mod.Hamiltonian(norb, na, nb, h, eri)
    dets = _crowded(norb, na, nb, ndet, 7)
    c = S.random_coefs(len(dets), 11, decay=0.03)
    e0 = min(ham.diag(d) for d in dets) - 1.0
    ref = ham.sweep(dets, c, e0, k=60)
    pt2 = qp.PT2(norb, na, nb, torch.from_numpy(h).cuda(), torch.from_numpy(eri).cuda())
    got = pt2.eval(torch.from_numpy(dets.view(np.int64)).cuda(), torch.from_numpy(c).cuda(), e0, 60, per_generator=True)
    check_totals(got, ref)
    check_per_generator(got, ref)
    check_selection(got["sel_dets"], got["sel_e"], ref["sel_dets"], ref["sel_e"])
    pt2.close()
