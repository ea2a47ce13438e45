"""The largest spaces that the no-allocation entry point's fixed array holds:
a space of that size gets past the layout of the array, to the checks of its
determinants (wrong on purpose, so that nothing is swept)."""
import numpy as np
import pytest

from paper_1902_08154_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


# 152 SMs: 309,000 determinants of three electrons need 64 MiB to 0.1 MiB
@pytest.mark.parametrize("na,nb", [(1, 2), (3, 0)])
@pytest.mark.parametrize("ndet,fits", [(308700, True), (345000, False)])
def test_three_electrons(na, nb, ndet, fits):
    import torch

    import paper_1902_08154_gb300 as qp

    norb = 128
    h, eri = S.hamiltonian(norb, 1, 3)
    dets = torch.zeros((ndet, 2, 2), dtype=torch.int64, device="cuda")
    dets[:, 0, 0] = torch.arange(ndet, device="cuda")
    c = torch.full((ndet,), 1.0 / np.sqrt(ndet), dtype=torch.float64, device="cuda")
    rc, _ = qp.qp_pt2_eval_noalloc(norb, na, nb, torch.from_numpy(h).cuda(), torch.from_numpy(eri).cuda(), ndet, dets, c, -9.0, 0)
    assert rc == qp.QP_EINVAL
    assert (b"wrong occupation" if fits else b"too large") in qp.load().qp_pt2_last_error()
