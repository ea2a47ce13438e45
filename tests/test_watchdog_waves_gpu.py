"""Once the watchdog's time has passed no CTA takes another work item: not in
the later waves of a sweep, nor in the later instances of a batch's launch."""
import ctypes
import json
import os

import numpy as np
import pytest

from paper_1902_08154_gb300 import synthetic as S

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden")


def _dev(a):
    import torch

    return torch.from_numpy(np.ascontiguousarray(a.view(np.int64) if a.dtype == np.uint64 else a)).cuda()


def test_later_waves_do_nothing():
    import paper_1902_08154_gb300 as qp

    P = np.load(os.path.join(GOLDEN, "cfg2_psi0.npz"))
    meta = json.loads(str(P["meta"]))
    h, eri = S.hamiltonian(meta["norb"], meta["rank"], meta["seed"])
    pt2 = qp.PT2(meta["norb"], meta["nalpha"], meta["nbeta"], _dev(h), _dev(eri), timeout_s=1e-6)
    got = pt2.eval(_dev(P["dets"]), _dev(P["coefs"]), float(P["e0"]), 100, per_generator=True, check=False)
    assert got["rc"] == qp.QP_ETIMEOUT
    na = got["na_by_rank"].cpu().numpy()
    # 4 GiB of records hold about 2,600 of its 10,000 generators; of the first
    # wave only the items already taken are run, a few hundred of the first ranks
    assert na[1000:].sum() == 0
    pt2.close()


def test_later_instances_do_nothing():
    import paper_1902_08154_gb300 as qp

    insts = []
    for i in range(3):  # 7,800 items each: every CTA has some in the first
        norb, na, nb, n = 24, 6, 6, 100
        h, eri = S.hamiltonian(norb, 10, 30 + i)
        dets = S.random_excited_dets(norb, na, nb, n, 40 + i)
        c = S.random_coefs(n, 50 + i, decay=0.05)
        pt2 = qp.PT2(norb, na, nb, _dev(h), _dev(eri), timeout_s=1e-6)
        insts.append(dict(pt2=pt2, dets=_dev(dets), coefs=_dev(c), e0=-200.0, k=10))
    batch = qp.Batch(insts)
    res = (qp.Result * 3)()
    ms = ctypes.c_double()
    assert qp.load().qp_pt2_batch_run(batch.handle, res, ctypes.byref(ms)) == qp.QP_ETIMEOUT
    assert sum(r.n_perturbers > 0 for r in res) <= 1
    batch.close()
    for inst in insts:
        inst["pt2"].close()
