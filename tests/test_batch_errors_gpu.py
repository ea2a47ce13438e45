"""A batch whose second instance holds determinants of the wrong occupation:
the graph's kernels run on after the check, so they have to leave that
instance alone; the call reports it and the device stays usable."""
import numpy as np
import pytest

from paper_1902_08154_gb300 import synthetic as S
from tests.test_batch_gpu import _dev, qp  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fused", [True, False])
@pytest.mark.parametrize("change", ["one more", "one less", "other spin"])
def test_wrong_occupations_are_reported(qp, fused, change):  # noqa: F811
    norb, na, nb = 16, 4, 4
    h, eri = S.hamiltonian(norb, 18, 401)
    dets = S.random_excited_dets(norb, na, nb, 60, 402)
    c = np.random.default_rng(403).standard_normal(len(dets))
    c[:] = sorted(c, key=abs, reverse=True)
    bad = dets.copy()
    for i in (3, 17, 41):
        free = [q for q in range(norb) if not (int(bad[i, 0, 0]) >> q) & 1]
        occ = [q for q in range(norb) if (int(bad[i, 0, 0]) >> q) & 1]
        if change == "one more":
            bad[i, 0, 0] |= np.uint64(1 << free[0])
        else:
            bad[i, 0, 0] &= np.uint64(~(1 << occ[0]) & (2**64 - 1))
        if change == "other spin":
            bad[i, 1, 0] |= np.uint64(1 << [q for q in range(norb) if not (int(bad[i, 1, 0]) >> q) & 1][0])
    pts = [qp.PT2(norb, na, nb, _dev(h), _dev(eri)) for _ in range(2)]
    inst = lambda p, d: {"pt2": p, "dets": _dev(d), "coefs": _dev(c), "e0": -30.0, "k": 20}
    single = pts[0].eval(_dev(dets), _dev(c), -30.0, 20)
    batch = qp.Batch([inst(pts[0], dets), inst(pts[1], bad)], fused=fused)
    for _ in range(2):
        with pytest.raises(qp.QPError) as ei:
            batch.run()
        assert ei.value.code == qp.QP_EINVAL
    batch.close()
    batch = qp.Batch([inst(pts[0], dets), inst(pts[1], dets)], fused=fused)
    res, _ = batch.run()
    for r in res:
        assert r["e_pt2"] == single["e_pt2"] and r["n_perturbers"] == single["n_perturbers"]
    batch.close()
    for p in pts:
        p.close()
