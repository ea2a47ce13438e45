"""Two threads with contexts of different sizes: kernels whose shared memory
depends on the sizes are launched by both, again and again."""
import threading

import numpy as np
import pytest

from paper_1902_08154_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


def test_contexts_of_different_sizes_in_two_threads():
    import paper_1902_08154_gb300 as qp

    # ban masks of 100 KB per generator against 4 KB, the same kernels (two words)
    runs, errors = [], []
    for norb, na, nb, ndet, reps in ((128, 24, 24, 2, 150), (66, 2, 2, 4, 1500)):
        h, eri = S.hamiltonian(norb, 1, 3)
        dets = S.random_excited_dets(norb, na, nb, ndet, 4)
        c = S.random_coefs(ndet, 5)
        pt2 = qp.PT2(norb, na, nb, h, eri)
        runs.append((pt2, dets, c, pt2.eval(dets, c, -300.0, 0)["e_pt2"], reps))

    def work(pt2, dets, c, want, reps):
        try:
            for _ in range(reps):
                assert pt2.eval(dets, c, -300.0, 0)["e_pt2"] == want
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=r) for r in runs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]
    assert np.isfinite(runs[0][3])
    for r in runs:
        r[0].close()
