"""The Hamiltonian's rows as a bit map of their columns: one determinant, the
edges of a word, of a warp and of a block, rows with more neighbouring spin-up
strings than the block's queue holds, and more determinants than one map.  The
test of every pair is the reference: the same columns, and elements by the same
function, bit for bit."""
import numpy as np
import pytest

from paper_1902_08154_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qp():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1902_08154_gb300 import build

    build.build()
    import paper_1902_08154_gb300 as qp

    qp.load()
    return qp


def _strings(rng, count, norb, nocc):
    """Distinct strings in groups of four that differ by one orbital."""
    seen = []
    have = set()
    while len(seen) < count:
        base = [int(p) for p in rng.choice(norb, nocc, replace=False)]
        for _ in range(4):
            key = sum(1 << p for p in base)
            if key not in have and len(seen) < count:
                have.add(key)
                seen.append(key)
            free = [p for p in range(norb) if p not in base]
            base[-1] = free[int(rng.integers(len(free)))]
    return seen


def _words(strings, nint):
    return np.array([[(s >> (64 * w)) & (2**64 - 1) for w in range(nint)] for s in strings], dtype=np.uint64)


def _product(up, dn, nint):
    u, d = _words(up, nint), _words(dn, nint)
    return np.ascontiguousarray(np.stack([np.repeat(u, len(dn), axis=0), np.tile(d, (len(up), 1))], axis=1))


def _case(name):
    rng = np.random.default_rng(len(name))
    if name == "queue":  # 1 + 16 * 48 spin-up strings within one excitation, ten determinants each
        base = (1 << 16) - 1
        up = [base] + [(base ^ (1 << p)) | (1 << q) for p in range(16) for q in range(16, 64)]
        return 64, 16, 3, _product(up, _strings(rng, 10, 64, 3), 1)
    if name == "windows":  # 1,051,050 determinants
        return 64, 6, 5, _product(_strings(rng, 1050, 64, 6), _strings(rng, 1001, 64, 5), 1)
    if name == "two words":
        return 96, 4, 3, _product(_strings(rng, 33, 96, 4), _strings(rng, 31, 96, 3), 2)
    n = int(name)
    dets = _product(_strings(rng, 18, 24, 4), _strings(rng, 16, 24, 3), 1)
    return 24, 4, 3, dets[rng.permutation(len(dets))[:n]].copy()


@pytest.mark.parametrize("name", ["1", "2", "31", "32", "33", "256", "257", "two words", "queue", "windows"])
def test_rows_match_the_test_of_every_pair(qp, name):
    norb, na, nb, dets = _case(name)
    h, eri = S.hamiltonian_fast(norb, 4, 7)
    pt2 = qp.PT2(norb, na, nb, h, eri)
    a = pt2.hamiltonian(dets, search=0)
    b = pt2.hamiltonian(dets, search=1)
    if len(dets) < 300:  # the lowest eigenpair of the same matrix, dense
        n = len(dets)
        H = np.diag(a[3])
        for i in range(n):
            H[i, a[1][a[0][i]:a[0][i + 1]]] = a[2][a[0][i]:a[0][i + 1]]
        e0, c, info = pt2.davidson(dets, tol=1e-10)
        # |E0 - lambda| <= |residual|^2 / gap for the lowest pair, and the
        # rounding of sums of n terms of the size of H
        assert info["converged"] and info["nnz"] == a[0][-1]
        assert e0 == pytest.approx(np.linalg.eigvalsh(H)[0], abs=1e-10)
        assert np.abs(H @ c - e0 * c).max() <= 2e-10 and c[0] >= 0
    pt2.close()
    for x, y in zip(a[:4], b[:4]):
        assert np.array_equal(x, y)
