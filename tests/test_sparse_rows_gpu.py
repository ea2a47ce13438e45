"""Rows of the Hamiltonian with few connected determinants beside rows with
many, in spaces where the map of a row is long: against the all-pairs search
bit for bit, and, above 2^20 determinants, against brute force for some rows."""
import numpy as np
import pytest

from paper_1902_08154_gb300 import synthetic as S

pytestmark = pytest.mark.gpu

NORB, NEL = 64, 10


def _strings(rng, nsingle, nrand):
    """The reference string, `nsingle` of its single excitations (all connected
    with one another) and random strings."""
    ref = (1 << NEL) - 1
    singles = [ref ^ (1 << i) ^ (1 << a) for i in range(NEL) for a in range(NEL, NORB)]
    out = [ref] + [singles[i] for i in rng.permutation(len(singles))[:nsingle]]
    while len(set(out)) < 1 + nsingle + nrand:
        out.append(sum(1 << int(q) for q in rng.choice(NORB, NEL, replace=False)))
    return np.array(sorted(set(out)), dtype=np.uint64)


def _space(rng, a, b):
    d = np.zeros((len(a) * len(b), 2, 1), dtype=np.uint64)
    d[:, 0, 0], d[:, 1, 0] = np.repeat(a, len(b)), np.tile(b, len(a))
    return np.ascontiguousarray(d[rng.permutation(len(d))])


def _pt2():
    import paper_1902_08154_gb300 as qp

    return qp.PT2(NORB, NEL, NEL, *S.hamiltonian(NORB, 2, 3))


# columns per row around the lengths at which counting and the map change
# over: 3 (n / 32) words against len * 256 comparisons
@pytest.mark.parametrize("singles_b,rand_b,rand_a", [(9, 140, 200), (10, 140, 200), (11, 140, 200), (40, 110, 200),
                                                     (1, 0, 500), (300, 0, 100)])
def test_matches_all_pairs(singles_b, rand_b, rand_a):
    rng = np.random.default_rng(singles_b)
    dets = _space(rng, _strings(rng, 2, rand_a), _strings(rng, singles_b, rand_b))
    pt2 = _pt2()
    got, want = pt2.hamiltonian(dets, search=0), pt2.hamiltonian(dets, search=1)
    for x, y in zip(got[:4], want[:4]):
        assert np.array_equal(x, y)
    pt2.close()


def test_two_windows():
    rng = np.random.default_rng(7)
    dets = _space(rng, _strings(rng, 0, 99), _strings(rng, 540, 9959))
    assert len(dets) > 1 << 20
    pt2 = _pt2()
    rowptr, cols, _, _, _ = pt2.hamiltonian(dets)
    pt2.close()
    nnz = np.diff(rowptr)
    many, few = np.flatnonzero(nnz > 512), np.flatnonzero((nnz > 0) & (nnz < 20))
    assert len(many) and len(few)
    for r in np.concatenate([rng.choice(many, 8), rng.choice(few, 8), [0, len(dets) - 1]]):
        deg = np.bitwise_count(dets ^ dets[r]).sum(axis=(1, 2)) // 2
        want = np.flatnonzero((deg == 1) | (deg == 2))
        assert np.array_equal(cols[rowptr[r]:rowptr[r + 1]], want)
