"""F1 of covers where its kernel changes paths: detected communities of 256 and 257
reference memberships (a warp or the block), above the block's table (several
parts), ids dense enough for the table of ranges and too sparse for it, and a
detected community that shares no node.  Compared with the oracle exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def covers(scale, offset):
    rng = np.random.default_rng(3)
    n = 6000
    ref = [rng.choice(n, size=int(k), replace=False) for k in rng.integers(2, 60, 400)]
    ref += [np.arange(i, n, 2500) for i in range(2500)]          # every node in one of these: 2,500 candidates
    det = [rng.choice(n, size=k, replace=False) for k in (1, 2, 31, 33, 300, 5000)]
    held = np.bincount(np.concatenate(ref), minlength=n)          # reference memberships of each node
    order = rng.permutation(n)
    total = np.cumsum(held[order])
    for want in (255, 256, 257):
        det.append(order[:int(np.searchsorted(total, want)) + 1])
    det.append(np.array([n + 5, n + 9]))                          # in no reference community
    f = lambda cover: [np.sort(c).astype(np.int64) * scale + offset for c in cover]   # noqa: E731
    return [c.astype(np.int32) for c in f(det)], [c.astype(np.int32) for c in f(ref)]


@pytest.mark.parametrize("scale,offset", [(1, 0), (3, 7), (300000, 11), (1, 2**31 - 6100)])
def test_f1_paths_equal_the_oracle(scale, offset):
    import oracle
    from paper_2210_03211_gb300 import lazyfox
    det, ref = covers(scale, offset)
    want, best = oracle.cover_f1(det, ref)
    got, gbest = lazyfox.cover_f1(det, ref)
    assert got == want and np.array_equal(gbest, best)
    for k in range(len(det)):
        w1, b1 = oracle.cover_f1(det[k:k + 1], ref)
        g1, h1 = lazyfox.cover_f1(det[k:k + 1], ref)
        assert g1 == w1 and np.array_equal(h1, b1), k
