"""F1 of covers where its blocks share out the detected communities: numbers of them
around one a block (760 blocks) and eight a block, with some that a whole block takes
(more than 256 reference memberships) anywhere among the small ones.  Compared
with the oracle exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [1, 9, 759, 760, 761, 6079, 6080, 6081, 12161])
def test_f1_by_number_of_communities(count):
    import oracle
    from paper_2210_03211_gb300 import lazyfox
    rng = np.random.default_rng(count)
    n = 40000
    ref = [rng.choice(n, size=int(k), replace=False).astype(np.int32) for k in rng.integers(2, 40, 4000)]
    sizes = rng.integers(1, 20, count)
    sizes[rng.integers(0, count, min(count, 40))] = 400
    det = [rng.choice(n, size=int(k), replace=False).astype(np.int32) for k in sizes]
    want, best = oracle.cover_f1(det, ref)
    got, gbest = lazyfox.cover_f1(det, ref)
    assert got == want and np.array_equal(gbest, best)
