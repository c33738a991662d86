"""A hub whose part of the candidates has more distinct communities than the
part's table has slots: the part is done in ranges of a second hash, halved until
a range fits.  Parts are chosen by a hash of the community id, so on a graph of
ordinary size the communities next to the hub get ids of one part (and, for
several halvings in a row, of one end of the second hash); the hashes are taken from
the source.  One queue of all nodes, so that the hub meets exactly these
communities; every result equal to the oracle's."""
import numpy as np
import pytest

from device_source import build

pytestmark = pytest.mark.gpu

TRIANGLES = 5000


@pytest.fixture(scope="module")
def hashes(tmp_path_factory):
    return build(tmp_path_factory.mktemp("hub"), ["hash32", "lh_parts", "lh_part_of", "lh_range_of"],
                 ["LH_PART", "LH_PARTS", "LH_SLOTS"], """
extern "C" int parts(uint32_t total) { return lh_parts(total); }
extern "C" int part_of(int32_t C, int P) { return lh_part_of(C, P); }
extern "C" uint32_t range_of(int32_t C) { return lh_range_of(C); }
extern "C" int slots() { return (int)LH_SLOTS; }
""")


def graph_and_cover(h, below):
    """A hub joined to two corners of each triangle, whose third corners have zero to
    three neighbours in a ring; triangle i is a community whose id is of the hub's
    part 1 and below `below` in the second hash.  The other ids are single nodes of
    the ring.  The hub is in communities of both kinds."""
    P = h.parts(2 * TRIANGLES)
    ids, c = [], 0
    while len(ids) < TRIANGLES:
        if h.part_of(c, P) == 1 and h.range_of(c) < below:
            ids.append(c)
        c += 1
    assert len(ids) > h.slots()
    k = ids[-1] + 1
    t = np.arange(TRIANGLES)
    a, b, z = 1 + 3 * t, 2 + 3 * t, 3 + 3 * t
    ring = 1 + 3 * TRIANGLES + np.arange(max(k - TRIANGLES, 3))
    zero = np.zeros(TRIANGLES)
    src = np.concatenate([zero, zero, a, b, a, ring] + [z[t % 4 > j] for j in range(3)]).astype(np.int32)
    dst = np.concatenate([a, b, b, z, z, np.roll(ring, 1)] +
                         [ring[(7 * t + j) % len(ring)][t % 4 > j] for j in range(3)]).astype(np.int32)
    cover, other = [None] * k, iter(ring)
    for i, c in enumerate(ids):
        cover[c] = [a[i], b[i], z[i]]
    for c in range(k):
        if cover[c] is None:
            cover[c] = [next(other)]
    fillers = [c for c in range(k) if len(cover[c]) == 1]
    mine = [ids[0], ids[TRIANGLES // 2], ids[-1]] + fillers[:2]
    mine += [c for c in fillers if h.part_of(c, P) == 1][:4]   # none where the part is all triangles
    for c in set(mine):
        cover[c] = [0] + list(cover[c])
    return src, dst, [np.array(c, np.int32) for c in cover]


@pytest.mark.parametrize("below", [1 << 16, 1 << 14], ids=["one_halving", "three_halvings"])
@pytest.mark.parametrize("opts", [{}, dict(debug_checks=True)], ids=["plain", "bounds_checked"])
def test_hub_part_larger_than_its_table(hashes, below, opts):
    import oracle
    from paper_2210_03211_gb300 import lazyfox
    src, dst, cover = graph_and_cover(hashes, below)
    og = oracle.OracleGraph(src, dst)
    og.set_partition(cover)
    ref = og.run(1 << 30, -np.inf, 2, rule="literal")
    with lazyfox.Graph(src, dst, gain_rule="literal", **opts) as g:
        g.set_partition(cover)
        st = g.run(1 << 30, -np.inf, 2)
        assert st.wcc_initial == ref["T0"] and np.array_equal(st.wcc_history, ref["T"])
        assert np.array_equal(st.joins, ref["joins"]) and np.array_equal(st.leaves, ref["leaves"])
        s, o = g.state(), og.state()
        for key in ("mem_off", "mem_ids", "n", "m", "vol"):
            assert np.array_equal(s[key], o[key]), key
