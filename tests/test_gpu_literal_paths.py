"""Runs under the paper's gain where its kernels change paths: communities around
the sizes at which the member sums go from eight lanes to a warp to a block
(64, 128, 512), degrees around the evaluation's small-node limit (32), the apply's
piece of 512 neighbours and the hub limit (1024), and rows longer than the
eight ids that load together and than a warp.  Both launch modes, team sizes and
queue sizes; every result compared with the oracle exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def graph_and_cover(top, seed=0):
    """Seven nodes of exactly the degrees in question over 1,300 others with a
    sparse random background, and a cover with communities of the sizes in
    question; the first nodes are members of 40, 33 and 9 more of them."""
    rng = np.random.default_rng(seed)
    n, rest = 1307, np.arange(7, 1307)
    src, dst = [rng.choice(rest, 2500)], [rng.choice(rest, 2500)]
    for i, d in enumerate((31, 32, 33, 511, 512, 513, top)):
        src.append(np.full(d, i))
        dst.append(rng.permutation(rest)[:d])
    cover = [rng.choice(n, size=k, replace=False) for k in (1, 2, 8, 9, 63, 64, 65, 127, 128, 129, 511, 512, 513)]
    cover += [rng.choice(n, size=int(k), replace=False) for k in rng.integers(2, 40, 60)]
    for x, times in ((0, 40), (3, 33), (6, 9)):
        for c in rng.choice(np.arange(13, len(cover)), size=times, replace=False):
            cover[c] = np.union1d(cover[c], [x])
    src, dst = np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32)
    present = np.unique(np.concatenate([src[src != dst], dst[src != dst]]))
    cover = [np.intersect1d(c, present).astype(np.int32) for c in cover]
    return src, dst, [c for c in cover if c.shape[0]]


@pytest.mark.parametrize("top,q,opts", [
    (1024, 1, {}), (1024, 3, {}), (1024, 64, {}), (1024, 64, dict(warps_per_node=1)),
    (1024, 64, dict(warps_per_node=2)), (1024, 300, dict(per_queue_launches=False)),
    (1024, 300, dict(per_queue_launches=True)), (1024, 1300, dict(per_queue_launches=False, warps_per_node=1)),
    (1024, 40, dict(per_queue_launches=True)), (1025, 3, {}), (1200, 64, {}), (1200, 1300, {}),
    (1024, 64, dict(exhaustive_fp64=True)), (1024, 64, dict(debug_checks=True)),
    (1024, 64, dict(barrier_mode=1)),
])
def test_literal_paths_equal_the_oracle(top, q, opts):
    import oracle
    from paper_2210_03211_gb300 import lazyfox
    src, dst, cover = graph_and_cover(top)
    og = oracle.OracleGraph(src, dst)
    og.set_partition(cover)
    iters = 2 if q < 10 else 3
    ref = og.run(q, -np.inf, iters, rule="literal")
    with lazyfox.Graph(src, dst, gain_rule="literal", **opts) as g:
        g.set_partition(cover)
        st = g.run(q, -np.inf, iters)
        assert st.iterations == ref["iterations"] and st.wcc_initial == ref["T0"]
        assert np.array_equal(st.joins, ref["joins"]) and np.array_equal(st.leaves, ref["leaves"])
        assert np.array_equal(st.wcc_history, ref["T"])
        assert [c.tolist() for c in g.community_list()] == [c.tolist() for c in og.communities()]
        s, o = g.state(), og.state()
        for k in ("mem_off", "mem_ids", "n", "m", "vol"):
            assert np.array_equal(s[k], o[k]), k


def test_literal_loop_times_out_and_recovers():
    """A block of the persistent loop that never arrives ends the call with
    LF_ERR_TIMEOUT (bounded waits); a normal run afterwards is right."""
    import oracle
    from paper_2210_03211_gb300 import lazyfox
    src, dst, cover = graph_and_cover(1024)
    with lazyfox.Graph(src, dst, inject_barrier_stall=True, barrier_timeout_ms=50,
                       per_queue_launches=False) as g:
        with pytest.raises(lazyfox.LazyFoxError) as e:
            g.run(64, 0.01, 3)
        assert e.value.status == lazyfox.LF_ERR_TIMEOUT
    ref = oracle.OracleGraph(src, dst).run(64, 0.01, 3, rule="literal")
    with lazyfox.Graph(src, dst) as g:
        assert np.array_equal(g.run(64, 0.01, 3).wcc_history, ref["T"])
