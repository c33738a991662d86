"""The persistent queue loop under the paper's gain: which queues take it, what it
plans (on graphs with nodes of 513 to 1,024 neighbours and rows of more than four
communities, which launches per queue give to the hub kernels and the loop evaluates
in its own block), its central barrier over many blocks, and a handle's runs after a
barrier ran out of time.  Compared with the oracle exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def graph(nodes=900, busy=12, seed=0):
    """`busy` nodes of 520 to 880 neighbours over a sparse random background."""
    rng = np.random.default_rng(seed)
    rest = np.arange(busy, nodes)
    src, dst = [rng.choice(rest, 2000)], [rng.choice(rest, 2000)]
    for i, d in enumerate(np.linspace(520, 880, busy).astype(int)):
        src.append(np.full(d, i))
        dst.append(rng.permutation(rest)[:d])
    return np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32)


def test_loop_plans_no_hub_kernels():
    """The hub plan is thirteen allocations; the loop makes none of them, keeps tables
    in global memory for its own large nodes, and its run is the oracle's."""
    import oracle
    import torch
    from paper_2210_03211_gb300 import lazyfox
    src, dst = graph()
    ref = oracle.OracleGraph(src, dst).run(1, -np.inf, 2, rule="literal")
    made = {}
    for per_queue in (None, True):
        alloc = lazyfox.CountingAllocator(torch.device("cuda", torch.cuda.current_device()))
        with lazyfox.Graph(src, dst, gain_rule="literal", member_slots=32, allocator=alloc,
                           per_queue_launches=per_queue) as g:
            before = alloc.calls
            st = g.run(1, -np.inf, 2)
            made[per_queue] = alloc.calls - before
            assert np.array_equal(st.wcc_history, ref["T"])
            assert np.array_equal(st.joins, ref["joins"]) and np.array_equal(st.leaves, ref["leaves"])
        assert alloc.live == 0
    # the loop's own: its barrier flags and one area of global tables
    assert made[None] <= made[True] - 13 + 2, made


@pytest.mark.parametrize("q", [2, 64, 300])
def test_longer_queues_are_launched_where_the_loop_is_preferred(q):
    """Above one node the loop's grid barriers cost more than launches: preferring it
    launches every queue all the same (the loop is one launch an iteration), and the
    run is the same."""
    from paper_2210_03211_gb300 import lazyfox
    src, dst = graph()
    runs = []
    for per_queue in (False, True):
        with lazyfox.Graph(src, dst, gain_rule="literal", profile=True, per_queue_launches=per_queue) as g:
            runs.append(g.run(q, -np.inf, 3))
        assert runs[-1].prof_move_launches == runs[-1].num_batches, per_queue
    assert np.array_equal(runs[0].wcc_history, runs[1].wcc_history)


@pytest.mark.parametrize("rule", ["literal", "meanfield"])
@pytest.mark.parametrize("q", [2, 40, 700])
def test_loop_of_many_blocks_with_the_central_barrier(rule, q):
    """Several blocks meet at grid barriers that block 0 gathers and releases: the
    oracle's run."""
    import oracle
    from paper_2210_03211_gb300 import lazyfox
    src, dst = graph()
    og = oracle.OracleGraph(src, dst)
    ref = og.run(q, -np.inf, 3, rule=rule)
    with lazyfox.Graph(src, dst, gain_rule=rule, barrier_mode=1, per_queue_launches=False, profile=True) as g:
        st = g.run(q, -np.inf, 3)
        assert st.prof_move_launches == st.iterations   # the loop: one launch an iteration
        assert np.array_equal(st.wcc_history, ref["T"])
        assert np.array_equal(st.joins, ref["joins"]) and np.array_equal(st.leaves, ref["leaves"])
        s, o = g.state(), og.state()
        for key in ("mem_off", "mem_ids", "n", "m", "vol"):
            assert np.array_equal(s[key], o[key]), key


@pytest.mark.parametrize("mode", [0, 1])
def test_handle_is_usable_after_a_timeout(mode):
    """A block that never arrives ends the run with LF_ERR_TIMEOUT in either barrier
    mode.  The same handle then runs at queue size 1, where one block meets nobody:
    nothing of the abandoned run is left over."""
    import oracle
    from paper_2210_03211_gb300 import lazyfox
    src, dst = graph()
    ref = oracle.OracleGraph(src, dst).run(1, 0.01, 3, rule="literal")
    with lazyfox.Graph(src, dst, gain_rule="literal", inject_barrier_stall=True, barrier_timeout_ms=50,
                       barrier_mode=mode, per_queue_launches=False) as g:
        for _ in range(2):
            with pytest.raises(lazyfox.LazyFoxError) as e:
                g.run(64, 0.01, 3)
            assert e.value.status == lazyfox.LF_ERR_TIMEOUT
            st = g.run(1, 0.01, 3)
            assert np.array_equal(st.wcc_history, ref["T"])
            assert np.array_equal(st.joins, ref["joins"]) and np.array_equal(st.leaves, ref["leaves"])
