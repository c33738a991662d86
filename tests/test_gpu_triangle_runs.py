"""Triangle counts where the source-vertex kernels share out their work: enough nodes
that warps take runs of them from a counter (and one node fewer), mean out-degrees on
both sides of the lines between the flat kernel, the hash kernel and the
middle-vertex kernels, and triangles that nearly all close on a few nodes, whose credits
are added up within a warp.  Integers, compared with the oracle exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

COUNTER_FROM = 4 * 8 * 6 * 152   # nodes


def cliques(k, count, spare=0):
    iu, ju = np.triu_indices(k, 1)
    base = np.repeat(k * np.arange(count), iu.shape[0])
    at = k * count
    return (np.concatenate([base + np.tile(iu, count), at + 2 * np.arange(spare)]),
            np.concatenate([base + np.tile(ju, count), at + 1 + 2 * np.arange(spare)]))


def clique_of_hubs(hubs, leaves):
    iu, ju = np.triu_indices(hubs, 1)
    return (np.concatenate([iu, np.repeat(np.arange(hubs), leaves)]),
            np.concatenate([ju, np.tile(hubs + np.arange(leaves), hubs)]))


def skewed(n, mean):
    rng = np.random.default_rng(mean)
    x = lambda: (n * rng.random(n * mean) ** 3).astype(np.int64)   # noqa: E731
    return x(), x()


GRAPHS = {
    "cliques_of_13_mean_6": lambda: cliques(13, 2300),
    "cliques_of_14": lambda: cliques(14, 2100),
    "cliques_of_19_just_below": lambda: cliques(19, COUNTER_FROM // 19 - 1, (COUNTER_FROM % 19 + 19 - 1) // 2),
    "cliques_of_20": lambda: cliques(20, 1600),
    "cliques_of_33_and_pairs": lambda: cliques(33, 900, 40),
    "cliques_of_130": lambda: cliques(130, 230),
    "two_hubs": lambda: clique_of_hubs(2, 40000),
    "nine_hubs": lambda: clique_of_hubs(9, 31000),
    "forty_hubs": lambda: clique_of_hubs(40, 3000),
    "one_hub_of_triangles": lambda: (np.concatenate([np.zeros(60000), 1 + 2 * np.arange(30000)]),
                                     np.concatenate([1 + np.arange(60000), 2 + 2 * np.arange(30000)])),
    "skewed_mean_7": lambda: skewed(31000, 8),
    "skewed_mean_20": lambda: skewed(31000, 22),
}


@pytest.mark.parametrize("name", GRAPHS)
def test_triangles_by_runs(name):
    import torch

    import oracle
    from paper_2210_03211_gb300 import lazyfox
    src, dst = (a.astype(np.int32) for a in GRAPHS[name]())
    t, vt, cc = oracle.OracleGraph(src, dst).node_stats()
    with lazyfox.Graph(src, dst) as g:
        gt, gvt, gcc = g.node_stats()
        off, adj = g.oriented()
        total = g.create_stats()["num_triangles"]
    assert np.array_equal(gt, t) and np.array_equal(gvt, vt) and gcc == cc and 3 * total == t.sum()
    o, a = torch.from_numpy(off).cuda(), torch.from_numpy(adj).cuda()
    nt = torch.empty(t.shape[0], dtype=torch.int64, device="cuda")
    nvt = torch.empty(t.shape[0], dtype=torch.int32, device="cuda")
    for _ in range(2):   # the counter starts anew
        lazyfox.lf_triangles_noalloc(o, a, nt, nvt)
        assert np.array_equal(nt.cpu().numpy(), t) and np.array_equal(nvt.cpu().numpy(), vt)
