"""Triangle counts where the paths of the source-vertex kernels meet: out-degrees
around the flat path's limit (32) and the warp path's (128), node runs that start
anywhere in a warp, and mean degrees on both sides of the line at which
lf_graph_create changes to the middle-vertex kernels.  Integers, compared with
the oracle exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def cliques_and_pairs(sizes, pairs, lead):
    """Disjoint cliques (a clique of k+1 nodes holds out-degrees k, k-1, ..., 0)
    behind `lead` single edges, and `pairs` single edges after them."""
    src, dst, at = [], [], 0
    for _ in range(lead):
        src.append(at), dst.append(at + 1)
        at += 2
    for k in sizes:
        iu, ju = np.triu_indices(k, 1)
        src.extend((at + iu).tolist())
        dst.extend((at + ju).tolist())
        at += k
    for _ in range(pairs):
        src.append(at), dst.append(at + 1)
        at += 2
    return np.array(src, np.int32), np.array(dst, np.int32)


@pytest.mark.parametrize("pairs", [0, 3000])          # mean out-degree above and below 10
@pytest.mark.parametrize("lead", [0, 1, 16])
@pytest.mark.parametrize("sizes", [(2, 3), (32, 33, 34), (128, 129, 130), (3, 33, 65, 33, 130, 4)])
def test_triangles_at_the_path_limits(sizes, lead, pairs):
    import torch

    import oracle
    from paper_2210_03211_gb300 import lazyfox
    src, dst = cliques_and_pairs(sizes, pairs, lead)
    t, vt, cc = oracle.OracleGraph(src, dst).node_stats()
    with lazyfox.Graph(src, dst) as g:
        gt, gvt, gcc = g.node_stats()
        off, adj = g.oriented()
        total = g.create_stats()["num_triangles"]
    assert np.array_equal(gt, t) and np.array_equal(gvt, vt) and gcc == cc and 3 * total == t.sum()
    o, a = torch.from_numpy(off).cuda(), torch.from_numpy(adj).cuda()
    nt = torch.empty(t.shape[0], dtype=torch.int64, device="cuda")
    nvt = torch.empty(t.shape[0], dtype=torch.int32, device="cuda")
    lazyfox.lf_triangles_noalloc(o, a, nt, nvt)
    assert np.array_equal(nt.cpu().numpy(), t) and np.array_equal(nvt.cpu().numpy(), vt)
