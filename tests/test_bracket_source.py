"""The bracket of the paper's gain, |X - gain| <= E, on the arithmetic that runs: member
sums, stored factors, corrections and bracket are the functions of the CUDA source,
compiled for the CPU, against the oracle's exactly summed gain.  Where every term
after the move is zero the bracket is replaced by X = -WCC-hat(C), E = 0, which drops
the candidate: then the gain must not be positive.  Paper passages: Heuristic Counting
of Triangles (the estimator), the WCC-hat sum equations, Node Changes (Joining /
Leaving a Community)."""
import ctypes as C

import numpy as np
import pytest

from device_source import build
from test_bracket_bounds import oracle_gain, random_case

f32 = np.float32


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    lib = build(tmp_path_factory.mktemp("bracket"),
                ["lit_h32", "lit_g32", "lit_screen", "lit_g3", "lit_fsum_factor", "lit_fsum_store"],
                ["OWN_FLAG", "CNT_MASK"], """
extern "C" float h32(int own, uint32_t k, uint32_t d, uint32_t n) { return lit_h32(own != 0, k, d, n); }
extern "C" void bracket(int32_t n, uint32_t m2, double cc, const int32_t *k, const int32_t *d, int own, uint32_t xk,
                        int32_t xd, float hs, float *out) {
    CommRec c{n, m2, 0u, 0};
    float litF[8] = {};
    RunArgs a{&c, litF, nullptr, cc};
    double f0 = 0.0, f1 = 0.0, f2 = 0.0;
    for (int32_t i = 0; i < n; ++i) lit_g3(k[i], d[i], n, f0, f1, f2);
    for (int t = 0; t < 3; ++t)
        lit_fsum_store(a, 0, t, lit_fsum_factor(a, int4{n, (int)m2, 0, 0}, t), f0, f1, f2);
    lit_screen(a, 0, xk | (own ? OWN_FLAG : 0u), xd, hs, out[0], out[1]);
}
""")
    lib.h32.restype = C.c_float
    return lib


def bracket(dev, members, nbrs, x_k, x_d, own, cc, rng):
    """X and E of a case of test_bracket_bounds: members (k, d, count), x's neighbours
    in C as indices of them, sums in a random order."""
    n = sum(c for _, _, c in members)
    m2 = sum(k * c for k, _, c in members)
    reps = [c for _, _, c in members]
    order = rng.permutation(n)
    k = np.ascontiguousarray(np.repeat([m[0] for m in members], reps)[order], np.int32)
    d = np.ascontiguousarray(np.repeat([m[1] for m in members], reps)[order], np.int32)
    hs = f32(0)
    for i in rng.permutation(len(nbrs)):
        ky, dy, _ = members[nbrs[i]]
        hs = f32(hs + f32(dev.h32(int(own), ky, dy, n)))
    out = (C.c_float * 2)()
    p = C.POINTER(C.c_int32)
    dev.bracket(n, C.c_uint32(m2), C.c_double(cc), k.ctypes.data_as(p), d.ctypes.data_as(p), int(own),
                C.c_uint32(x_k), x_d, C.c_float(hs), out)
    return out[0], out[1]


def check(dev, oracle_lib, members, nbrs, x_k, x_d, own, cc, rng):
    want = oracle_gain(oracle_lib, members, nbrs, x_k, x_d, own, cc)
    X, E = bracket(dev, members, nbrs, x_k, x_d, own, cc, rng)
    case = (members, nbrs, x_k, x_d, own, cc, X, E, want)
    assert np.isfinite(X) and np.isfinite(E), case
    if E == 0.0:    # every term after the move is zero
        assert want <= 0.0, case
        assert abs(X - want) <= 2.0 ** -23 * abs(want), case   # one stored float, summed in FP64
    else:
        assert abs(X - want) <= E, case
    return E == 0.0


@pytest.mark.parametrize("big", [False, True], ids=["small_communities", "communities_up_to_240k"])
def test_bracket_of_the_source_holds(dev, oracle_lib, big):
    rng = np.random.default_rng(41 + int(big))
    for _ in range(1500 if not big else 300):
        members, nbrs, x_k, x_d, own = random_case(rng, big)
        cc = float(rng.choice([1.0, 0.5, 0.13, 1e-3, 3e-7]))
        check(dev, oracle_lib, members, nbrs, x_k, x_d, own, cc, rng)


def zero_cases():
    """(members, neighbours, x_k, x_d, own, whether every term after the move is zero)."""
    out = []
    for d in (1, 2, 3, 7, 50):
        # leaving: the only member; a pair; the middle of a path of three; the centre of a star
        out.append(([(0, d, 1)], [], 0, d, True, True))
        out.append(([(1, d, 1), (1, 3, 1)], [1], 1, d, True, True))
        for leaves in (2, 3, 12, 200):
            if d >= leaves:
                out.append(([(leaves, d, 1)] + [(1, 4, 1)] * leaves, list(range(1, leaves + 1)), leaves, d, True, True))
        # leaving a community of pairs (nobody has two neighbours inside): F(n-1) = 0 though edges stay
        out.append(([(1, d, 1), (1, 3, 1), (1, 2, 6)], [1], 1, d, True, True))
        # leaving a triangle with tails: a pair stays, with no member of two neighbours; then a path of three stays
        if d >= 2:
            out.append(([(2, d, 1), (2, 3, 1), (2, 3, 1)], [1, 2], 2, d, True, False))
        out.append(([(1, d, 1), (2, 4, 1), (2, 4, 1), (1, 3, 1)], [1], 1, d, True, False))
        # joining: a single node, a node of a pair, both nodes of a pair, the middle of a path of three
        out.append(([(0, 3, 1)], [0], 1, d, False, True))
        out.append(([(1, 3, 1), (1, 4, 1)], [0], 1, d, False, False))
        out.append(([(1, 1, 1), (1, 4, 1)], [1], 1, d, False, False))
        if d >= 2:
            out.append(([(1, 3, 1), (1, 4, 1)], [0, 1], 2, d, False, False))
        out.append(([(1, 3, 1), (2, 4, 1), (1, 2, 1)], [1], 1, d, False, False))
        # joining a community without edges through several members: only x's own term is left
        if d >= 3:
            out.append(([(0, 5, 1), (0, 6, 1), (0, 2, 1), (0, 9, 4)], [0, 1, 2], 3, d, False, False))
    return out


@pytest.mark.parametrize("cc", [1.0, 0.13, 1e-3, 3e-7])
def test_candidates_without_a_term_after_the_move(dev, oracle_lib, cc):
    rng = np.random.default_rng(7)
    for members, nbrs, x_k, x_d, own, zero in zero_cases():
        fired = check(dev, oracle_lib, members, nbrs, x_k, x_d, own, cc, rng)
        assert fired == zero, (members, nbrs, x_k, x_d, own)
