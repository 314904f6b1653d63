"""hinge_moves of graphs peeled in one launch (small.cu): the claims of a round are
not ordered there, and every edge that two or more of its vertices claim in its
round counts, once."""
import numpy as np
import pytest

import oracle
from paper_1312_0526_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1312_0526_gb300 as hp  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1312_0526_gb300 import build
    build.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _dev(a, dtype):
    return torch.from_numpy(np.ascontiguousarray(a).view(dtype)).cuda()


def _claimed_twice(edges, claim):
    """Edges that have two or more vertices of degree 1 in their round."""
    rounds = np.where(claim == 0xFFFFFFFF, 1 << 30, claim >> 2).astype(np.int64)
    deg = np.bincount(edges.ravel(), minlength=int(edges.max()) + 1)
    total = 0
    for t in range(int(rounds[rounds < (1 << 30)].max(initial=-1)) + 1):
        layer = rounds == t
        total += int(((deg[edges[layer]] == 1).sum(axis=1) >= 2).sum())
        np.subtract.at(deg, edges[layer].ravel(), 1)
    return total


def _stats(e, m, general):
    a = hp.peel_async(e, m, max_layers=1 << 17, general=general)
    torch.cuda.synchronize()
    return (hp.peel(e, m, max_layers=1 << 17, general=general).stats["hinge_moves"],
            hp.stats_from_device(a.stats)["hinge_moves"])


# one, four and sixteen edges per thread, one block and a cluster
# (parts of more than 2^16 vertices, as of 100,003 edges at r = 2, go the general path)
@pytest.mark.parametrize("n,gamma,r", [(n, g, r) for g, r in ((1230, 3), (1300, 4), (2300, 2))
                                       for n in (1000, 4000, 12_000, 100_003 if r > 2 else 50_003)])
def test_small_hinge_moves(n, gamma, r):
    m = oracle.num_vertices(n, gamma, r)
    total = 0
    for seed in range(1, 6):
        edges = oracle.hash_edges(inputs.keys(n, 60 + seed), m, r, 1)
        want = _claimed_twice(edges.astype(np.int64), oracle.peel_rounds(edges, m).claim)
        assert _stats(_dev(edges, np.int32), m, False) == (want, want)
        total += want
    assert total > 0


@pytest.mark.parametrize("n", [1000, 4000, 9000, 60_000])
@pytest.mark.parametrize("r", [2, 3, 4])
def test_small_hinge_moves_count_an_edge_once(n, r):
    # disjoint rows: all r vertices claim theirs, in round 0
    edges = np.stack([np.arange(n) + n * (r - 1 - j) for j in range(r)], axis=1).astype(np.uint32)
    assert _stats(_dev(edges, np.int32), r * n, True) == (n, n)


@pytest.mark.parametrize("n", [4000, 100_003])
def test_small_build_hinge_moves(n):
    keys = inputs.keys(n, 4)
    dk = _dev(keys, np.int64)
    m = oracle.num_vertices(n, 1230, 3)
    for build in (lambda: hp.mphf_build(dk, max_tries=64).stats,
                  lambda: hp.stats_from_device(hp.mphf_build_async(dk, max_tries=64)[2]),
                  lambda: hp.sf_build(dk, _dev(np.zeros(n, np.uint32), np.int32), 3,
                                      max_tries=64).stats):
        st = build()
        edges = oracle.hash_edges(keys, m, 3, st["seed_used"])
        want = _claimed_twice(edges.astype(np.int64), oracle.peel_rounds(edges, m).claim)
        assert st["hinge_moves"] == want > 0
