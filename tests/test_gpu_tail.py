"""Runs of small layers in one cluster launch (k_tail): graphs past the
one-launch size whose layers cross its limits -- a block's share of a layer
(dealt out again) and the largest layer it takes (back to the round kernel and
in again) -- against the oracle, bit for bit, in both loop modes."""
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


def _check(edges, m, general=False):
    want = (oracle.peel_rounds_general if general else oracle.peel_rounds)(edges, m)
    e = torch.from_numpy(np.ascontiguousarray(edges).view(np.int32)).cuda()
    a = hp.peel_async(e, m, general=general)
    for host in (0, 1):
        hp.set_tuning(host_round_loop=host)
        try:
            got = hp.peel(e, m, general=general)
        finally:
            hp.set_tuning()
        assert np.array_equal(got.order.cpu().numpy().view(np.uint32), want.order)
        assert np.array_equal(got.claim.cpu().numpy().view(np.uint32), want.claim)
        assert got.rounds == want.rounds and got.n_peeled == want.n_peeled
    st = hp.stats_from_device(a.stats)
    assert np.array_equal(a.order.cpu().numpy().view(np.uint32), want.order)
    for f in ("first_layer", "frontier", "rounds", "n_peeled"):
        assert st[f] == got.stats[f], f
    return want


def _trees(roots, depth, stubs, filler):
    """`roots` binary trees of edges that peel level by level from their roots,
    `stubs` edges that peel in round 0 and free nothing, and a core the leaves
    and stubs hang on: part-0 ids of the roots come first, so round 0 lists
    them next to each other.  Level t holds roots * 2^t edges."""
    fresh = [roots + stubs, 0, 0]  # next unused id of each part
    rows, level = [], [(0, i) for i in range(roots)]  # (part, id) each edge hangs from
    for d in range(depth):
        nxt = []
        for p, v in level:
            row = [0, 0, 0]
            row[p] = v
            for q in range(3):
                if q == p:
                    continue
                if d == depth - 1:
                    row[q] = -1  # a core vertex
                else:
                    row[q] = fresh[q]
                    nxt.append((q, fresh[q]))
                    fresh[q] += 1
            rows.append(row)
        level = nxt
    rows += [[roots + i, -1, -1] for i in range(stubs)]
    core = list(fresh)
    e = np.array(rows, dtype=np.int64)
    for q in range(3):
        e[e[:, q] < 0, q] = core[q]
    f = np.arange(filler)
    pad = np.stack([core[q] + f // 2 for q in range(3)], axis=1)  # every core edge twice
    e = np.concatenate([e, pad])
    P = int(max(core[q] + filler // 2 + 1 for q in range(3)))
    return (e + np.arange(3) * P).astype(np.uint32), 3 * P


def test_tail_deals_a_lopsided_layer_out_again_and_hands_a_large_one_back():
    # L_0: 2,000 roots next to each other among 30,000 stubs, so one block of
    # sixteen holds nearly all roots; L_5 = 64,000 is past the cluster kernel
    e, m = _trees(2000, 6, 30_000, 4_000)
    rng = np.random.default_rng(1)
    want = _check(e, m)
    assert want.rounds == 6
    _check(e[rng.permutation(len(e))], m)


@pytest.mark.parametrize("n,gamma,r", [(150_000, 1222, 3), (150_000, 1300, 4), (140_000, 2300, 2),
                                       (150_000, 1100, 3), (1_000_000, 1230, 3)])
def test_tail_random_graphs(n, gamma, r):
    m = oracle.num_vertices(n, gamma, r)
    _check(oracle.hash_edges(inputs.keys(n, 15), m, r, 1), m)


@pytest.mark.parametrize("n,gamma,r", [(150_000, 1230, 3), (140_000, 1400, 4)])
def test_tail_general_graphs(n, gamma, r):
    m = (n * gamma + 999) // 1000
    _check(oracle.hash_edges_general(inputs.keys(n, 16), m, r, 1), m, general=True)


@pytest.mark.parametrize("n", [140_000, 1_000_000])
@pytest.mark.parametrize("host", [0, 1])
def test_assignment_of_small_and_large_layers(n, host):
    # runs of layers in one cluster launch, larger ones by one grid each
    keys = inputs.keys(n, 23)
    dk = torch.from_numpy(keys.view(np.int64)).cuda()
    want = oracle.mphf_build(keys, seed=1, max_tries=16)
    vals = (inputs.keys(n, 24) % np.uint64(1000)).astype(np.uint32)
    dv = torch.from_numpy(vals.view(np.int32)).cuda()
    sf = oracle.sf_build(keys, vals, 1000, seed=1, max_tries=16)
    hp.set_tuning(host_round_loop=host)
    try:
        got = hp.mphf_build(dk, max_tries=16)
        gsf = hp.sf_build(dk, dv, 1000, max_tries=16)
        G, D, _ = hp.mphf_build_async(dk, max_tries=16)
        U, _ = hp.sf_build_async(dk, dv, 1000, max_tries=16)
    finally:
        hp.set_tuning()
    for g, d in ((got.G, got.rank_dir), (G, D)):
        assert np.array_equal(g.cpu().numpy().view(np.uint64), want.G)
        assert np.array_equal(d.cpu().numpy().view(np.uint64), want.dir)
    for u in (gsf.U, U[:len(sf.U)]):
        assert np.array_equal(u.cpu().numpy().view(np.uint64), sf.U)
