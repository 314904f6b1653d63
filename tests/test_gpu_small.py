"""Small graphs in one launch (small.cu): the edges of its forms -- 1, 4 and 16
edges per thread, one block and a cluster -- against the oracle, bit for bit,
and the vertex degrees its 32-bit records cannot hold."""
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


def _dev32(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).cuda()


def _dev64(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int64)).cuda()


def _check(edges, m, general=False):
    want = (oracle.peel_rounds_general if general else oracle.peel_rounds)(edges, m)
    e = _dev32(edges)
    got = hp.peel(e, m, max_layers=1 << 17, general=general)
    a = hp.peel_async(e, m, max_layers=1 << 17, general=general)
    torch.cuda.synchronize()
    st = hp.stats_from_device(a.stats)
    R = want.rounds
    for order, claim, loff in ((got.order, got.claim, got.layer_off),
                               (a.order, a.claim, a.layer_off)):
        assert np.array_equal(order.cpu().numpy().view(np.uint32), want.order)
        assert np.array_equal(claim.cpu().numpy().view(np.uint32), want.claim)
        assert np.array_equal(loff[:R + 1].cpu().numpy().astype(np.uint64),
                              want.layer_off[:R + 1].astype(np.uint64))
    assert got.rounds == R == st["rounds"] and got.n_peeled == want.n_peeled == st["n_peeled"]
    hp.set_tuning(host_round_loop=1)  # the general path: same counts
    try:
        ref = hp.peel(e, m, max_layers=1 << 17, general=general)
    finally:
        hp.set_tuning()
    for f in ("first_layer", "frontier", "core_nonempty"):
        assert got.stats[f] == ref.stats[f] == st[f], f


# one, four and sixteen edges per thread; one block and (from about 13,000
# edges) a cluster; the largest graph of the route and the first past it
SIZES = [1, 31, 33, 1023, 1024, 1025, 4096, 4097, 12_800, 13_900, 100_003, 131_072, 131_073]


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("gamma,r", [(1230, 3), (1100, 3), (1300, 4), (2300, 2)])
def test_small_peel(n, gamma, r):
    m = oracle.num_vertices(n, gamma, r)
    _check(oracle.hash_edges(inputs.keys(n, 5), m, r, 1), m)


@pytest.mark.parametrize("n", [1, 33, 1025, 4097, 9_000, 30_000])
@pytest.mark.parametrize("gamma,r", [(1230, 3), (1500, 4), (2300, 2)])
def test_small_general_peel(n, gamma, r):
    m = (n * gamma + 999) // 1000
    _check(oracle.hash_edges_general(inputs.keys(n, 8), m, r, 1), m, general=True)


def test_small_peel_sparse_parts():
    # far more vertices than edges, up to parts of 2^16 and past them
    for P in (3000, 65_536, 65_537):
        rng = np.random.default_rng(P)
        e = np.stack([rng.integers(0, P, 500) + j * P for j in range(3)], axis=1)
        _check(e.astype(np.uint32), 3 * P)


@pytest.mark.parametrize("n", [40_000, 100_000])
def test_small_peel_degree_past_15_bits(n):
    # every edge shares a vertex; half of them also hang on vertices of their own
    P = n
    rng = np.random.default_rng(n)
    e = np.stack([np.zeros(n, np.int64), P + rng.integers(0, n // 2, n),
                  2 * P + rng.permutation(n)], axis=1) if n <= 65_536 else \
        np.stack([np.zeros(n, np.int64), 60_000 + rng.integers(0, 60_000, n),
                  120_000 + rng.integers(0, 60_000, n)], axis=1)
    _check(e.astype(np.uint32), 3 * P if n <= 65_536 else 180_000)


def test_small_general_degree_past_15_bits_in_one_block():
    n = 11_000  # rows of one vertex three times: 33,000 incidences, no edge peels
    e = np.zeros((n, 3), np.uint32)
    e[:1000, 0] = 1 + np.arange(1000)
    _check(e, 2000, general=True)


@pytest.mark.parametrize("n", [1, 3, 1000, 1025, 4097, 12_800, 13_900, 131_072, 131_073])
def test_small_builds(n):
    keys = inputs.keys(n, 4)
    want = oracle.mphf_build(keys, seed=1, max_tries=64)
    dk = _dev64(keys)
    order = torch.empty(n, dtype=torch.int32, device="cuda")
    got = hp.mphf_build(dk, seed=1, max_tries=64, order=order)
    assert got.stats["seed_used"] == want.seed_used
    G, D, st = hp.mphf_build_async(dk, seed=1, max_tries=64)
    for g, d in ((got.G, got.rank_dir), (G, D)):
        assert np.array_equal(g.cpu().numpy().view(np.uint64), want.G)
        assert np.array_equal(d.cpu().numpy().view(np.uint64), want.dir)
    m = oracle.num_vertices(n, 1230, 3)
    peel = oracle.peel_rounds(oracle.hash_edges(keys, m, 3, want.seed_used), m)
    assert np.array_equal(order.cpu().numpy().view(np.uint32), peel.order)
    for sigma in (2, 1000, 1 << 32):
        vals = (inputs.keys(n, 9) % np.uint64(sigma)).astype(np.uint32)
        sf = oracle.sf_build(keys, vals, sigma, seed=1, max_tries=64)
        sg = hp.sf_build(dk, _dev32(vals), sigma, seed=1, max_tries=64)
        assert np.array_equal(sg.U.cpu().numpy().view(np.uint64), sf.U)


def test_small_build_seeds_past_one_launch():
    keys = np.concatenate([inputs.keys(500, 3)] * 2)  # duplicates never peel
    for fn in (lambda: hp.mphf_build(_dev64(keys), max_tries=130),
               lambda: hp.sf_build(_dev64(keys), _dev32(np.zeros(1000, np.uint32)), 3,
                                   max_tries=130)):
        with pytest.raises(hp.HpeelError, match="RETRIES_EXHAUSTED.*seeds 1..130"):
            fn()


@pytest.mark.parametrize("n", [1, 3, 100, 330, 341, 350, 416, 417, 1000, 4097, 200_003])
def test_lookup_sectors_equal_the_word_path(n):
    # the sector form needs a 32-byte aligned G; an unaligned copy takes the
    # word form: equal on the set (a bijection) and on other keys, whatever the
    # last block holds
    keys = inputs.keys(n, 27)
    dk = _dev64(keys)
    b = hp.mphf_build(dk, max_tries=64)
    seed = b.stats["seed_used"]
    odd = torch.empty(b.G.numel() + 4, dtype=torch.int64, device="cuda")
    other = _dev64(inputs.keys(20_000, 28))
    got = hp.mphf_lookup(dk, seed, b.m, b.G, b.rank_dir).cpu().numpy()
    assert np.array_equal(np.sort(got), np.arange(n))
    for q in (dk, other):
        a = hp.mphf_lookup(q, seed, b.m, b.G, b.rank_dir)
        for shift in (1, 2, 3):
            G = odd[shift:shift + b.G.numel()]
            G.copy_(b.G)
            assert torch.equal(a, hp.mphf_lookup(q, seed, b.m, G, b.rank_dir))


@pytest.mark.parametrize("m", [1, 2, (1 << 31) - 1, 1 << 31, (1 << 31) + 1, (1 << 32) - 1])
def test_remainders_about_2_to_the_31(m):
    # hashes into [0, m): the 32-bit and the 64-bit form of the remainder
    keys = np.concatenate([inputs.keys(20_000, 31), np.arange(64, dtype=np.uint64),
                           ~np.arange(64, dtype=np.uint64)])
    got = hp.hash_edges(_dev64(keys), m, 3, 1, general=True).cpu().numpy().view(np.uint32)
    assert np.array_equal(got, oracle.hash_edges_general(keys, m, 3, 1))
