"""The general path where graphs of up to 131,072 edges take the one-launch path
by default: caller-captured and cached graphs on new contents, peels of
thousands of rounds (the runs of small layers and the order sort's later
passes), and the error outcomes.  Either the graph is larger, or the tuning asks
for the L2-blocked build, which keeps any graph on the general path."""
import numpy as np
import pytest

import oracle
from paper_1312_0526_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1312_0526_gb300 as hp  # noqa: E402

DONE, EXHAUSTED, DEVICE_ERROR, LAYERS_FULL = 1, 2, 3, 4
LARGE, BLOCKED = 150_000, 30_000


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1312_0526_gb300 import build
    build.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.fixture(params=["large", "blocked"])
def n(request):
    if request.param == "blocked":
        hp.set_tuning(bucket_shift=10, bucket_min_vertices=0)
    yield LARGE if request.param == "large" else BLOCKED
    hp.set_tuning()


@pytest.fixture
def blocked():
    hp.set_tuning(bucket_min_vertices=0)
    yield
    hp.set_tuning()


def _dev32(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).cuda()


def _dev64(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int64)).cuda()


def _u32(t):
    return t.cpu().numpy().view(np.uint32)


def _u64(t):
    return t.cpu().numpy().view(np.uint64)


def _captured(call):
    g = torch.cuda.CUDAGraph()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        with torch.cuda.graph(g, stream=s):
            call()
    torch.cuda.synchronize()
    return g.replay


def _same_peel(got, want):
    torch.cuda.synchronize()
    st = hp.stats_from_device(got.stats)
    assert st["async_status"] == DONE and st["device_err"] == 0
    assert st["rounds"] == want.rounds and st["n_peeled"] == want.n_peeled
    assert np.array_equal(_u32(got.order), want.order)
    assert np.array_equal(_u32(got.claim), want.claim)
    assert np.array_equal(_u64(got.layer_off[:want.rounds + 1]),
                          want.layer_off[:want.rounds + 1].astype(np.uint64))
    return st


@pytest.mark.parametrize("captured", [False, True], ids=["cached", "captured"])
def test_mphf_build_async_replayed_on_new_keys(n, captured):
    k = _dev64(inputs.keys(n, 31))
    ws = torch.empty(hp.mphf_workspace_size(n), dtype=torch.uint8, device="cuda")
    G, D, st = hp.mphf_build_async(k, seed=1, max_tries=32, workspace=ws)
    torch.cuda.synchronize()
    again = lambda: hp.mphf_build_async(k, seed=1, max_tries=32, workspace=ws,  # noqa: E731
                                        G=G, rank_dir=D, stats=st)
    if captured:
        again = _captured(again)
    # the third set's duplicates never peel
    twice = np.concatenate([inputs.keys(n - n // 2, 34), inputs.keys(n // 2, 34)])
    for keys in (inputs.keys(n, 32), inputs.keys(n, 33), twice, inputs.keys(n, 35)):
        k.copy_(_dev64(keys))
        G.fill_(-1)
        again()
        torch.cuda.synchronize()
        got = hp.stats_from_device(st)
        if keys is twice:
            assert got["async_status"] == EXHAUSTED and got["attempts"] == 32
            continue
        want = oracle.mphf_build(keys, seed=1, max_tries=32)
        assert got["async_status"] == DONE and got["seed_used"] == want.seed_used
        assert np.array_equal(_u64(G), want.G) and np.array_equal(_u64(D), want.dir)


@pytest.mark.parametrize("captured", [False, True], ids=["cached", "captured"])
@pytest.mark.parametrize("general", [False, True])
def test_peel_async_replayed_on_new_edges(n, captured, general):
    m = oracle.num_vertices(n, 1230, 3)
    hashed = oracle.hash_edges_general if general else oracle.hash_edges
    peeled = oracle.peel_rounds_general if general else oracle.peel_rounds
    graphs = [hashed(inputs.keys(n, s), m, 3, 1) for s in (21, 22)]
    if not general:
        # vertices crowded at the start of each part: a blocked build's buckets
        # overflow, and the graph does the build and the rounds over
        rng = np.random.default_rng(9)
        graphs.append(np.stack([rng.integers(0, 1024, n) + j * (m // 3) for j in range(3)],
                               axis=1).astype(np.uint32))
    de = _dev32(graphs[0])
    ws = torch.empty(hp.peel_workspace_size(n, m, 3, general), dtype=torch.uint8, device="cuda")
    out = hp.peel_async(de, m, workspace=ws, general=general)
    torch.cuda.synchronize()
    again = lambda: hp.peel_async(de, m, workspace=ws, out=out, general=general)  # noqa: E731
    if captured:
        again = _captured(again)
    for e in graphs[1:] + graphs[:1]:
        de.copy_(_dev32(e))
        out.order.fill_(-1)
        again()
        _same_peel(out, peeled(e, m))


@pytest.mark.parametrize("captured", [False, True], ids=["cached", "captured"])
def test_sf_build_async_replayed_on_new_values(n, captured):
    sigma = 1000
    keys = inputs.keys(n, 45)
    vals = [(inputs.keys(n, s) % np.uint64(sigma)).astype(np.uint32) for s in (1, 2, 3)]
    dk, dv = _dev64(keys), _dev32(vals[0])
    ws = torch.empty(hp.sf_workspace_size(n), dtype=torch.uint8, device="cuda")
    U, st = hp.sf_build_async(dk, dv, sigma, max_tries=32, workspace=ws)
    torch.cuda.synchronize()
    again = lambda: hp.sf_build_async(dk, dv, sigma, max_tries=32, workspace=ws,  # noqa: E731
                                      U=U, stats=st)
    if captured:
        again = _captured(again)
    bad = vals[1].copy()
    bad[n // 2] = sigma
    for v in (vals[1], bad, vals[2]):
        dv.copy_(_dev32(v))
        again()
        torch.cuda.synchronize()
        got = hp.stats_from_device(st)
        if v is bad:
            assert got["async_status"] == DEVICE_ERROR and got["device_err"] == 7
            continue
        want = oracle.sf_build(keys, v, sigma, seed=1, max_tries=32)
        assert got["async_status"] == DONE and got["seed_used"] == want.seed_used
        assert np.array_equal(_u64(U[:len(want.U)]), want.U)


# ----------------------------------------------------- thousands of rounds --

def _chain(n):
    """A band-shaped 3-hypergraph that peels from its two ends, a few edges per
    round."""
    i = np.arange(n)
    e = np.stack([(i + 1) // 2, n + i // 2, 2 * n + 2 * (i // 4) + i % 2], axis=1)
    return e.astype(np.uint32), 3 * n


@pytest.mark.parametrize("n_edges", [1203, 2500, 12_000])
def test_chain_on_the_general_path(blocked, n_edges):
    e, m = _chain(n_edges)
    want = oracle.peel_rounds(e, m)
    assert want.rounds > 300
    d = _dev32(e)
    _same_peel(hp.peel_async(d, m, max_layers=8192), want)
    for host in (0, 1):
        hp.set_tuning(bucket_min_vertices=0, host_round_loop=host)
        got = hp.peel(d, m, max_layers=8192)
        assert got.rounds == want.rounds
        assert np.array_equal(_u32(got.order), want.order)
        assert np.array_equal(_u32(got.claim), want.claim)


def test_chain_past_the_one_launch_size():
    e, m = _chain(140_000)
    want = oracle.peel_rounds(e, m)
    assert want.rounds > 50_000
    d = _dev32(e)
    _same_peel(hp.peel_async(d, m, max_layers=1 << 17), want)
    got = hp.peel(d, m, max_layers=1 << 17)
    assert got.rounds == want.rounds
    assert np.array_equal(_u32(got.order), want.order)
    assert np.array_equal(_u32(got.claim), want.claim)
    assert np.array_equal(_u64(got.layer_off), want.layer_off[:want.rounds + 1].astype(np.uint64))


# ------------------------------------------------------------------- errors --

@pytest.mark.parametrize("n_edges", [1200, 140_000])
def test_layer_table_too_small_on_the_general_path(blocked, n_edges):
    if n_edges > 131_072:
        hp.set_tuning()
    e, m = _chain(n_edges)
    want = oracle.peel_rounds(e, m)
    d = _dev32(e)
    got = hp.peel_async(d, m, max_layers=8)
    torch.cuda.synchronize()
    st = hp.stats_from_device(got.stats)
    assert st["async_status"] == LAYERS_FULL and st["rounds"] == want.rounds
    assert np.array_equal(_u32(got.order), want.order)
    assert np.array_equal(_u32(got.claim), want.claim)
    with pytest.raises(hp.HpeelError, match="CAPACITY"):
        hp.peel(d, m, max_layers=8)


def test_vertex_outside_its_part_on_the_general_path(n):
    m = oracle.num_vertices(n, 1230, 3)
    e = oracle.hash_edges(inputs.keys(n, 3), m, 3, 1)
    e[n // 3, 1] = 1  # a vertex of part 0 at position 1
    d = _dev32(e)
    got = hp.peel_async(d, m)
    torch.cuda.synchronize()
    st = hp.stats_from_device(got.stats)
    assert st["async_status"] == DEVICE_ERROR and st["device_err"] == 1
    with pytest.raises(hp.HpeelError, match="DEVICE_CHECK"):
        hp.peel(d, m)
