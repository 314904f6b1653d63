"""Rounds of a bucket that one warp runs (layers of at most 32 edges) and rounds
of the whole block: buckets whose layers lie around the limit, grow past it
again after a small one, or run out of their layer table in the middle of a
warp's run -- order, rounds, status and g values bucket by bucket against the
oracle."""
import numpy as np
import pytest

import oracle
from paper_1312_0526_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1312_0526_gb300 as hp  # noqa: E402

LIMIT = 32
SIZES = np.array([n for n in range(60, 200, 2) for _ in range(4)] + [2000, 5000] * 8)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1312_0526_gb300 import build
    build.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.fixture(scope="module")
def want():
    keys, off = inputs.bucketed_keys(SIZES, seed=21)
    res = []
    for b, n in enumerate(SIZES):
        m = oracle.num_vertices(int(n), 1230, 3)
        e = oracle.hash_edges(keys[int(off[b]):int(off[b + 1])], m, 3, b)
        res.append((e, m, oracle.peel_rounds(e, m)))
    layers = [np.diff(p.layer_off[:p.rounds + 1].astype(np.int64)) for _, _, p in res]
    sizes = set(np.concatenate(layers).tolist())
    assert {LIMIT - 1, LIMIT, LIMIT + 1} <= sizes
    assert any(((x[:-1] <= LIMIT) & (x[1:] > LIMIT)).any() for x in layers if len(x) > 1)
    return keys, off, res


@pytest.mark.parametrize("tuning", [
    None, {"threads": 64, "ctas_per_sm": 8}, {"threads": 1024, "ctas_per_sm": 1},
    {"smem_rounds": 6}, {"smem_rounds": 6, "global16_rounds": 9},
    {"threads": 256, "ctas_per_sm": 2, "smem_bytes": 1024}])
def test_small_and_large_layers(want, tuning):
    keys, off, res = want
    got = hp.peel_batched(torch.from_numpy(keys.view(np.int64)).cuda(),
                          torch.from_numpy(off.view(np.int64)).cuda(), with_g=True, tuning=tuning)
    order = got.order.cpu().numpy().view(np.uint32)
    G, G_off = got.G.cpu().numpy().view(np.uint64), got.G_off.cpu().numpy()
    for b, (e, m, p) in enumerate(res):
        assert int(got.rounds[b]) == p.rounds and int(got.status[b]) == int(p.core_nonempty), b
        assert np.array_equal(order[int(off[b]):int(off[b + 1])], p.order), b
        g = G[int(G_off[b]):int(G_off[b + 1])]
        assert not g.any() if p.core_nonempty else np.array_equal(g, oracle.mphf_assign(e, m, p)), b
