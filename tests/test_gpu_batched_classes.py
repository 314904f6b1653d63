"""The batched form's launches by size class (no shape given): buckets at the
edges of every class, buckets that need more rounds than their class's shared
memory holds, and few or no buckets in a class -- equal to the one-launch form,
which is checked against the oracle bucket by bucket elsewhere, and a sample to
the oracle here."""
import numpy as np
import pytest

import oracle
from paper_1312_0526_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1312_0526_gb300 as hp  # noqa: E402

SMEM_PER_SM, BLOCK_MAX = 233_472, 232_384
CLASSES = [(24, True), (12, True), (8, True), (6, True), (4, True), (3, True), (4, False),
           (2, True), (3, False), (2, False), (1, False)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1312_0526_gb300 import build
    build.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _bytes(n, verts):
    m = oracle.num_vertices(n, 1230, 3)
    a = lambda x: (x + 15) // 16 * 16  # noqa: E731
    r = min(n + 1, 256)
    return (a(4 * m) + a(2 * n) + a(2 * n) + 2 * a(4 * (r + 2)) + a((m + 15) // 16 * 4)
            + (a(6 * n) if verts else 0))


def _edges_of_classes():
    sizes = []
    for ctas, verts in CLASSES:
        room = min(BLOCK_MAX, (SMEM_PER_SM // ctas - 1088) & ~15)
        lo, hi = 1, 65_536
        while lo + 1 < hi:  # largest n that fits
            mid = (lo + hi) // 2
            lo, hi = (mid, hi) if _bytes(mid, verts) <= room else (lo, mid)
        sizes += [lo - 1, lo, lo + 1]
    return sizes


def _run(keys, off, tuning, with_g=True):
    r = hp.peel_batched(keys, off, with_g=with_g, tuning=tuning)
    torch.cuda.synchronize()
    return r


@pytest.mark.parametrize("tuning", [None, {}, {"smem_rounds": 4},
                                    {"smem_rounds": 2, "global16_rounds": 2}])
@pytest.mark.parametrize("sizes", [
    _edges_of_classes() + [0, 1, 2, 3, 65_534, 65_535, 65_536, 70_000],
    [5], [0, 7, 0], list(range(1, 700)), [30_000] * 3])
def test_classes_equal_one_launch(sizes, tuning):
    sizes = np.array(sizes, dtype=np.int64)
    keys, off = inputs.bucketed_keys(sizes, seed=6)
    dk = torch.from_numpy(keys.view(np.int64)).cuda()
    do = torch.from_numpy(off.view(np.int64)).cuda()
    want = _run(dk, do, {"threads": 256, "ctas_per_sm": 3})
    got = _run(dk, do, tuning)
    whole = torch.from_numpy(np.repeat(sizes <= 65_536, sizes)).cuda()
    assert torch.equal(got.order[whole], want.order[whole])
    assert torch.equal(got.rounds, want.rounds) and torch.equal(got.status, want.status)
    assert torch.equal(got.G, want.G)
    order = got.order.cpu().numpy().view(np.uint32)
    for b in range(0, len(sizes), max(1, len(sizes) // 12)):
        n = int(sizes[b])
        if 0 < n <= 65_536:
            m = oracle.num_vertices(n, 1230, 3)
            e = oracle.hash_edges(keys[int(off[b]):int(off[b + 1])], m, 3, b)
            assert np.array_equal(order[int(off[b]):int(off[b + 1])],
                                  oracle.peel_rounds(e, m).order)
