"""hpeel_kernel_launches against the launches a device-driven round loop makes:
round kernels stand eight to a turn of the loop over large layers, and each run
of them is followed by the kernel that runs small layers, whether or not it
finds one.  The host's loop, which launches one kernel per round, is the
yardstick: the rest of a peel's kernels are the same."""
import numpy as np
import pytest

from paper_1312_0526_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1312_0526_gb300 as hp  # noqa: E402

BODY = 8  # round kernels in one turn


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1312_0526_gb300 import build
    build.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _launches(edges, m, general):
    hp.peel(edges, m, general=general)  # (a graph is built on its first call)
    before = hp.kernel_launches()
    p = hp.peel(edges, m, general=general)
    return hp.kernel_launches() - before, p


def _loop_kernels(sizes, small):
    """Launches of the loop of random rounds over layers of these sizes."""
    sizes = list(sizes) + [0]
    t = total = 0
    while sizes[t] > 0:
        run = 0
        while sizes[t] > small:
            run += 1
            t += 1
        total += 2 + -(-run // BODY) * BODY
        while 0 < sizes[t] <= small:
            t += 1
    return total


# one run of large layers, of fewer and of more than eight, none at all, and an
# r whose small layers are smaller
@pytest.mark.parametrize("n,gamma,r,general", [
    (140_000, 1230, 3, False), (400_000, 1230, 3, False), (1_000_003, 1230, 3, False),
    (1_000_003, 1230, 3, True), (3_000_000, 1225, 3, False), (2_000_000, 1300, 4, False),
    (1_000_000, 1100, 3, False)])
def test_round_loop_launches(n, gamma, r, general):
    keys = torch.from_numpy(inputs.keys(n, 3).view(np.int64)).cuda()
    m = hp.num_vertices(n, gamma, r)
    edges = hp.hash_edges(keys, m, r, seed=1, general=general)
    graph, p = _launches(edges, m, general)
    hp.set_tuning(host_round_loop=1)
    try:
        host, _ = _launches(edges, m, general)
    finally:
        hp.set_tuning()
    sizes = np.diff(p.layer_off.cpu().numpy())
    small = 16 * (1024 if r == 4 else 2048)  # entries of a layer that one cluster runs
    assert graph - host == _loop_kernels(sizes, small) - p.rounds
