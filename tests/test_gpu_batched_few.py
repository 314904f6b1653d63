"""The batched form without a shape on few buckets: only the size classes that the
buckets could fill are launched.  On both sides of every line of that rule, equal
to the one-launch form, which is checked against the oracle elsewhere."""
import numpy as np
import pytest

from paper_1312_0526_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1312_0526_gb300 as hp  # noqa: E402

STEPS = [1, 2, 3, 4, 6, 8, 12, 24]  # blocks per SM of the class launches


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1312_0526_gb300 import build
    build.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("past", [0, 1])
@pytest.mark.parametrize("ctas", [0, 1, 2, 3, 4, 6, 8, 12])
def test_few_buckets_launch_what_they_can_fill(ctas, past):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    B = ctas * sms + past or 2
    most = next((c for c in STEPS if c * sms >= B), STEPS[-1])
    rng = np.random.default_rng(B)
    sizes = np.minimum(np.exp(rng.normal(5.0, 1.5, B)).astype(np.int64), 9000)
    sizes[: min(B, 4)] = [30_000, 0, 65_536, 70_000][: min(B, 4)]  # global regions, empty, refused
    rng.shuffle(sizes)
    keys, off = inputs.bucketed_keys(sizes, seed=6)
    dk = torch.from_numpy(keys.view(np.int64)).cuda()
    do = torch.from_numpy(off.view(np.int64)).cuda()
    want = hp.peel_batched(dk, do, with_g=True, tuning={"threads": 256, "ctas_per_sm": 3})
    ws = torch.empty(hp.batched_workspace_size(B, 1230, None), dtype=torch.uint8, device="cuda")
    for rounds in (256, 4):  # the second sends most buckets to the last launch
        before = hp.kernel_launches()
        got = hp.peel_batched(dk, do, tuning={"smem_rounds": rounds}, workspace=ws)
        # the schedule, the first and the last launch, and the classes'
        assert hp.kernel_launches() - before == 3 + sum(c <= most for c in STEPS)
        whole = torch.from_numpy(np.repeat(sizes <= 65_536, sizes)).cuda()
        assert torch.equal(got.order[whole], want.order[whole])
        assert torch.equal(got.rounds, want.rounds) and torch.equal(got.status, want.status)
    got = hp.peel_batched(dk, do, with_g=True, workspace=ws)
    assert torch.equal(got.G, want.G) and torch.equal(got.order[whole], want.order[whole])
