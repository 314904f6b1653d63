"""The 64-bit build's incidences bucketed by vertex range (graphs of several
chunks): equal to the 32-bit build, which is checked against the oracle, with
the layer list in device memory (one pass over the keys per part) and in host
memory (several), and with chunk arrays that overflow."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("n,on_host", [(6_819_000, False), (6_830_000, False), (12_000_001, False),
                                       (20_000_003, False), (40_000_000, True)])
def test_bucketed_build_equals_the_32_bit_build(n, on_host):
    keys = inputs.keys_torch(n, 61)
    want = hp.mphf_build(keys)
    hl = torch.empty(n, dtype=torch.int64, pin_memory=True) if on_host else None
    got = hp.mphf_build_large(keys, host_list=hl)
    assert torch.equal(got.G, want.G) and torch.equal(got.rank_dir, want.rank_dir)
    for f in ("seed_used", "rounds", "n_peeled", "first_layer", "frontier", "attempts"):
        assert got.stats[f] == want.stats[f], f


def test_chunk_arrays_that_overflow():
    # identical keys fall into one chunk per part: never peel; a degree of
    # 2^24 is reported
    for n, code in ((15_000_000, "RETRIES_EXHAUSTED"), (20_000_000, "CAPACITY")):
        keys = torch.full((n,), 12345, dtype=torch.int64, device="cuda")
        with pytest.raises(hp.HpeelError, match=code):
            hp.mphf_build_large(keys, max_tries=1)
