"""Rule V11 where an event starts with a hit: the hit run of the road before it
ends at the event's offset, so that an unpaired run there is the smallest key and
not the event's missing header."""
import numpy as np
import pytest

import oracle
from paper_1311_0380_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


BEFORE = {"none": [], "4": [4], "5": [5], "45": [4, 5], "445": [4, 4, 5], "0455": [0, 4, 5, 5],
          "4 in 17": [4] * 17, "all": [l for l in range(6) for _ in range(16)],
          "one short": [l for l in range(6) for _ in range(16)][:-1]}
AFTER = {"4": [4], "5": [5], "45": [4, 5], "55 and on": [5, 5, 0, 1], "a row": [4] * 40}


# the event's offset in the middle of a row, at the edges of rows and tiles
@pytest.mark.parametrize("at", [200, 256, 1023, 1024, 1025, 2048, 3000])
@pytest.mark.parametrize("lost_twice", [False, True])
def test_a_run_ends_at_the_next_event(at, lost_twice):
    import torch
    from paper_1311_0380_gb300 import api
    n_unpaired = 0
    for before in BEFORE.values():
        for after in AFTER.values():
            n = at - 2 - len(before)   # roads without hits, then the run's road
            words = [int(synth.event_word(0, n + 1))] + [int(synth.road_word(3, k)) for k in range(n + 1)]
            words += [int(synth.hit_word(l, 50 + l)) for l in before]
            assert len(words) == at
            words += [int(synth.hit_word(l, 9)) for l in after]
            off = [0, at] + ([at + 1] if lost_twice and len(after) > 1 else [])
            off.append(len(words))
            w, o = np.array(words, np.uint32), np.array(off, np.uint64)
            d = dict(dtype=torch.int32, device="cuda")
            status = torch.zeros(1, dtype=torch.int64, device="cuda")
            n_roads = torch.zeros_like(status)
            ws = torch.empty(api.svt_unpack_workspace_size(len(w)), dtype=torch.uint8, device="cuda")
            api.svt_unpack(api.to_device_u32(w), len(w), api.to_device_u64(o), len(o) - 1, 64, len(w),
                           torch.zeros(len(w), **d), torch.zeros(len(w), **d), torch.zeros(len(o), **d),
                           n_roads, status, ws, xft_pairs=1)
            key = oracle.validate(w, o, 64, 1)
            assert int(api.u64(status)[0]) == key, (before, after)
            n_unpaired += oracle.decode_key(key)[1] == oracle.E_XFT_UNPAIRED
    assert n_unpaired
