"""Constants at an odd (2-byte aligned) address in a batch that is screened: the
records' constants are then fetched 16 bits at a time."""
import numpy as np
import pytest

from paper_1311_0380_gb300 import synth
from svt_testlib import assert_same, cfg_pair, oracle_run

pytestmark = pytest.mark.gpu
CONSTS = synth.make_constants(64)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("small_max", [0, 1024])   # whole roads, items of split roads
@pytest.mark.parametrize("odd", ["F", "q", "Fq"])
def test_constants_at_an_odd_address(odd, small_max):
    import torch
    from paper_1311_0380_gb300 import api
    b = synth.make_batch(synth.BatchSpec("large", 64, ("const", 12), ("const", 4), 262144, 3), 5, CONSTS)
    cfg, ocfg = cfg_pair(n_sectors=64, chi2_cut=CONSTS.chi2_cut_99)
    dc = api.DeviceConstants.from_numpy(CONSTS.F, CONSTS.q, cfg)
    off = lambda t: torch.cat([t.new_zeros(1), t.reshape(-1)])[1:]
    dc.F = off(dc.F) if "F" in odd else dc.F
    dc.q = off(dc.q) if "q" in odd else dc.q
    assert (dc.F.data_ptr() | dc.q.data_ptr()) % 4 == 2
    fp = api.FusedPath(len(b.words), b.n_events, b.total_roads, dc, api.schedule(small_max=small_max))
    fp.run(api.to_device_u32(b.words), len(b.words), api.to_device_u64(b.event_off), b.n_events)
    status, rec, counts = fp.result()
    key, ref = oracle_run(b.words, b.event_off, CONSTS.F, CONSTS.q, ocfg)
    assert_same(status, rec, key, ref, odd)
    # the batch lies above the line from which on batches are screened
    assert counts[2] >= 1024 * counts[0] and counts[3] == int(np.sum(rec[:, 0] >> 24 & 1)) > 0
