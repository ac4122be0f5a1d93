"""The fit kernel's chunks of roads where the chunks of several roads give way to
single ones (two roads per warp of the grid before the end): every record against
the oracle, in both forms of the fit, with and without split roads."""
import numpy as np
import pytest

from paper_1311_0380_gb300 import api, synth
from svt_testlib import assert_same, cfg_pair, gpu_run, oracle_run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("hits,small_max", [(("const", 2), 4096), (("uniform", 1, 4), 200),
                                            (("const", 4), 4096), (("const", 4), 1024)])
@pytest.mark.parametrize("per", [1, 3, 32])
@pytest.mark.parametrize("beyond", [None, -1, 0, 1, 40])
def test_the_last_roads_come_one_by_one(hits, small_max, per, beyond):
    # one block of one warp on each SM; `beyond` multiples of a chunk, and one
    # road, past the single ones
    tail = 2 * api.svt_device_sm_count(0)
    n = 1 if beyond is None else tail + (beyond * per + 1 if beyond > 0 else beyond)
    consts = synth.make_constants(64)
    spec = synth.BatchSpec("chunks", 64, ("const", n), hits, 262144, 5)
    b = synth.make_batch(spec, 1, consts)
    g, o = cfg_pair(n_sectors=64, chi2_cut=consts.chi2_cut_99)
    key, rec = oracle_run(b.words, b.event_off, consts.F, consts.q, o)
    st, got, counts = gpu_run(b.words, b.event_off, consts.F, consts.q, g, "fused",
                              sched=api.schedule(1, 1, 16, per, small_max, 0))
    assert int(counts[0]) == n
    assert_same(st, got, key, rec, (hits, per, n))
