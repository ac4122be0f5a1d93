"""Batches of large roads, which the fused path screens in single precision
before it evaluates what can be the best combination exactly: every record
against the oracle where the bound of the screen, the cut-off last row, the
list of candidates or the order of ties can go wrong."""
import numpy as np
import pytest

from paper_1311_0380_gb300 import synth
from svt_testlib import assert_same, cfg_pair, gpu_run, oracle_run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


CONSTS = synth.make_constants(64)


def batch(hits, n_events=6, seed=3, xft=False):
    spec = synth.BatchSpec("large", 64, ("const", 12), hits, 262144, seed, xft=xft)
    return synth.make_batch(spec, n_events, CONSTS)


def check(b, F=CONSTS.F, q=CONSTS.q, sched=None, what="", **cfg):
    g, o = cfg_pair(n_sectors=64, **dict({"chi2_cut": CONSTS.chi2_cut_99}, **cfg))
    key, rec = oracle_run(b.words, b.event_off, F, q, o)
    st, got, counts = gpu_run(b.words, b.event_off, F, q, g, "fused", sched=sched)
    assert_same(st, got, key, rec, what)
    assert counts[2] >= 1024 * counts[0] or what == "small"
    assert counts[3] == int(np.sum(rec[:, 0] >> 24 & 1))
    return rec


# last rows cut short at every kind of place, roads of one row, of several
# rounds of rows, and small roads among large ones
@pytest.mark.parametrize("max_comb", [1100, 1111, 1151, 2048, 4097, 20011, 262144])
@pytest.mark.parametrize("hits", [("uniform", 1, 16), ("const", 5)])
def test_rows_cut_short(hits, max_comb):
    rec = check(batch(hits), max_comb=max_comb)
    assert np.any(rec[:, 0] >> 24 & 1)


@pytest.mark.parametrize("sched", [(0, 0, 1, 0, 1024, 0), (4, 1, 7, 3, 1500, 0), (16, 0, 256, 4, 4096, 0),
                                   (1, 1, 64, 32, 16384, 0)])
def test_items_of_split_roads(sched):
    from paper_1311_0380_gb300 import api
    check(batch(("uniform", 2, 8), 4), sched=api.schedule(*sched), max_comb=30000)


# shifts widen the bound (more candidates); cuts at both ends and around the
# square at which the clamp starts to count
@pytest.mark.parametrize("oshift,qshift", [(15, 15), (9, 0), (9, 24), (31, 24), (20, 3)])
@pytest.mark.parametrize("cut", [0, 1, 171004, 32767 ** 2 - 1, 32767 ** 2, 0xFFFFFFFE, 0xFFFFFFFF])
def test_shifts_and_cuts(oshift, qshift, cut):
    check(batch(("const", 4), 2, seed=cut % 97), oshift=oshift, qshift=qshift, chi2_cut=cut)


@pytest.mark.parametrize("kind", ["zero", "extreme", "small", "constant"])
@pytest.mark.parametrize("cut", [171004, 0xFFFFFFFF])
def test_constants_that_tie_or_saturate(kind, cut):
    rng = np.random.default_rng(11)
    F, q = CONSTS.F.copy(), CONSTS.q.copy()
    if kind == "zero":
        F[:], q[:] = 0, 0
    elif kind == "extreme":
        F = rng.choice(np.array([-32768, 32767], np.int16), F.shape)
        q = rng.choice(np.array([-32768, 0, 32767], np.int16), q.shape)
    elif kind == "small":   # many equal chi2
        F = rng.integers(-2, 3, F.shape).astype(np.int16)
        q[:] = 0
    else:   # every combination the same, not zero
        F[:], q[:] = 0, 100
    check(batch(("uniform", 3, 6), 3), F, q, chi2_cut=cut, max_comb=6000)


def test_equal_hits_and_pairs():
    b = batch(("const", 4), 3)
    hit = b.words >> 30 == 0
    b.words[hit] = (b.words[hit] & ~np.uint32(0x7FFF)) | np.uint32(16000)
    check(b, chi2_cut=0xFFFFFFFF)
    for max_comb in (1300, 262144):
        check(batch(("uniform", 3, 8), 4, xft=True), xft_pairs=1, max_comb=max_comb)


def test_missing_layers_and_min_layers():
    spec_hits = ("uniform", 0, 9)
    for ml in (0, 4, 6):
        check(batch(spec_hits, 8, seed=ml), min_layers=ml)


def test_constants_at_an_odd_address():
    """The constants only have to be 2-byte aligned."""
    import torch
    from paper_1311_0380_gb300 import api
    b = batch(("const", 4), 3)
    cfg, ocfg = cfg_pair(n_sectors=64, chi2_cut=CONSTS.chi2_cut_99)
    dc = api.DeviceConstants.from_numpy(CONSTS.F, CONSTS.q, cfg)
    off = lambda t: torch.cat([t.new_zeros(1), t.reshape(-1)])[1:]
    dc.F, dc.q = off(dc.F), off(dc.q)
    assert dc.F.data_ptr() % 4 == 2
    fp = api.FusedPath(len(b.words), b.n_events, b.total_roads, dc)
    fp.run(api.to_device_u32(b.words), len(b.words), api.to_device_u64(b.event_off), b.n_events)
    status, rec, _ = fp.result()
    key, ref = oracle_run(b.words, b.event_off, CONSTS.F, CONSTS.q, ocfg)
    assert_same(status, rec, key, ref, "odd address")
