"""The per-stage combine and select at the sizes where their tiles and groups
can go wrong: more roads to a tile of combinations than it stages, roads
without combinations between others, long roads, and combination arrays that
start off a 16-byte boundary."""
import numpy as np
import pytest

from paper_1311_0380_gb300 import synth
from svt_testlib import assert_same, cfg_pair, oracle_run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def roads(counts, seed):
    """One event per 100 roads with the given hits per layer, random coordinates."""
    rng = np.random.default_rng(seed)
    words, off = [], [0]
    for e in range(0, len(counts), 100):
        part = counts[e: e + 100]
        words.append(int(synth.event_word(e // 100, len(part))))
        for r, n in enumerate(part):
            words.append(int(synth.road_word(int(rng.integers(0, 64)), e + r)))
            for l in range(6):
                words += [int(synth.hit_word(l, int(x))) for x in rng.integers(0, 32768, n[l])]
        off.append(len(words))
    return np.array(words, np.uint32), np.array(off, np.uint64)


ONE = (1, 1, 1, 1, 1, 1)
CASES = {
    "one combination each": [ONE] * 4500,
    "none between": ([ONE, (0, 0, 1, 1, 1, 1), (2, 1, 1, 3, 1, 1)] * 900),
    "long ones": [(16, 16, 4, 2, 1, 1), ONE, (16, 8, 8, 1, 1, 1), (1, 1, 1, 1, 16, 16),
                  (2, 0, 2, 2, 2, 2)] * 3 + [(16, 16, 16, 1, 16, 1)],
}


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("name", list(CASES))
def test_combine_and_select_at_the_edges_of_tiles(name, off):
    import torch
    from paper_1311_0380_gb300 import api
    counts = CASES[name]
    words, eoff = roads(counts, 7)
    consts = synth.make_constants(64)
    cfg, ocfg = cfg_pair(chi2_cut=3 << 26, n_sectors=64, min_layers=5)
    combs = [int(np.prod([max(v, 1) for v in n])) if sum(v > 0 for v in n) >= 5 else 0
             for n in counts]
    total = sum(combs)
    p = api.PlainPath(len(words), len(eoff) - 1, len(counts), total + 4,
                      api.DeviceConstants.from_numpy(consts.F, consts.q, cfg))
    p.comb_cap = total
    p.comb_road, p.comb_hits = p.comb_road[off:], p.comb_hits[off:]
    p.run(api.to_device_u32(words), len(words), api.to_device_u64(eoff), len(eoff) - 1)
    status, rec, _ = p.result()
    key, ref = oracle_run(words, eoff, consts.F, consts.q, ocfg)
    assert_same(status, rec, key, ref, name)
    # every combination in order: road, then one hit per layer, layer 5 fastest
    road = np.repeat(np.arange(len(counts)), combs)
    assert np.array_equal(p.comb_road[:total].cpu().numpy(), road)
    c = np.arange(total) - np.repeat(np.cumsum([0] + combs[:-1]), combs)
    n = np.maximum(np.array(counts), 1)[road]
    hits = np.zeros(total, np.int64)
    for l in range(5, -1, -1):
        hits |= (c % n[:, l]) << (4 * l)
        c //= n[:, l]
    assert np.array_equal(p.comb_hits[:total].cpu().numpy(), hits)
