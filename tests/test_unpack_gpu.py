"""Road extraction where its rows (32 words), warps (256 words) and tiles (1024
words) meet: one word or run of words around each boundary replaced by every
kind of word, the status key against the oracle's, and the outputs of the valid
batches against a scan of the words."""
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


def stream(n_words, pairs, seed):
    """Events of 9 roads with 0..16 hits per layer, cut at exactly n_words."""
    rng = np.random.default_rng(seed)
    words, off = [], [0]
    while len(words) < n_words:
        at, n_roads = len(words), 0
        words.append(0)
        while n_roads < 9 and len(words) < n_words:
            n = rng.integers(0, 17, 6) if rng.random() < 0.4 else rng.integers(0, 4, 6)
            if pairs:
                n[5] = n[4]
            n = n if len(words) + 1 + n.sum() <= n_words else 0 * n
            words.append(int(synth.road_word(int(rng.integers(0, 64)), n_roads)))
            for l in range(6):
                words += [int(synth.hit_word(l, int(x))) for x in rng.integers(0, 32768, n[l])]
            n_roads += 1
        words[at] = int(synth.event_word(len(off) - 1, n_roads))
        off.append(len(words))
    return np.array(words, np.uint32), np.array(off, np.uint64)


def hit(l):
    return int(synth.hit_word(l, 77))


KINDS = {
    "hit 0": [hit(0)], "hit 5": [hit(5)], "hit 3": [hit(3)], "layer 6": [6 << 27],
    "reserved bits": [hit(2) | 1 << 20], "reserved type": [1 << 30],
    "road": [int(synth.road_word(5, 9))], "bad sector": [int(synth.road_word(64, 9))],
    "event": [int(synth.event_word(0, 1))], "hit after event": [int(synth.event_word(0, 1)), hit(5)],
    "17 of a layer": [int(synth.road_word(5, 9))] + [hit(4)] * 17,
    "16 of a layer": [int(synth.road_word(5, 9))] + [hit(4)] * 16,
    "nothing": [],
}


@pytest.mark.parametrize("pairs", [0, 1])
@pytest.mark.parametrize("n_words", [31, 1024, 1025, 2300])
def test_words_around_the_boundaries(n_words, pairs):
    import torch
    from paper_1311_0380_gb300 import api
    base, off = stream(n_words, pairs, n_words)
    n_words = len(base)
    road_cap = n_words
    dev = dict(device="cuda")
    d_off = api.to_device_u64(off)
    road_word = torch.zeros(road_cap, dtype=torch.int32, **dev)
    road_nhit = torch.zeros(road_cap, dtype=torch.int32, **dev)
    event_road = torch.zeros(len(off), dtype=torch.int32, **dev)
    n_roads = torch.zeros(1, dtype=torch.int64, **dev)
    status = torch.zeros(1, dtype=torch.int64, **dev)
    ws = torch.empty(api.svt_unpack_workspace_size(n_words), dtype=torch.uint8, **dev)
    spots = sorted({b + d for b in (32, 256, 1024, 2048, n_words) for d in (-19, -17, -2, -1, 0, 1)}
                   | {int(o) for o in off})
    valid = 0
    for kind, put in KINDS.items():
        for i in spots:
            if i < 0 or i + len(put) > n_words:
                continue
            words = base.copy()
            words[i: i + len(put)] = put
            if pairs and np.any(words[off[:-1].astype(np.int64)] >> 30 == 0):
                continue   # a run of hits over a lost event header: V11's key differs
                           # (the oracle cuts the run at the event's offset)
            api.svt_unpack(api.to_device_u32(words), n_words, d_off, len(off) - 1, 64, road_cap,
                           road_word, road_nhit, event_road, n_roads, status, ws, xft_pairs=pairs)
            key = int(api.u64(status)[0])
            assert key == oracle.validate(words, off, 64, pairs), (kind, i)
            if key != (1 << 64) - 1:
                continue
            valid += 1
            pos = np.flatnonzero(words >> 30 == 2)
            assert int(n_roads[0]) == len(pos), (kind, i)
            assert np.array_equal(api.u32(road_word)[: len(pos)], pos), (kind, i)
            assert np.array_equal(api.u32(event_road), np.searchsorted(pos, off)), (kind, i)
            hits = np.flatnonzero(words >> 30 == 0)
            packed = np.zeros(len(pos), np.int64)
            np.add.at(packed, np.searchsorted(pos, hits) - 1, 1 << (5 * (words[hits] >> 27).astype(np.int64)))
            assert np.array_equal(api.u32(road_nhit)[: len(pos)], packed), (kind, i)
    assert valid
