"""The per-stage fit at the ends of its ranges: extreme constants, coordinates
whose bytes are all zero or all one, the smallest and largest shifts, tiles whose
roads are staged and tiles with too many of them; chi2 and parameters of every
combination against int64."""
import numpy as np
import pytest

from paper_1311_0380_gb300 import api, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("hits", [(2, 2, 1, 3, 2, 2), (1, 1, 1, 1, 1, 1), (2, 1, 0, 2, 1, 1)])
@pytest.mark.parametrize("oshift,qshift", [(9, 0), (9, 24), (15, 15), (31, 0), (31, 24)])
def test_extreme_rows(hits, oshift, qshift):
    rng = np.random.default_rng([oshift, qshift])
    R, S = 300, 4
    xs = rng.choice([0, 1, 255, 256, 32512, 32767], (R, 6, 3))
    words = [int(synth.event_word(0, R))]
    sector = rng.integers(0, S, R)
    for r in range(R):
        words.append(int(synth.road_word(int(sector[r]), r)))
        words += [int(synth.hit_word(l, int(xs[r, l, h]))) for l in range(6) for h in range(hits[l])]
    words, off = np.array(words, np.uint32), np.array([0, len(words)], np.uint64)
    ends = np.array([-32768, -32767, -256, -1, 0, 1, 255, 32767])
    F = rng.choice(ends, (S, 64, 6, 6)).astype(np.int16)
    q = rng.choice(ends, (S, 64, 6)).astype(np.int16)
    F[0], q[0] = -32768, -32768   # every term at its end
    F[1], q[1] = 32767, 32767
    cfg = api.config(oshift, qshift, 0xFFFFFFFF, 262144, 5, S)
    C = int(np.prod(np.maximum(hits, 1)))
    p = api.PlainPath(len(words), 1, R, R * C, api.DeviceConstants.from_numpy(F, q, cfg))
    p.run(api.to_device_u32(words), len(words), api.to_device_u64(off), 1)
    assert int(api.u64(p.status)[0]) == (1 << 64) - 1
    c = np.arange(C)
    x = np.zeros((R, C, 6), np.int64)
    for l in range(5, -1, -1):
        n = max(hits[l], 1)
        if hits[l]:
            x[:, :, l] = xs[:, l, :][:, c % n]
        c = c // n
    mask = sum(1 << l for l in range(6) if hits[l])
    acc = np.einsum("rkl,rcl->rck", F[sector, mask].astype(np.int64), x)
    y = (acc + (q[sector, mask].astype(np.int64) << qshift)[:, None]) >> oshift
    chi = np.clip(y[:, :, 3:], -32767, 32767)
    assert np.array_equal(api.u32(p.fit_chi2)[: R * C], (chi * chi).sum(2).ravel())
    for k in range(3):
        got = p.fit_par[k * R * C: (k + 1) * R * C].cpu().numpy()
        assert np.array_equal(got, y[:, :, k].ravel()), k
