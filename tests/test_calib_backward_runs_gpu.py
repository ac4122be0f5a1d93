"""The general calibration backward where a run of a warp holds several items:
both buffers in turn, sums carried from item to item and over the ends of
sectors, sectors of many runs, and runs of more items than one batch of lookups
(32); against float64 sums on the GPU."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def sector_sizes(n, S, rng):
    """Sizes that sum up to n: empty sectors, sectors around one item, the rest uneven."""
    sizes = rng.choice([0, 1, 31, 255, 256, 257, 512], S)
    left = n - int(sizes.sum())
    share = rng.random(S) ** 3 + 1e-3
    sizes = sizes + np.floor(left * share / share.sum()).astype(np.int64) * (rng.random(S) < 0.6)
    sizes[rng.integers(0, S)] += n - int(sizes.sum())
    return sizes


# 256 tracks an item and six runs an SM: 1 M tracks make runs of four or five
# items, 8 M of about 34, 230,003 of one, with one run of two
@pytest.mark.parametrize("n,S", [(230_003, 1), (1_000_003, 1), (1_000_003, 16), (1_000_001, 512),
                                 (8_000_003, 1), (8_000_002, 16), (8_000_003, 512)])
@pytest.mark.parametrize("off", [0, 2])
def test_several_items_a_run(n, S, off):
    import torch
    from paper_1311_0380_gb300 import api, calib
    rng = np.random.default_rng([n, S])
    sizes = sector_sizes(n, S, rng)
    assert sizes.sum() == n and sizes.min() >= 0
    g = torch.Generator(device="cuda").manual_seed(n + S)
    x = torch.rand(n, 6, device="cuda", generator=g) * 32767
    sector = torch.repeat_interleave(torch.arange(S, device="cuda", dtype=torch.int32),
                                     torch.as_tensor(sizes, device="cuda"))
    data = calib.CalibData(x, sector, torch.zeros(n, 3, device="cuda"), S)
    F = torch.zeros(S, 6, 6, device="cuda", requires_grad=True)
    q = torch.zeros(S, 6, device="cuda", requires_grad=True)
    gy = torch.empty(n * 6 + off, device="cuda")[off:].view(n, 6)
    gy.copy_(torch.randn(n, 6, device="cuda", generator=g))
    calib.fit_fp32(F, q, data).backward(gy)
    items = -(-sizes // 256)
    runs = min(6 * api.svt_device_sm_count(), int(items.sum()))
    a = 0
    for s in range(S):
        z = a + int(sizes[s])
        xs, gs = x[a:z].double(), gy[a:z].double()
        a = z
        # roundings on the way of a term: eight tracks of a lane in an item, the
        # items of its run, the sums over the lanes, and one partial for every run
        # that holds some of the sector (staged) or for every item (not)
        per_run = -(-int(items.sum()) // runs)
        partials = int(items[s]) if off else min(int(items[s]), int(items[s]) // max(per_run - 1, 1) + 2)
        bound = (8 + per_run + 12 + partials) * 2.0 ** -24
        for got, exact, size in ((F.grad[s], gs.T @ xs, gs.abs().T @ xs),
                                 (q.grad[s], gs.sum(0), gs.abs().sum(0))):
            assert bool(((got.double() - exact).abs() <= bound * size).all()), (s, int(sizes[s]))
