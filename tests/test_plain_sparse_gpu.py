"""The per-stage combine where few roads have combinations: any number of roads
without one may lie between two that have some, at no more than the cost of
counting them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# the distances between roads that have combinations: neighbours, a few, more
# than a tile stages, and a whole batch
@pytest.mark.parametrize("gap", [1, 2, 3, 7, 511, 512, 513, 1000, 199_999])
def test_roads_without_combinations_between_others(gap):
    import torch
    from paper_1311_0380_gb300 import api
    R = 200_000
    some = np.arange(0, R, gap)[:3000]
    nhit = np.full(R, 1 | 1 << 5 | 1 << 10, np.uint32)          # three layers of five
    nhit[some] = sum((2 if l < 4 else 1) << 5 * l for l in range(6))   # 16 combinations
    total = 16 * len(some)
    z = lambda n, dt=torch.int32: torch.zeros(n, dtype=dt, device="cuda")
    flags, off, road, hits, n_comb = z(R), z(R + 1, torch.int64), z(total), z(total), z(1, torch.int64)
    status = torch.full((1,), -1, dtype=torch.int64, device="cuda")
    ws = torch.empty(api.svt_combine_workspace_size(R), dtype=torch.uint8, device="cuda")
    d_nhit, n_roads = api.to_device_u32(nhit), torch.tensor([R], device="cuda")
    ms = []
    for _ in range(4):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        api.svt_combine(d_nhit, n_roads, R, api.config(min_layers=5), total, flags, off, road, hits,
                        n_comb, status, ws)
        b.record()
        torch.cuda.synchronize()
        ms.append(a.elapsed_time(b))
    assert int(status[0]) == -1 and int(n_comb[0]) == total
    assert np.array_equal(road.cpu().numpy(), np.repeat(some, 16))
    c = np.tile(np.arange(16), len(some))
    ref = (c >> 3) | (c >> 2 & 1) << 4 | (c >> 1 & 1) << 8 | (c & 1) << 12
    assert np.array_equal(hits.cpu().numpy(), ref)
    # the call reads 0.8 MB and writes 2.4 MB (about 25 us); forty times that
    # is far below any walk over the roads one by one (13 ms)
    assert min(ms) < 1.0, ms
