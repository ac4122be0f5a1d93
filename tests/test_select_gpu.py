"""svt_select alone on made-up chi2: roads of no, few and many combinations around
the sizes at which a lane, a warp and a block take over, in small and in large
groups, with ties, against numpy; and the time of many short roads."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


class Select:
    def __init__(self, counts, chi2, cut):
        import torch
        from paper_1311_0380_gb300 import api
        R, n = len(counts), int(counts.sum())
        self.off = np.concatenate([[0], np.cumsum(counts)]).astype(np.uint64)
        self.par = np.arange(3 * n, dtype=np.uint32).reshape(3, n)
        self.best = torch.zeros(R * 6, dtype=torch.int32, device="cuda")
        self.status = torch.full((1,), -1, dtype=torch.int64, device="cuda")
        flags = np.arange(R, dtype=np.uint32) & 14
        self.args = (api.to_device_u32(chi2), api.to_device_u32(self.par.reshape(-1)), n,
                     api.to_device_u64(self.off), api.to_device_u32(flags),
                     torch.tensor([R], device="cuda"), R, api.config(chi2_cut=cut), self.best,
                     self.status)

    def run(self):
        from paper_1311_0380_gb300 import api
        api.svt_select(*self.args)


def expected(counts, chi2, cut):
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    n = len(chi2)
    out = np.zeros((len(counts), 6), np.uint32)   # svt_best: flags, comb, chi2, p
    out[:, 0] = np.arange(len(counts)) & 14
    out[:, 1] = 0xFFFFFFFF
    for r in np.flatnonzero(counts):
        v = chi2[off[r]: off[r + 1]]
        c = int(np.argmin(v))
        if v[c] <= cut:
            j = off[r] + c
            out[r] = [out[r, 0] | 1, c, v[c], j, n + j, 2 * n + j]
    return out


SHORT = [0, 1, 2, 31, 32, 33, 63, 64, 65, 130]


# 300 and 38,913 roads: groups of 16 and the first size that has more; 150,001
# roads: of 62; 320,000: the largest; with long roads among short ones, and all long
@pytest.mark.parametrize("n_roads,long", [(1, []), (300, [1023, 1024, 1025, 5000]), (38_913, []),
                                          (38_913, [1024, 1025, 40_000]), (150_001, [3000]),
                                          (320_000, [70_000])])
@pytest.mark.parametrize("cut,top", [(0xFFFFFFFF, 40), (5, 60), (0, 3)])
def test_best_combination(n_roads, long, cut, top):
    from paper_1311_0380_gb300 import api
    rng = np.random.default_rng(n_roads + top)
    counts = rng.choice(SHORT[:7] if n_roads > 100_000 else SHORT, n_roads)
    for i, v in enumerate(long):
        counts[rng.integers(0, n_roads, 1 if v > 9000 else 5)] = v
    chi2 = rng.integers(0, top, int(counts.sum())).astype(np.uint32)   # ties everywhere
    s = Select(counts, chi2, cut)
    s.run()
    assert np.array_equal(api.u32(s.best).reshape(-1, 6), expected(counts, chi2, cut))


def test_many_short_roads_take_little_time():
    """200,000 roads of one combination: 12 MB in and out, 21 us; a block's warps
    that claim such roads one by one took 89."""
    import torch
    s = Select(np.ones(200_000, np.int64), np.zeros(200_000, np.uint32), 9)
    us = []
    for _ in range(8):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(20):
            s.run()
        b.record()
        torch.cuda.synchronize()
        us.append(a.elapsed_time(b) * 50.0)
    assert min(us) < 60.0, us
