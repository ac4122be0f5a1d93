"""The calibration sort (svt_calib_sort, svt_calib_index) against a stable
argsort: sizes at the edges of its tiles, few and many sectors, inputs that
start off a 16-byte boundary, empty sectors and a bad one."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("n,S", [(1, 1), (31, 512), (2047, 3), (2048, 512), (2049, 337),
                                 (700_001, 512), (700_000, 1)])
def test_tracks_come_in_stable_sector_order(n, S, off):
    import torch
    from paper_1311_0380_gb300 import _native as N, calib
    rng = np.random.default_rng(n + S)
    # sectors 0 mod 3 stay empty when there are several
    sector = rng.integers(0, S, n)
    sector = np.where(sector % 3 == 0, np.minimum(sector + 1, S - 1), sector).astype(np.int32)
    x = torch.randn(off + n * 6, device="cuda")[off:].reshape(n, 6)
    theta = torch.randn(off + n * 3, device="cuda")[off:].reshape(n, 3)
    sec = torch.empty(off + n, dtype=torch.int32, device="cuda")[off:]
    sec.copy_(torch.from_numpy(sector))
    perm = np.argsort(sector, kind="stable")
    d = calib.CalibData(x, sec, theta, S)
    assert np.array_equal(d.perm.cpu().numpy(), perm)
    assert torch.equal(d.x, x[d.perm.long()]) and torch.equal(d.theta, theta[d.perm.long()])
    # the index alone gives the same order and tables
    L = N.load()
    index = torch.zeros_like(d.index)
    p2 = torch.empty_like(d.perm)
    status = torch.zeros(1, dtype=torch.int64, device="cuda")
    v = lambda t: ctypes.c_void_p(t.data_ptr())
    N.check(L.svt_calib_index(v(sec), n, S, v(index), index.numel(), v(p2), v(status),
                              ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)), "index")
    assert torch.equal(p2, d.perm) and int(status.item()) == -1


def test_the_first_bad_sector_is_named():
    import torch
    from paper_1311_0380_gb300 import _native as N, calib
    n = 5000
    sector = torch.zeros(n, dtype=torch.int32, device="cuda")
    sector[4321] = 7
    sector[3210] = -1
    with pytest.raises(N.SvtError, match="3210"):
        calib.CalibData(torch.zeros(n, 6), sector, torch.zeros(n, 3), 7)
