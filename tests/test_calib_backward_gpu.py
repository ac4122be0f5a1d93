"""The general calibration backward (sum of grad_y x^T and of grad_y per sector)
at the edges of its items and copies, staged (grad_y on a 16-byte boundary) and
not, against float64."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [1, 16, 512])
@pytest.mark.parametrize("n", [1, 3, 255, 256, 258, 1021, 30001])
@pytest.mark.parametrize("off", [0, 2])
def test_general_backward_sums(n, S, off):
    import torch
    from paper_1311_0380_gb300 import calib
    rng = np.random.default_rng([n, S])
    x = rng.uniform(0, 32767, (n, 6)).astype(np.float32)
    sector = rng.integers(0, S, n).astype(np.int32)
    data = calib.CalibData(x, sector, np.zeros((n, 3), np.float32), S)
    perm = data.perm.cpu().numpy()
    F = torch.zeros(S, 6, 6, device="cuda", requires_grad=True)
    q = torch.zeros(S, 6, device="cuda", requires_grad=True)
    g = rng.standard_normal((n, 6)).astype(np.float32)
    gy = torch.empty(n * 6 + off, device="cuda")[off:].view(n, 6)
    gy.copy_(torch.from_numpy(g))
    calib.fit_fp32(F, q, data).backward(gy)
    s, xs, g64 = sector[perm], x[perm].astype(np.float64), g.astype(np.float64)
    # no entry passes through more than 160 roundings (8 tracks of an item, the
    # items of a run, 32 lanes, at most 118 runs of a sector): each adds at most
    # 2^-24 of the sum of magnitudes
    for got, terms in ((F.grad, g64[:, :, None] * xs[:, None, :]), (q.grad, g64)):
        exact = np.zeros((S,) + terms.shape[1:])
        size = np.zeros_like(exact)
        np.add.at(exact, s, terms)
        np.add.at(size, s, np.abs(terms))
        assert np.all(np.abs(got.cpu().numpy() - exact) <= 160 * 2.0 ** -24 * size)
