"""The fit kernel of the default schedule as svt_run launches it: shared memory
per block and blocks per SM, read from the captured launch."""
import ctypes

import pytest

from paper_1311_0380_gb300 import synth
from svt_testlib import cfg_pair

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


class KernelNode(ctypes.Structure):   # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3),
                ("shared", ctypes.c_uint), ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p),
                ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def captured_kernels(run):
    """Launches that `run(stream)` makes, in no order."""
    import torch
    cu = ctypes.CDLL("libcuda.so.1")
    stream = torch.cuda.Stream()
    h, graph = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
    assert cu.cuStreamBeginCapture_v2(h, 1) == 0   # thread-local
    try:
        run(stream)
    finally:
        assert cu.cuStreamEndCapture(h, ctypes.byref(graph)) == 0
    n = ctypes.c_size_t()
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    out = []
    for node in nodes:
        p = KernelNode()
        if cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), ctypes.byref(p)) == 0:
            out.append(p)
    cu.cuGraphDestroy(graph)
    return out


# 228 KB of shared memory an SM, of which 1 KB per block is reserved: 6528 bytes
# a warp leave 30 blocks of one warp, and 16, 8, 4 and 2 of the larger ones
@pytest.mark.parametrize("warps,blocks", [(1, 30), (2, 16), (4, 8), (8, 4), (16, 2)])
def test_blocks_of_the_default_fit_per_sm(warps, blocks):
    from paper_1311_0380_gb300 import api
    consts = synth.make_constants(64)
    b = synth.make_batch(synth.BatchSpec("s", 64, ("const", 4), ("const", 2), 1000, 1), 2, consts)
    cfg, _ = cfg_pair(n_sectors=64)
    p = api.FusedPath(len(b.words), b.n_events, b.total_roads,
                      api.DeviceConstants.from_numpy(consts.F, consts.q, cfg),
                      api.schedule(warps_per_block=warps))
    w, e = api.to_device_u32(b.words), api.to_device_u64(b.event_off)
    p.run(w, len(b.words), e, b.n_events)   # limits and attributes are set
    fit = max(captured_kernels(lambda s: p.run(w, len(b.words), e, b.n_events, stream=s)),
              key=lambda k: k.shared)
    assert fit.block[0] == 32 * warps and fit.shared <= 6528 * warps
    assert fit.grid[0] == blocks * api.svt_device_sm_count()
