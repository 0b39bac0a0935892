"""trace_device on a stream of its own shares no memory with what other streams have queued."""
import numpy as np
import pytest
import torch

import oracle
import paper_2002_07704_gb300 as lsq
from gpu_common import cuda, gpu_geometry, si

pytestmark = pytest.mark.gpu


def test_result_outlives_work_queued_on_the_current_stream():
    lsq.build()
    lsq.load()
    pos, cell = si(2, 0.1, 94)
    g = gpu_geometry(pos, cell, [4.0])
    p = oracle.neighbour_list(pos, cell, 4.0)
    X, Y = (cuda(np.random.default_rng(k).standard_normal((p.nnzb, 4, 4))) for k in (0, 1))
    want = lsq.trace(g, 4, X, 0, Y, 0)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    # small blocks of the current stream's memory, as many as it has; what is queued there may still
    # write to them when they are free again
    old = [torch.empty(n, dtype=torch.float64, device="cuda") for n in (1, 1024) for _ in range(4096)]
    spans = [(t.data_ptr(), t.data_ptr() + 8 * t.numel()) for t in old]
    del old
    out = lsq.trace_device(g, 4, X, 0, Y, 0, stream=side)
    side.synchronize()
    torch.cuda.synchronize()
    assert abs(out.item() - want) <= 1e-12 * abs(want)
    assert not any(lo <= out.data_ptr() < hi for lo, hi in spans)
