"""Blocks of freed objects serve later ones: same results, and the memory goes back with the last context."""
import numpy as np
import pytest
import torch

import oracle
from tests import helpers
from workloads import configs

pytestmark = pytest.mark.gpu


def test_objects_made_from_returned_blocks():
    from paper_2410_03462_b200 import api
    w = configs.tiny()
    f = oracle.deconvolve(w.alpha).astype(np.float32)
    other = api.Context(0)
    ctx = api.Context(0)
    for N in (700, 300, 650, 700):
        g = configs.point_cloud_4096(N).graph()
        feat = api.sample(ctx, api.DeviceGraph(g), N, w.n_walks, w.p_halt, w.max_len, f)
        for which, want in enumerate(oracle.sample(g.rowptr, g.col, g.w, N, w.n_walks, w.p_halt, w.max_len, f)[:3]):
            helpers.assert_csr_equal(feat.to_host(which), want, f"N={N} matrix {which}", val_rtol=0)
        feat.free()
    ctx.close()
    other.close()
    torch.cuda.synchronize()
