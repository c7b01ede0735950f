"""Contexts on several streams that share a feature object, and calls under stream capture."""
import numpy as np
import pytest
import torch

import oracle
from workloads import configs, tensors

pytestmark = pytest.mark.gpu


def _context_on(stream):
    from paper_2410_03462_b200 import api
    with torch.cuda.stream(stream):
        return api.Context(0)


def _inputs(w, N, m, d, seed):
    return [t.cuda() for t in tensors.qkv(4, N, m, d, "bf16", seed)]


@pytest.mark.parametrize("m", [32, 128])     # over the mask; by the gather's tiles
def test_second_context_right_behind_the_first(m):
    from paper_2410_03462_b200 import api
    w = configs.point_cloud_4096(2048)
    f = oracle.deconvolve(w.alpha).astype(np.float32)
    sa, sb = torch.cuda.Stream(), torch.cuda.Stream()
    a, b = _context_on(sa), _context_on(sb)
    dg = api.DeviceGraph(w.graph())
    q, k, v = _inputs(w, 2048, m, 64, 3)
    for seed in range(5):
        feat = api.sample(a, dg, seed, w.n_walks, w.p_halt, w.max_len, f)
        torch.cuda.synchronize()
        with torch.cuda.stream(sa):
            first = api.masked_linear_attn(a, feat, q, k, v)
        with torch.cuda.stream(sb):
            second = api.masked_linear_attn(b, feat, q, k, v)
        torch.cuda.synchronize()
        assert torch.equal(first, second)
        feat.free()
    a.close()
    b.close()


def test_attention_and_remodulation_under_capture():
    from paper_2410_03462_b200 import api, binding as B
    w = configs.point_cloud_4096(2048)
    f = oracle.deconvolve(w.alpha).astype(np.float32)
    s = torch.cuda.Stream()
    ctx = _context_on(s)
    dg = api.DeviceGraph(w.graph())
    q, k, v = _inputs(w, 2048, 32, 64, 5)
    ws = torch.empty(B.grf_attn_workspace_bytes(4, 2048, 32, 64, B.dtype_code(q)), dtype=torch.uint8, device="cuda")
    B.grf_ctx_keep_walks(ctx.handle, True)
    feat = api.sample(ctx, dg, 7, w.n_walks, w.p_halt, w.max_len, f)
    new = (f * np.linspace(1.0, 1.3, f.size)).astype(np.float32)

    def step(coefficients):
        B.grf_remodulate(ctx.handle, feat.handle, w.max_len, coefficients, None)
        B.grf_features_materialise(ctx.handle, feat.handle)
        return api.masked_attn_mhat(ctx, feat, q, k, v), api.masked_linear_attn(ctx, feat, q, k, v, workspace=ws)

    with torch.cuda.stream(s):
        want = [t.clone() for t in step(new)]
        other = [t.clone() for t in step(f)]
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            got = step(new)
        for t in got:
            t.zero_()
        graph.replay()
        s.synchronize()
    for x, y, z in zip(want, got, other):
        assert torch.equal(x, y) and not torch.equal(x, z)
    del graph
    feat.free()
    ctx.close()
