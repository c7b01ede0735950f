"""grf_masked_linear_attn chooses between the per-node states and the materialised mask: both give the oracle's values,
and the choice depends on neither the workspace nor earlier calls."""
import numpy as np
import pytest
import torch

import oracle
from tests import helpers
from workloads import configs, tensors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [16, 32, 64])
@pytest.mark.parametrize("N,G", [(127, 8), (129, 40), (1000, 96)])
def test_both_routes_match_oracle(N, G, m):
    from paper_2410_03462_b200 import api, binding as B
    ctx = api.Context(0)
    w = configs.point_cloud_4096(N)
    g = w.graph()
    f = oracle.deconvolve(w.alpha).astype(np.float32)
    feat = api.sample(ctx, api.DeviceGraph(g), 3, w.n_walks, w.p_halt, w.max_len, f)
    Phi, _, PsiT, _, _ = helpers.oracle_features(w, g, 3, f)
    q, k, v = tensors.qkv(G, N, m, 64, "bf16", 4)
    qd, kd, vd = q.cuda(), k.cuda(), v.cuda()
    one = slice(G - 1, G)
    ref = oracle.attn_sparse(tensors.widen(q[one]), tensors.widen(k[one]), tensors.widen(v[one]), Phi, PsiT)
    out = {}
    for mode in (1, 2):                     # 1: the cheaper route, 2: always the states
        B.grf_ctx_use_tensor_cores(ctx.handle, mode)
        out[mode], den = api.masked_linear_attn(ctx, feat, qd, kd, vd, want_den=True)
        B.grf_ctx_check(ctx.handle)
        helpers.assert_attn_close(out[mode][one].float().cpu().numpy(), ref, helpers.TOL["bf16"], den[one].cpu().numpy(),
                                  f"mode {mode}", same_sign=True)
    B.grf_ctx_use_tensor_cores(ctx.handle, 1)
    small = B.grf_attn_workspace_bytes(1, N, m, 64, B.GRF_DTYPE_BF16)
    assert torch.equal(out[1], api.masked_linear_attn(ctx, feat, qd, kd, vd, workspace_bytes=small))
    with pytest.raises(B.GrfError):         # the caller never asked for the mask
        api.masked_attn_mhat(ctx, feat, qd, kd, vd)
    feat.free()
    ctx.close()
