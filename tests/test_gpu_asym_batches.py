"""Asymmetric attention around its batches of 32 non-zeros and its whole and partial steps of value rows."""
import numpy as np
import pytest

import oracle
from tests import helpers
from workloads import tensors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,d", [(8, 8), (8, 128), (16, 64), (32, 64), (128, 16), (128, 128)])
def test_rows_around_batches_and_steps(m, d):
    from paper_2410_03462_b200 import api, binding as B
    ctx = api.Context(0)
    lengths = [0, 1, 2, 3, 7, 8, 9, 15, 16, 17, 23, 24, 25, 31, 32, 33, 39, 40, 41, 47, 48, 63, 64, 65, 95, 96, 97]
    rng = np.random.default_rng(m + d)
    N, G = len(lengths) * 4, 3
    rows = [np.sort(rng.choice(N, size=lengths[i % len(lengths)], replace=False)) for i in range(N)]
    rp = np.concatenate([[0], np.cumsum([len(c) for c in rows])]).astype(np.int32)
    col = np.concatenate(rows).astype(np.int32)
    Phi = oracle.CSR(rp, col, rng.uniform(0.1, 1.0, col.size).astype(np.float32), None, (N, N))
    eye = (np.arange(N + 1, dtype=np.int32), np.arange(N, dtype=np.int32), np.ones(N, np.float32))
    feat = api.features_from_csr(ctx, N, N, (Phi.rowptr, Phi.col, Phi.val), eye)
    for dtype in ("fp32", "bf16"):
        q, k, v = tensors.qkv(G, N, m, d, dtype, 3)
        q, k = (q.float() * 0.2 + 0.05).to(q.dtype), (k.float() * 0.2 + 0.05).to(k.dtype)
        for softmax in (False, True):
            ref = oracle.attn_bruteforce(tensors.widen(q), tensors.widen(k), tensors.widen(v), Phi.dense(),
                                         kernel="exp" if softmax else "linear")
            out = api.masked_attn_asym(ctx, feat, q.cuda(), k.cuda(), v.cuda(), softmax=softmax)
            B.grf_ctx_check(ctx.handle)
            helpers.assert_attn_close(out.float().cpu().numpy(), ref, helpers.TOL[dtype], None,
                                      f"m{m} d{d} {dtype} softmax={softmax}")
    feat.free()
    ctx.close()
