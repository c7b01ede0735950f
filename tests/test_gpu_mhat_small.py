"""Masked attention on graphs of at most 512 nodes: key lists of whole aligned tiles, several problems per CTA."""
import numpy as np
import pytest
import torch

import oracle
from tests import helpers
from workloads import tensors

pytestmark = pytest.mark.gpu


def band_features(N, kind, rng, width=1):
    """Phi, Psi (N x N) whose blocks of 128 rows reach: every key; a few keys of one tile; nothing; keys far apart."""
    far = np.unique(np.clip([at + x for at in (0, N // 2, N - width) for x in range(width)], 0, N - 1))
    rows_phi, rows_psi = [], []
    for i in range(N):
        blk = i // 128
        if kind == "dense":
            c = rng.choice(N, size=min(N, 20), replace=False)
        elif kind == "local" or (kind == "mixed" and blk % 4 == 0):
            c = np.unique(np.clip(i + rng.integers(-2 * width, 2 * width + 1, size=4 * width), 0, N - 1))
        elif kind == "mixed" and blk % 4 == 1:
            c = np.array([], dtype=np.int64)
        else:
            c = np.unique(rng.choice(far, size=2 * width))
        rows_phi.append(np.sort(c))
        rows_psi.append(np.unique(np.clip([i, i + 1], 0, N - 1)))

    def csr(rows):
        rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
        col = np.concatenate(rows).astype(np.int32) if rp[-1] else np.zeros(0, np.int32)
        return oracle.CSR(rp, col, rng.uniform(0.1, 1.0, col.size).astype(np.float32), None, (N, N))

    return csr(rows_phi), csr(rows_psi)


@pytest.mark.parametrize("kind", ["dense", "local", "mixed"])
@pytest.mark.parametrize("N,G,m,d", [(1, 3, 16, 64), (63, 40, 32, 64), (64, 1, 64, 64), (65, 700, 16, 64), (128, 1301, 32, 32),
                                     (129, 777, 64, 32), (196, 777, 64, 64), (257, 150, 32, 64), (320, 650, 16, 32),
                                     (449, 130, 64, 64), (449, 403, 32, 32), (512, 200, 32, 64), (513, 20, 32, 64)])
def test_small_graphs(N, G, m, d, kind):
    """d = 32 is served by the main call alone, over the mask where that is the cheaper way: enough problems, wider rows."""
    from paper_2410_03462_b200 import api, binding as B
    ctx = api.Context(0)
    rng = np.random.default_rng(N + m)
    Phi, Psi = band_features(N, kind, rng, 1 if d == 64 else 10)
    feat = api.features_from_csr(ctx, N, N, (Phi.rowptr, Phi.col, Phi.val), (Psi.rowptr, Psi.col, Psi.val))
    q, k, v = tensors.qkv(G, N, m, d, "bf16", 5)
    qd, kd, vd = q.cuda() + 0.125, k.cuda() + 0.125, v.cuda()
    B.grf_features_materialise(ctx.handle, feat.handle)
    if d == 64:
        out, den = api.masked_attn_mhat(ctx, feat, qd, kd, vd, want_den=True)
    else:
        (out, den), ran = helpers.kernel_classes(B, ctx, lambda: api.masked_linear_attn(ctx, feat, qd, kd, vd, want_den=True))
        assert "mhat_attention" in ran, ran
    B.grf_ctx_check(ctx.handle)
    pick = sorted({0, G // 2, G - 1})
    ref = oracle.attn_sparse(tensors.widen(qd[pick].cpu()), tensors.widen(kd[pick].cpu()), tensors.widen(v[pick]), Phi, oracle.transpose(Psi))
    helpers.assert_attn_close(out[pick].float().cpu().numpy(), ref, helpers.TOL["bf16"], den[pick].cpu().numpy(), min_ok=0.0)
    # every problem against whole states on the plain ALUs: both round to bf16 (2^-9) at most three times
    B.grf_ctx_use_tensor_cores(ctx.handle, 0)
    other = api.masked_linear_attn(ctx, feat, qd, kd, vd)
    assert float((out.float() - other.float()).norm()) <= 2.0 ** -7 * float(other.float().norm())
    empty = np.diff(Phi.rowptr) == 0
    assert not out[:, torch.from_numpy(empty).cuda()].any() and not out.isnan().any()
    feat.free()
    ctx.close()


def reached_keys(Phi, Psi, N, rows):
    """Keys that any of the rows reaches: the support of Phi Psi^T."""
    nodes = np.zeros(N, bool)
    for r in rows:
        nodes[Phi.col[Phi.rowptr[r]:Phi.rowptr[r + 1]]] = True
    keys = np.zeros(N, bool)
    for j in range(N):
        keys[j] = nodes[Psi.col[Psi.rowptr[j]:Psi.rowptr[j + 1]]].any()
    return keys


@pytest.mark.parametrize("kind", ["local", "mixed", "far"])
@pytest.mark.parametrize("N,G,m,d", [(65, 9, 16, 64), (129, 7, 32, 64), (196, 40, 64, 64), (300, 150, 32, 64), (449, 300, 64, 32), (512, 400, 16, 32), (650, 8, 32, 64)])
def test_keys_that_no_row_of_a_block_reaches_do_not_matter(N, G, m, d, kind):
    """Infinities and NaNs in their rows of K and V (padded nodes, say) leave the block's bits alone, also where they lie between,
    before or behind keys that it does reach; the mask's own rows hold zeros there."""
    from paper_2410_03462_b200 import api, binding as B
    ctx = api.Context(0)
    rng = np.random.default_rng(N + m)
    Phi, Psi = band_features(N, kind, rng, 1 if d == 64 else 10)
    feat = api.features_from_csr(ctx, N, N, (Phi.rowptr, Phi.col, Phi.val), (Psi.rowptr, Psi.col, Psi.val))
    q, k, v = (t.cuda() for t in tensors.qkv(G, N, m, d, "bf16", 5))
    B.grf_features_materialise(ctx.handle, feat.handle)
    if d == 64:
        def attn(k, v):
            return api.masked_attn_mhat(ctx, feat, q, k, v, want_den=True)
    else:
        def attn(k, v):
            result, ran = helpers.kernel_classes(B, ctx, lambda: api.masked_linear_attn(ctx, feat, q, k, v, want_den=True))
            assert "mhat_attention" in ran, ran
            return result
    want, want_den = attn(k, v)
    for first in range(0, N, 128):
        rows = np.arange(first, min(N, first + 128))
        free = torch.from_numpy(~reached_keys(Phi, Psi, N, rows)).cuda()
        for bad in (float("nan"), float("inf")):
            k2, v2 = k.clone(), v.clone()
            k2[:, free], v2[:, free] = bad, -bad
            out, den = attn(k2, v2)
            at = slice(first, first + len(rows))
            assert torch.equal(out[:, at], want[:, at]) and torch.equal(den[:, at], want_den[:, at])
    # and a NaN that rows do reach stays one, in its own problem
    k2 = k.clone()
    k2[G // 2, N // 2, 3] = float("nan")
    out, den = attn(k2, v)
    assert out[G // 2].isnan().any() and not out[:G // 2].isnan().any() and not out[G // 2 + 1:].isnan().any()
    mask = torch.empty((N, N), device="cuda")
    B.grf_mask_rows(ctx.handle, feat.handle, N, torch.arange(N, dtype=torch.int32, device="cuda"), mask)
    import scipy.sparse as sp
    dense = (sp.csr_matrix((Phi.val, Phi.col, Phi.rowptr), (N, N)) @ sp.csr_matrix((Psi.val, Psi.col, Psi.rowptr), (N, N)).T).toarray()
    # sums of at most N positive products in fp32, rounded to bf16 once
    assert np.abs(mask.cpu().numpy() - dense).max() <= 2.0 ** -8 * np.abs(dense).max()
    assert (mask.cpu().numpy()[dense == 0] == 0).all()
    feat.free()
    ctx.close()
