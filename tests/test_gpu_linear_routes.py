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
@pytest.mark.parametrize("N,G,d", [(127, 8, 64), (129, 40, 64), (1000, 96, 64), (64, 2, 64), (1000, 2, 64), (128, 96, 32), (1000, 97, 32)])
def test_both_routes_match_oracle(N, G, d, m):
    from paper_2410_03462_b200 import api, binding as B
    ctx = api.Context(0)
    w = configs.point_cloud_4096(N)
    g = w.graph()
    f = oracle.deconvolve(w.alpha).astype(np.float32)
    feat = api.sample(ctx, api.DeviceGraph(g), 3, w.n_walks, w.p_halt, w.max_len, f)
    Phi, _, PsiT, _, _ = helpers.oracle_features(w, g, 3, f)
    q, k, v = tensors.qkv(G, N, m, d, "bf16", 4)
    qd, kd, vd = q.cuda(), k.cuda(), v.cuda()
    one = slice(G - 1, G)
    ref = oracle.attn_sparse(tensors.widen(q[one]), tensors.widen(k[one]), tensors.widen(v[one]), Phi, PsiT)
    out = {}
    for mode in (1, 2, 3):                  # 1: the cheaper route, 2: always the states, 3: all on the tensor cores
        B.grf_ctx_use_tensor_cores(ctx.handle, mode)
        out[mode], den = api.masked_linear_attn(ctx, feat, qd, kd, vd, want_den=True)
        B.grf_ctx_check(ctx.handle)
        helpers.assert_attn_close(out[mode][one].float().cpu().numpy(), ref, helpers.TOL["bf16"], den[one].cpu().numpy(),
                                  f"mode {mode}", same_sign=True)
    B.grf_ctx_use_tensor_cores(ctx.handle, 1)
    small = B.grf_attn_workspace_bytes(1, N, m, d, B.GRF_DTYPE_BF16)
    assert torch.equal(out[1], api.masked_linear_attn(ctx, feat, qd, kd, vd, workspace_bytes=small))
    B.grf_ctx_use_tensor_cores(ctx.handle, 2)
    assert torch.equal(out[2], api.masked_linear_attn(ctx, feat, qd, kd, vd, workspace_bytes=small))
    B.grf_ctx_use_tensor_cores(ctx.handle, 1)
    with pytest.raises(B.GrfError):         # the caller never asked for the mask
        api.masked_attn_mhat(ctx, feat, qd, kd, vd)
    feat.free()
    ctx.close()


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("R,m,d", [(300, 32, 64), (36863, 32, 64), (36865, 128, 8), (147457, 16, 32), (294913, 8, 16)])
def test_sliced_gather_widths(R, m, d, dtype):
    """The plain-ALU gather takes tiles in slices of 2 KB or 512 bytes by the number of nodes (smaller tiles whole): rows of Phi
    with 0, 1, 31, 32, 33 and 70 non-zeros over few and many nodes."""
    from paper_2410_03462_b200 import api, binding as B
    ctx = api.Context(0)
    rng = np.random.default_rng(R + m)
    N, G = 67, 2

    def csr(lengths):
        cols = [np.sort(rng.choice(R, size=n, replace=False)) for n in lengths]
        rp = np.concatenate([[0], np.cumsum([len(c) for c in cols])]).astype(np.int32)
        c = np.concatenate(cols).astype(np.int32)
        return oracle.CSR(rp, c, rng.uniform(0.1, 1.0, c.size).astype(np.float32), None, (N, R))

    Phi = csr([(0, 1, 31, 32, 33, 70)[i % 6] for i in range(N)])
    # every node that a row of Phi touches has keys
    keys = np.tile(np.unique(Phi.col), 2)
    Psi = csr([3] * N)
    Psi.col[:] = np.sort(rng.choice(np.unique(keys), size=(N, 3)), axis=1).ravel()
    dup = [i for i in range(N) if len(set(Psi.col[3 * i:3 * i + 3])) < 3]
    for i in dup:
        Psi.col[3 * i:3 * i + 3] = np.sort(np.unique(keys)[[0, 5, 9]])
    PsiT = oracle.transpose(Psi)
    feat = api.features_from_csr(ctx, N, R, (Phi.rowptr, Phi.col, Phi.val), (Psi.rowptr, Psi.col, Psi.val))
    q, k, v = tensors.qkv(G, N, m, d, dtype, 5)
    q = (q.float() + 0.1).to(q.dtype)
    k = (k.float() + 0.1).to(k.dtype)
    ref = oracle.attn_sparse(tensors.widen(q), tensors.widen(k), tensors.widen(v), Phi, PsiT)
    B.grf_ctx_use_tensor_cores(ctx.handle, 0)
    out, den = api.masked_linear_attn(ctx, feat, q.cuda(), k.cuda(), v.cuda(), want_den=True)
    B.grf_ctx_check(ctx.handle)
    helpers.assert_attn_close(out.float().cpu().numpy(), ref, helpers.TOL[dtype], den.cpu().numpy(), f"R={R}", min_ok=0.3)
    feat.free()
    ctx.close()


@pytest.mark.parametrize("N,G", [(1000, 2), (1000, 96)])        # by the states, over the mask
def test_a_mask_that_the_caller_formed_changes_no_bit_of_the_main_call(N, G):
    from paper_2410_03462_b200 import api, binding as B
    ctx = api.Context(0)
    w = configs.point_cloud_4096(N)
    f = oracle.deconvolve(w.alpha).astype(np.float32)
    feat = api.sample(ctx, api.DeviceGraph(w.graph()), 3, w.n_walks, w.p_halt, w.max_len, f)
    q, k, v = (t.cuda() for t in tensors.qkv(G, N, 32, 64, "bf16", 4))
    before = api.masked_linear_attn(ctx, feat, q, k, v)
    B.grf_features_materialise(ctx.handle, feat.handle)
    assert torch.equal(before, api.masked_linear_attn(ctx, feat, q, k, v))
    api.masked_attn_mhat(ctx, feat, q, k, v)
    assert torch.equal(before, api.masked_linear_attn(ctx, feat, q, k, v))
    feat.free()
    ctx.close()


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("m,d", [(8, 8), (16, 16), (16, 128), (64, 64), (128, 32)])
def test_plain_gather_beside_its_denominators(m, d, dtype):
    """The gather starts while the denominators are formed: rows of 0, 1 and 4000 entries side by side, call after call with other
    inputs into the same outputs, so that a denominator read too early is another call's."""
    from paper_2410_03462_b200 import api, binding as B
    rng = np.random.default_rng(m + d)
    N, R, G = 515, 4003, 3
    lengths = [(0, 1, 4000, 33, 32)[i % 5] if i < 40 else 20 for i in range(N)]
    rows = [np.sort(rng.choice(R, size=n, replace=False)) for n in lengths]
    rp = np.concatenate([[0], np.cumsum([len(c) for c in rows])]).astype(np.int32)
    c = np.concatenate(rows).astype(np.int32)
    Phi = oracle.CSR(rp, c, rng.uniform(0.1, 1.0, c.size).astype(np.float32), None, (N, R))
    cols = [np.sort(rng.choice(R, size=30, replace=False)) for _ in range(N)]
    Psi = oracle.CSR(np.arange(0, 30 * N + 1, 30, dtype=np.int32), np.concatenate(cols).astype(np.int32),
                     rng.uniform(0.1, 1.0, 30 * N).astype(np.float32), None, (N, R))
    ctx = api.Context(0)
    B.grf_ctx_use_tensor_cores(ctx.handle, 0)
    feat = api.features_from_csr(ctx, N, R, (Phi.rowptr, Phi.col, Phi.val), (Psi.rowptr, Psi.col, Psi.val))
    inputs = [tensors.qkv(G, N, m, d, dtype, seed) for seed in (1, 2)]
    ws = torch.empty(B.grf_attn_workspace_bytes(G, R, m, d, B.dtype_code(inputs[0][0])), dtype=torch.uint8, device="cuda")
    out, den = torch.empty_like(inputs[0][2], device="cuda"), torch.empty((G, N), device="cuda")
    got = []
    for q, k, v in [[t.cuda() * (1 + 3 * x) for t in inputs[x]] for x in (0, 1, 0, 1)]:
        B.grf_masked_linear_attn(ctx.handle, feat.handle, G, N, m, d, B.dtype_code(v), q, k, v, out, den, ws, ws.numel())
        got.append((out.clone(), den.clone()))
    for x in (0, 1):
        assert torch.equal(got[x][0], got[x + 2][0]) and torch.equal(got[x][1], got[x + 2][1])
        q, k, v = (tensors.widen(t * (1 + 3 * x)) for t in inputs[x])
        ref = oracle.attn_sparse(q, k, v, Phi, oracle.transpose(Psi))
        helpers.assert_attn_close(got[x][0].float().cpu().numpy(), ref, helpers.TOL[dtype], got[x][1].cpu().numpy(), min_ok=0.3)
    feat.free()
    ctx.close()


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("m,d", [(16, 16), (32, 64), (8, 64), (16, 128), (8, 8)])
def test_denominators_inside_and_by_themselves_give_the_same_bits(m, d, dtype):
    """While a sample runs only the expected number of its entries is known (more than 16 a row here; the real one is smaller), which
    makes the plain gather form the denominators by themselves; afterwards it forms them inside."""
    from paper_2410_03462_b200 import api, binding as B
    ctx = api.Context(0)
    B.grf_ctx_use_tensor_cores(ctx.handle, 0)
    N = 125
    w = configs.point_cloud_4096(N)
    dg = api.DeviceGraph(w.graph())
    f = oracle.deconvolve(w.alpha).astype(np.float32)
    q, k, v = (t.cuda() for t in tensors.qkv(1, N, m, d, dtype, 4))
    ws = torch.empty(B.grf_attn_workspace_bytes(1, N, m, d, B.dtype_code(v)), dtype=torch.uint8, device="cuda")
    out, den = torch.empty_like(v), torch.empty((1, N), device="cuda")
    feat = api.sample(ctx, dg, 3, w.n_walks, w.p_halt, w.max_len, f)

    def call():
        B.grf_ctx_enable_timing(ctx.handle, True)
        B.grf_masked_linear_attn(ctx.handle, feat.handle, 1, N, m, d, B.dtype_code(v), q, k, v, out, den, ws, ws.numel())
        launches = B.grf_ctx_kernel_times(ctx.handle)["row_denominators"][1]
        B.grf_ctx_enable_timing(ctx.handle, False)
        return launches, out.clone(), den.clone()

    for _ in range(2):                      # the second sample leaves its sizes open
        feat.handle = B.grf_sample(ctx.handle, dg.N, dg.rowptr, dg.col, dg.w, 3, 3, w.p_halt, w.max_len, f, None, feat.handle)
    running = call()
    assert feat.shape(0)[2] <= 16 * N       # reads the sizes
    settled = call()
    assert torch.equal(running[1], settled[1]) and torch.equal(running[2], settled[2])
    assert (running[0], settled[0]) == (1, 0)       # both ways were taken
    feat.free()
    ctx.close()
