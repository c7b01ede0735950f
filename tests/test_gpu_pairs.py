"""States used where they are made (records of (row, node) pairs): lists of every length class against the oracle, both types, all
shapes of the route; records of every width give the same bits; the route agrees with whole states."""
import numpy as np
import pytest
import torch

import oracle
from tests import helpers
from tests.helpers import kernel_classes
from workloads import configs, tensors

pytestmark = pytest.mark.gpu


def csr(rng, rows, cols, lengths):
    c = [np.sort(rng.choice(cols, size=min(n, cols), replace=False)) for n in lengths]
    rp = np.concatenate([[0], np.cumsum([len(x) for x in c])]).astype(np.int32)
    c = np.concatenate(c).astype(np.int32)
    return oracle.CSR(rp, c, rng.uniform(0.1, 1.0, c.size).astype(np.float32), None, (rows, cols))


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("m", [16, 32, 64])
@pytest.mark.parametrize("d", [32, 64])
def test_lists_of_every_length(m, d, dtype):
    """Nodes with 0, 1, 7 .. 9, 15 .. 17, 31 .. 33 and 100 keys and as many queries (chunks are of 8, 16 and 32), rows with none."""
    from paper_2410_03462_b200 import api, binding as B
    ctx = api.Context(0)
    rng = np.random.default_rng(m + d)
    N, R, G = 3001, 2569, 24
    lengths = (0, 1, 7, 8, 9, 15, 16, 17, 31, 32, 33, 100)
    # columns of these lengths: every node's queries and keys in two different orders
    phi_t = csr(rng, R, N, [lengths[l % 12] for l in range(R)])
    psi_t = csr(rng, R, N, [lengths[(l + l // 12) % 12] for l in range(R)])
    Phi, Psi = oracle.transpose(phi_t), oracle.transpose(psi_t)
    feat = api.features_from_csr(ctx, N, R, (Phi.rowptr, Phi.col, Phi.val), (Psi.rowptr, Psi.col, Psi.val))
    q, k, v = tensors.qkv(G, N, m, d, dtype, 5)
    qd, kd, vd = q.cuda(), k.cuda(), v.cuda()
    B.grf_ctx_use_tensor_cores(ctx.handle, 2)               # never over the mask
    (out, den), ran = kernel_classes(B, ctx, lambda: api.masked_linear_attn(ctx, feat, qd, kd, vd, want_den=True))
    assert "scan" in ran and "mhat_attention" not in ran, ran
    pick = [0, 1, G - 1]
    ref = oracle.attn_sparse(tensors.widen(q[pick]), tensors.widen(k[pick]), tensors.widen(v[pick]), Phi, oracle.transpose(Psi))
    helpers.assert_attn_close(out[pick].float().cpu().numpy(), ref, helpers.TOL[dtype], den[pick].cpu().numpy(), min_ok=0.3)
    # one problem's workspace: the same bits; whole states: the same values (every difference is within both routes' bounds)
    small = B.grf_attn_workspace_bytes(1, R, m, d, B.dtype_code(vd))
    assert torch.equal(out, api.masked_linear_attn(ctx, feat, qd, kd, vd, workspace_bytes=small))
    B.grf_ctx_use_tensor_cores(ctx.handle, 0)
    other, ran = kernel_classes(B, ctx, lambda: api.masked_linear_attn(ctx, feat, qd, kd, vd))
    assert "scan" not in ran, ran
    helpers.assert_attn_close(other[pick].float().cpu().numpy(), ref, helpers.TOL[dtype], min_ok=0.3)
    feat.free()
    ctx.close()


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("m,d,G", [(16, 32, 24), (16, 64, 24), (32, 32, 24), (32, 64, 24), (64, 32, 24), (64, 64, 24), (32, 64, 2), (64, 32, 2)])
def test_hub_nodes(m, d, G, dtype):
    """Nodes with more than 512 keys and queries (2 problems: 280 or so) are a CTA's work, with more than 8192 (2048) a cluster's: right
    below, at and above that, one side long only, nodes without keys or with a few (warps without a share), hubs that every row visits."""
    from paper_2410_03462_b200 import api, binding as B
    ctx = api.Context(0)
    rng = np.random.default_rng(m + d)
    N, R = 6001, 1500
    sides = [(100, x) for x in range(170, 200)] + [(1024, 1024), (1024, 1025), (1000, 1047), (256, 256), (256, 257), (1, 511), (511, 1), (1, 512), (512, 1), (0, 600), (600, 0), (7, 700), (700, 7), (6001, 6001),
             (2049, 33), (31, 2051), (513, 6001), (4096, 4096), (4096, 4097), (6001, 2192)]
    sides += [(40, 30)] * (R - len(sides))
    order = rng.permutation(R)
    phi_t = csr(rng, R, N, [sides[x][1] for x in order])
    psi_t = csr(rng, R, N, [sides[x][0] for x in order])
    Phi, Psi = oracle.transpose(phi_t), oracle.transpose(psi_t)
    feat = api.features_from_csr(ctx, N, R, (Phi.rowptr, Phi.col, Phi.val), (Psi.rowptr, Psi.col, Psi.val))
    q, k, v = tensors.qkv(G, N, m, d, dtype, 5)
    qd, kd, vd = q.cuda(), k.cuda(), v.cuda()
    B.grf_ctx_use_tensor_cores(ctx.handle, 2)
    (out, den), ran = kernel_classes(B, ctx, lambda: api.masked_linear_attn(ctx, feat, qd, kd, vd, want_den=True))
    assert "scan" in ran, ran
    pick = [0, G - 1]
    ref = oracle.attn_sparse(tensors.widen(q[pick]), tensors.widen(k[pick]), tensors.widen(v[pick]), Phi, oracle.transpose(Psi))
    helpers.assert_attn_close(out[pick].float().cpu().numpy(), ref, helpers.TOL[dtype], den[pick].cpu().numpy(), min_ok=0.3)
    # other shares of the batch: the same bits, every time
    small = B.grf_attn_workspace_bytes(1, R, m, d, B.dtype_code(vd))
    for _ in range(3):
        assert torch.equal(out, api.masked_linear_attn(ctx, feat, qd, kd, vd, workspace_bytes=small))
    feat.free()
    ctx.close()


@pytest.mark.parametrize("R", [3, 1023, 1024, 5000])
def test_entries_that_do_not_fill_a_cta(R):
    """The regrouping counts 1024 entries at a time in shared memory, in places that columns of one hash compete for: numbers of entries
    around 1024 and 4, columns that share places by chance and one that all rows use."""
    from paper_2410_03462_b200 import api, binding as B
    ctx = api.Context(0)
    rng = np.random.default_rng(R)
    for nnz_extra in (0, 1, 2, 3):
        N, G, m, d = 8000, 12, 32, 64
        lengths = np.full(N, min(R, 9))
        lengths[:nnz_extra] += 1 if R > 9 else 0
        Phi = csr(rng, N, R, lengths)
        hub = Phi.rowptr[:-1]
        Phi.col[hub] = 0                        # the first entry of every row (columns ascend)
        Psi = csr(rng, N, R, [min(R, 9)] * N)
        feat = api.features_from_csr(ctx, N, R, (Phi.rowptr, Phi.col, Phi.val), (Psi.rowptr, Psi.col, Psi.val))
        q, k, v = tensors.qkv(G, N, m, d, "fp32", 5)
        B.grf_ctx_use_tensor_cores(ctx.handle, 2)
        (out, den), ran = kernel_classes(B, ctx, lambda: api.masked_linear_attn(ctx, feat, q.cuda(), k.cuda(), v.cuda(), want_den=True))
        assert "scan" in ran, ran
        ref = oracle.attn_sparse(tensors.widen(q[:1]), tensors.widen(k[:1]), tensors.widen(v[:1]), Phi, oracle.transpose(Psi))
        helpers.assert_attn_close(out[:1].float().cpu().numpy(), ref, helpers.TOL["fp32"], den[:1].cpu().numpy(), min_ok=0.3)
        feat.free()
    ctx.close()


def test_few_nodes_for_many_rows():
    """Three nodes: all of them long, whatever the average.  (bf16 takes whole states by tiles there.)"""
    from paper_2410_03462_b200 import api, binding as B
    ctx = api.Context(0)
    rng = np.random.default_rng(3)
    N, R, G, m, d, dtype = 20011, 3, 16, 32, 64, "fp32"
    Phi, Psi = csr(rng, N, R, [1 + i % 3 for i in range(N)]), csr(rng, N, R, [2] * N)
    feat = api.features_from_csr(ctx, N, R, (Phi.rowptr, Phi.col, Phi.val), (Psi.rowptr, Psi.col, Psi.val))
    q, k, v = tensors.qkv(G, N, m, d, dtype, 5)
    B.grf_ctx_use_tensor_cores(ctx.handle, 2)
    (out, den), ran = kernel_classes(B, ctx, lambda: api.masked_linear_attn(ctx, feat, q.cuda(), k.cuda(), v.cuda(), want_den=True))
    assert "scan" in ran, ran
    pick = [0, G - 1]
    ref = oracle.attn_sparse(tensors.widen(q[pick]), tensors.widen(k[pick]), tensors.widen(v[pick]), Phi, oracle.transpose(Psi))
    helpers.assert_attn_close(out[pick].float().cpu().numpy(), ref, helpers.TOL[dtype], den[pick].cpu().numpy(), min_ok=0.3)
    feat.free()
    ctx.close()


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("m,d", [(16, 32), (32, 64), (64, 32)])
def test_infinite_sums_stay_infinite(m, d, dtype):
    """Positive features throughout: a row that uses an infinite value, or whose sum leaves the range of fp32, gives infinity of
    that sign as a plain sum does, other columns and other rows what they give without it."""
    from paper_2410_03462_b200 import api, binding as B
    ctx = api.Context(0)
    rng = np.random.default_rng(m)
    N, R, G = 2003, 1500, 24
    Phi, Psi = csr(rng, N, R, [25 + i % 40 for i in range(N)]), csr(rng, N, R, [25] * N)
    feat = api.features_from_csr(ctx, N, R, (Phi.rowptr, Phi.col, Phi.val), (Psi.rowptr, Psi.col, Psi.val))
    q, k, v = (t.cuda() for t in tensors.qkv(G, N, m, d, dtype, 5))
    q, k = q.abs() + 0.25, k.abs() + 0.25
    B.grf_ctx_use_tensor_cores(ctx.handle, 2)
    want = api.masked_linear_attn(ctx, feat, q, k, v)
    bad = v.clone()
    bad[1, 7, 3], bad[2, 11, 5] = float("inf"), -float("inf")
    bad[3, 13, 9] = 2.0 ** 126                                   # finite; its sums are not
    out, ran = kernel_classes(B, ctx, lambda: api.masked_linear_attn(ctx, feat, q, k, bad))
    assert "scan" in ran, ran
    # rows that reach a node: the support of Phi Psi^T
    rows = np.zeros((N, R), bool)
    rows[np.repeat(np.arange(N), np.diff(Phi.rowptr)), Phi.col] = True
    for g, node, column, sign in ((1, 7, 3, 1), (2, 11, 5, -1)):
        reached = torch.from_numpy(rows[:, Psi.col[Psi.rowptr[node]:Psi.rowptr[node + 1]]].any(1)).cuda()
        assert reached.any() and not reached.all()
        assert (out[g, reached, column] == sign * float("inf")).all()
        out[g, reached, column] = want[g, reached, column]
    assert not out.isnan().any() and (out[3, :, 9] == float("inf")).any()
    out[3, :, 9] = want[3, :, 9]
    assert torch.equal(out, want)
    feat.free()
    ctx.close()


@pytest.mark.parametrize("m,d", [(32, 64), (32, 32), (16, 64)])
def test_records_of_every_width_give_the_same_bits(m, d):
    """An expander whose whole records are larger than the context's scratch: a full workspace holds them, one problem's only
    records of 16 columns."""
    from paper_2410_03462_b200 import api, binding as B
    ctx = api.Context(0)
    w = configs.sweep(17)
    N = 1 << 17
    f = oracle.deconvolve(w.alpha).astype(np.float32)
    feat = api.sample(ctx, api.DeviceGraph(w.graph()), 3, w.n_walks, w.p_halt, w.max_len, f)
    gen = torch.Generator(device="cuda").manual_seed(1)
    G = 4
    q = torch.relu(torch.randn(G, N, m, generator=gen, device="cuda")).bfloat16()
    k = torch.relu(torch.randn(G, N, m, generator=gen, device="cuda")).bfloat16()
    v = torch.randn(G, N, d, generator=gen, device="cuda").bfloat16()
    out, ran = kernel_classes(B, ctx, lambda: api.masked_linear_attn(ctx, feat, q, k, v))
    assert "scan" in ran, ran
    for problems in (1, 2, 3):
        small = B.grf_attn_workspace_bytes(problems, N, m, d, B.GRF_DTYPE_BF16)
        assert torch.equal(out, api.masked_linear_attn(ctx, feat, q, k, v, workspace_bytes=small))
    B.grf_ctx_use_tensor_cores(ctx.handle, 0)
    other = api.masked_linear_attn(ctx, feat, q, k, v)
    # both round S and the outputs to bf16 (2^-9 each): the relative difference of two such results is below 2^-7
    assert float((out.float() - other.float()).norm() / other.float().norm()) < 2.0 ** -7
    feat.free()
    ctx.close()


def test_capture_keeps_to_whole_states():
    """The pairs' buffers belong to the context and may be replaced later: a captured call, also one on a sample whose sizes are
    not known yet, uses the caller's, and its replay gives the bits of whole states."""
    from paper_2410_03462_b200 import api, binding as B
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        ctx = api.Context(0)
        w = configs.point_cloud_4096(1500)
        f = oracle.deconvolve(w.alpha).astype(np.float32)
        q, k, v = (t.cuda() for t in tensors.qkv(4, 1500, 32, 64, "fp32", 4))
        ws = torch.empty(B.grf_attn_workspace_bytes(4, 1500, 32, 64, B.GRF_DTYPE_F32), dtype=torch.uint8, device="cuda")
        den = torch.empty(4, 1500, device="cuda")
        out = torch.empty_like(v)
        dg = api.DeviceGraph(w.graph())
        feat = api.sample(ctx, dg, 3, w.n_walks, w.p_halt, w.max_len, f)

        def call():
            B.grf_masked_linear_attn(ctx.handle, feat.handle, 4, 1500, 32, 64, B.GRF_DTYPE_F32, q, k, v, out, den, ws, ws.numel())
            return out.clone()

        direct, ran = kernel_classes(B, ctx, call)
        assert "scan" in ran, ran
        B.grf_ctx_use_tensor_cores(ctx.handle, 0)
        whole = call()
        B.grf_ctx_use_tensor_cores(ctx.handle, 1)
        feat.handle = B.grf_sample(ctx.handle, dg.N, dg.rowptr, dg.col, dg.w, 3, w.n_walks, w.p_halt, w.max_len, f, None, feat.handle)
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            call()
        out.zero_()
        graph.replay()
        s.synchronize()
        assert torch.equal(out, whole)
        # two fp32 evaluations of the same sums: the bound of fp32 outputs
        assert float((out - direct).norm() / direct.norm()) < 1e-5
        del graph
        feat.free()
        ctx.close()


@pytest.mark.parametrize("dtype,N,G,walks,length", [("fp32", 1500, 4, 32, 12), ("bf16", 20000, 8, 8, 6)])
def test_capture_behind_calls_by_pairs_and_before_larger_ones(dtype, N, G, walks, length):
    """On a fresh context, without room for denominators: the eager call uses the states where they are made, the captured one needs
    memory (bf16: and the coefficients of the gather by tiles) that no call has asked for yet, and larger calls leave it to the graph."""
    from paper_2410_03462_b200 import api, binding as B
    m, d = 32, 64
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        ctx = api.Context(0)
        w = configs.point_cloud_4096(N)
        f = oracle.deconvolve(w.alpha).astype(np.float32)[:length + 1]
        feat = api.sample(ctx, api.DeviceGraph(w.graph()), 3, walks, w.p_halt, length, f)
        q, k, v = (t.cuda() for t in tensors.qkv(G, N, m, d, dtype, 4))
        ws = torch.empty(B.grf_attn_workspace_bytes(G, N, m, d, B.dtype_code(v)), dtype=torch.uint8, device="cuda")
        B.grf_ctx_use_tensor_cores(ctx.handle, 2)
        direct, ran = kernel_classes(B, ctx, lambda: api.masked_linear_attn(ctx, feat, q, k, v, workspace=ws))
        assert "scan" in ran, ran
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            out = api.masked_linear_attn(ctx, feat, q, k, v, workspace=ws)
        B.grf_ctx_use_tensor_cores(ctx.handle, 0 if dtype == "fp32" else 3)
        whole = api.masked_linear_attn(ctx, feat, q, k, v, workspace=ws)
        q2, k2, v2 = (t.cuda() for t in tensors.qkv(2 * G, N, m, d, dtype, 5))
        larger = api.masked_linear_attn(ctx, feat, q2, k2, v2)
        other = api.Context(0)                          # blocks that have been given back would come to it
        B.grf_ctx_use_tensor_cores(other.handle, 0 if dtype == "fp32" else 3)
        beside = api.masked_linear_attn(other, feat, q2[:G], k2[:G], v2[:G])
        for _ in range(2):
            out.zero_()
            graph.replay()
            s.synchronize()
            assert torch.equal(out, whole)
        assert torch.equal(larger[:G], beside)
        # both round S and the outputs to bf16 (2^-9 each); fp32: two evaluations of the same sums
        assert float((out.float() - direct.float()).norm() / direct.float().norm()) < (1e-5 if dtype == "fp32" else 2.0 ** -7)
        del graph
        feat.free()
        ctx.close()
        other.close()


def test_captured_remodulation_before_the_gather_by_tiles():
    """The coefficients that the gather reads follow the values that the graph itself gives Phi, replay after replay, and eager calls
    between replays see the features as they are."""
    from paper_2410_03462_b200 import api, binding as B
    N, m, d = 2048, 128, 64
    w = configs.point_cloud_4096(N)
    f = oracle.deconvolve(w.alpha).astype(np.float32)
    new = (f * np.linspace(1.0, 1.3, f.size)).astype(np.float32)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        ctx = api.Context(0)
        B.grf_ctx_use_tensor_cores(ctx.handle, 3)
        B.grf_ctx_keep_walks(ctx.handle, True)
        feat = api.sample(ctx, api.DeviceGraph(w.graph()), 7, w.n_walks, w.p_halt, w.max_len, f)
        q, k, v = (t.cuda() for t in tensors.qkv(4, N, m, d, "bf16", 5))
        ws = torch.empty(B.grf_attn_workspace_bytes(4, N, m, d, B.dtype_code(v)), dtype=torch.uint8, device="cuda")

        def attend():
            return api.masked_linear_attn(ctx, feat, q, k, v, workspace=ws)

        def step(coefficients):
            B.grf_remodulate(ctx.handle, feat.handle, w.max_len, coefficients, None)
            return attend()

        want, old = step(new).clone(), step(f).clone()
        assert not torch.equal(want, old)
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            got = step(new)
        assert torch.equal(attend(), old)               # nothing of the graph has run
        for _ in range(2):
            got.zero_()
            graph.replay()
            assert torch.equal(got, want) and torch.equal(attend(), want)
            assert torch.equal(step(f), old)
        del graph
        feat.free()
        ctx.close()
