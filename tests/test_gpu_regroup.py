"""Row pointers by one launch or three, buckets of every class, and the sizes of a sample that the call did not wait for."""
import numpy as np
import pytest
import torch

import oracle
from tests import helpers
from workloads import configs, graphs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cols", [1, 4095, 4096, 4097, 8193, 262144, 262145])
def test_transpose_around_scan_tiles(cols):
    from paper_2410_03462_b200 import api, binding as B
    ctx = api.Context(0)
    rng = np.random.default_rng(cols)
    rows, per = 300, min(cols, 40)
    c = np.stack([np.sort(rng.choice(cols, size=per, replace=False)) for _ in range(rows)]).astype(np.int32).ravel()
    rp = (np.arange(rows + 1) * per).astype(np.int32)
    v = rng.standard_normal(c.size).astype(np.float32)
    want = oracle.transpose(oracle.CSR(rp, c, v, None, (rows, cols)))
    d = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    out = [torch.empty(cols + 1, dtype=torch.int32, device="cuda"), torch.empty(c.size, dtype=torch.int32, device="cuda"),
           torch.empty(c.size, dtype=torch.float32, device="cuda")]
    B.grf_csr_transpose(ctx.handle, rows, cols, c.size, d(rp), d(c), d(v), *out)
    torch.cuda.synchronize()
    helpers.assert_csr_equal(tuple(t.cpu().numpy() for t in out), want, f"cols={cols}", val_rtol=0)
    ctx.close()


def test_sizes_of_interleaved_samples_and_growing_graphs():
    """Two objects sampled one after the other before either's sizes are read, on graphs whose number of edges grows."""
    from paper_2410_03462_b200 import api
    ctx = api.Context(0)
    w = configs.tiny()
    f = oracle.deconvolve(w.alpha).astype(np.float32)
    feats, gs = [], [graphs.grid_graph(n, n + 1, 0.25, diag) for n, diag in ((3, False), (9, False), (13, True))]
    for g in gs:
        feats.append(api.sample(ctx, api.DeviceGraph(g), 5, w.n_walks, w.p_halt, w.max_len, f))
    for g, feat in zip(gs, feats):
        Phi, Psi, PsiT, _, _ = oracle.sample(g.rowptr, g.col, g.w, 5, w.n_walks, w.p_halt, w.max_len, f)
        for which, want in enumerate((Phi, Psi, PsiT)):
            helpers.assert_csr_equal(feat.to_host(which), want, f"matrix {which}", val_rtol=0)
        feat.free()
    feat = api.sample(ctx, api.DeviceGraph(gs[0]), 5, w.n_walks, w.p_halt, w.max_len, f)
    feat.free()                       # freed before its sizes were read
    ctx.close()


def test_objects_handed_from_one_context_to_another():
    """A producer samples without reading sizes and goes on with larger graphs; a consumer thread with its own context
    takes each object over."""
    import threading

    from paper_2410_03462_b200 import api
    w = configs.tiny()
    f = oracle.deconvolve(w.alpha).astype(np.float32)
    gs = [graphs.grid_graph(n, n + 1, 0.25, n % 2 == 0) for n in (5, 8, 13, 21)]
    producer, consumer = api.Context(0), api.Context(0)
    feats, got, ready = [], [], [threading.Event() for _ in gs]

    def consume():
        for x in range(len(gs)):
            ready[x].wait(60)
            feats[x].ctx = consumer
            got.append([feats[x].to_host(which) for which in range(3)])

    t = threading.Thread(target=consume)
    t.start()
    for x, g in enumerate(gs):
        feats.append(api.sample(producer, api.DeviceGraph(g), 11, w.n_walks, w.p_halt, w.max_len, f))
        producer.stream.synchronize()              # the hand-over is the caller's to order
        ready[x].set()
    t.join()
    for g, feat, matrices in zip(gs, feats, got):
        want = oracle.sample(g.rowptr, g.col, g.w, 11, w.n_walks, w.p_halt, w.max_len, f)[:3]
        for which in range(3):
            helpers.assert_csr_equal(matrices[which], want[which], f"N={g.N} matrix {which}", val_rtol=0)
        feat.free()
    producer.close()
    consumer.close()


def test_one_object_resampled_without_reading_its_sizes():
    """First sample (exact arrays), later ones (arrays for the largest sample), on graphs that grow and shrink."""
    from paper_2410_03462_b200 import api
    ctx = api.Context(0)
    w = configs.tiny()
    f = oracle.deconvolve(w.alpha).astype(np.float32)
    feat = None
    for n, reads in ((9, False), (6, True), (15, False), (15, False), (4, True), (17, True)):
        g = graphs.grid_graph(n, n + 1, 0.25, True)
        feat = api.sample(ctx, api.DeviceGraph(g), n, w.n_walks, w.p_halt, w.max_len, f, features=feat)
        if reads:
            for which, want in enumerate(oracle.sample(g.rowptr, g.col, g.w, n, w.n_walks, w.p_halt, w.max_len, f)[:3]):
                helpers.assert_csr_equal(feat.to_host(which), want, f"n={n} matrix {which}", val_rtol=0)
    feat.free()
    ctx.close()
