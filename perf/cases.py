"""Performance cases of the GRF-masked attention library: what a user of it runs, through its public entry points.

A case names a graph, the attention's shape and type, the walk parameters, and how the features come about:

  mode  "step"        the graph is new in every pass (particle clouds, dynamic graphs): walks are sampled in it
        "frozen"      walks were precomputed, the pass is the attention alone (image grids)
        "remodulated" the walks are kept, every pass gives them new modulation coefficients (training of f)
        "sample"      the pass precomputes the features themselves
  route "linear"      masked_linear_attn: linear attention under the mask estimate (the library's main call)
        "mask"        the mask materialised, then masked_attn_mhat
        "asym"        asymmetric features: linear or softmax similarity over Phi alone
        "host"        grf_step_host: the whole path from and to host buffers

Graphs: "grid" (image patches, 8 neighbours), "lattice" (4 neighbours), "cloud" (k nearest neighbours of points drawn
from a Gaussian mixture, numbered along a space-filling curve), "regular" (8-regular expander: no two neighbouring
nodes share anything).  phi(Q), phi(K) = ReLU of normals, V normal; the mask coefficients alpha_k = 2^-k give positive
modulation coefficients, so denominators do not cancel and outputs of different summation orders can be compared."""
import math

import numpy as np
import torch

from paper_2410_03462_b200 import api, binding as B

DTYPES = {"fp32": torch.float32, "bf16": torch.bfloat16}


def _case(name, graph, N, G, m, d, dtype, walks, p_halt, length, mode, route, degree=8, softmax=False):
    c = {"graph": graph, "N": N, "degree": degree, "G": G, "m": m, "d": d, "dtype": dtype, "walks": walks,
         "p_halt": p_halt, "length": length, "mode": mode, "route": route, "softmax": softmax}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one 8x8 lattice, one head; launches and host latency are all of it
        _case("tiny_step", "lattice", 64, 1, 16, 16, "fp32", 4, 0.5, 8, "step", "linear", degree=4),
        # one layer of an image transformer: 14x14 patches, 64 images x 12 heads, walks frozen; by the main call ...
        _case("vit_frozen_linear", "grid", 196, 768, 64, 64, "bf16", 16, 0.1, 10, "frozen", "linear"),
        # ... and by a program that materialised the mask once
        _case("vit_frozen_mask", "grid", 196, 768, 64, 64, "bf16", 16, 0.1, 10, "frozen", "mask"),
        # a moderate particle cloud whose graph changes every step
        _case("cloud4096_step", "cloud", 4096, 8, 32, 64, "bf16", 32, 0.1, 12, "step", "linear"),
        # the point-cloud transformer's size, the library's headline: sample, then attend over 8 heads
        _case("cloud32768_step", "cloud", 32768, 8, 32, 64, "bf16", 32, 0.1, 12, "step", "linear", degree=10),
        # the same step by a program that materialises the mask itself
        _case("cloud32768_step_mask", "cloud", 32768, 8, 32, 64, "bf16", 32, 0.1, 12, "step", "mask", degree=10),
        # training of the modulation coefficients on kept walks
        _case("cloud32768_remodulated", "cloud", 32768, 8, 32, 64, "bf16", 32, 0.1, 12, "remodulated", "mask", degree=10),
        # a caller that keeps nothing on the GPU: graph, Q, K, V up, outputs down, in pinned host memory
        _case("cloud32768_host", "cloud", 32768, 8, 32, 64, "bf16", 32, 0.1, 12, "step", "host", degree=10),
        # asymmetric features with the softmax similarity on the same clouds
        _case("cloud32768_asym_softmax", "cloud", 32768, 8, 32, 64, "bf16", 32, 0.1, 12, "step", "asym", degree=10,
              softmax=True),
        # full precision, an odd number of nodes and of heads
        _case("cloud5003_fp32_step", "cloud", 5003, 3, 32, 64, "fp32", 32, 0.1, 12, "step", "linear"),
        # precomputing the features that a model then freezes: walks, merging, CSR, regrouping, and reading them out
        _case("cloud20011_sample", "cloud", 20011, 1, 32, 64, "fp32", 32, 0.1, 12, "sample", "linear"),
        # the largest: a quarter of a million nodes of an expander, which no numbering makes local
        _case("regular262144_step", "regular", 262144, 4, 32, 64, "bf16", 16, 0.15, 10, "step", "linear"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["small", "grid", "grid", "cloud", "cloud", "cloud", "host", "asym", "fp32", "sample", "regular"])
    m = rng.choice([16, 32, 64])
    d = rng.choice([32, 64, 64])
    if kind == "small":
        side = rng.randint(6, 20)
        return _case(None, "lattice", side * side, rng.randint(1, 4), m, d, rng.choice(["fp32", "bf16"]),
                     rng.randint(4, 16), 0.5, 8, "step", "linear", degree=4)
    if kind == "grid":
        side = rng.randint(10, 20)
        route = rng.choice(["linear", "mask"])
        return _case(None, "grid", side * side, _log_int(rng, 48, 768), m, 64 if route == "mask" else d, "bf16",
                     rng.randint(12, 24), 0.1, rng.randint(8, 10), "frozen", route)
    if kind == "regular":
        return _case(None, "regular", _log_int(rng, 1024, 262144), rng.randint(2, 4), min(m, 32), d, "bf16",
                     rng.randint(12, 16), 0.15, rng.randint(8, 10), "step", "linear")
    N, G = _log_int(rng, 2048, 32768), rng.randint(4, 8)
    walks, length, degree = rng.randint(24, 32), rng.randint(10, 12), rng.randint(8, 10)
    if kind == "cloud":
        mode, route = rng.choice([("step", "linear"), ("step", "linear"), ("frozen", "linear"), ("step", "mask"),
                                  ("remodulated", "mask")])
        return _case(None, "cloud", N, G, m, 64 if route == "mask" else d, "bf16", walks, 0.1, length, mode, route, degree)
    if kind == "host":
        return _case(None, "cloud", N, G, m, d, "bf16", walks, 0.1, length, "step", "host", degree)
    if kind == "asym":
        return _case(None, "cloud", N, G, m, d, rng.choice(["bf16", "bf16", "fp32"]), walks, 0.1, length,
                     rng.choice(["step", "frozen"]), "asym", degree, softmax=rng.choice([True, False]))
    if kind == "fp32":
        return _case(None, "cloud", _log_int(rng, 1024, 8192), rng.randint(1, 4), m, d, "fp32", walks, 0.1, length, "step",
                     "linear", degree)
    return _case(None, "cloud", N, 1, 32, 64, "fp32", walks, 0.1, length, "sample", "linear", degree)


# ---------------------------------------------------------------------------------------------------
# Inputs

class _Graph:
    """CSR of a symmetric W, on the GPU."""

    def __init__(self, N, src, dst, w):
        order = torch.argsort(src * N + dst)
        self.N = N
        self.col = dst[order].to(torch.int32)
        self.w = w[order].to(torch.float32)
        self.rowptr = torch.zeros(N + 1, dtype=torch.int32, device=src.device)
        self.rowptr[1:] = torch.cumsum(torch.bincount(src, minlength=N), 0).to(torch.int32)


def _symmetric(N, code):
    """Both directions of the undirected edges `code` = low * N + high."""
    a, b = code // N, code % N
    return torch.cat([a, b]), torch.cat([b, a])


def _grid(N, diagonals, gen):
    side = math.isqrt(N)
    v = torch.arange(N, device="cuda")
    x, y = v // side, v % side
    src, dst = [], []
    for dx in (-1, 0, 1):
        for dy in (-1, 0, 1):
            if (dx, dy) == (0, 0) or (not diagonals and dx and dy):
                continue
            ok = (x + dx >= 0) & (x + dx < side) & (y + dy >= 0) & (y + dy < side)
            src.append(v[ok])
            dst.append((v + dx * side + dy)[ok])
    src, dst = torch.cat(src), torch.cat(dst)
    # similarities of neighbouring patches: a symmetric weight a little below 1 / (number of neighbours)
    noise = torch.rand(N, generator=gen, device="cuda")
    w = (0.9 + 0.1 * noise[src] * noise[dst]) / (8.0 if diagonals else 4.0)
    return _Graph(N, src, dst, w)


def _cloud(N, k, gen):
    """Points of a 16-component Gaussian mixture in Z order; an edge where either end lists the other among its k nearest."""
    centres = torch.rand(16, 3, generator=gen, device="cuda")
    sigma = 0.03 + 0.07 * torch.rand(16, generator=gen, device="cuda")
    which = torch.randint(16, (N,), generator=gen, device="cuda")
    p = centres[which] + torch.randn(N, 3, generator=gen, device="cuda") * sigma[which, None]
    lo, hi = p.min(0).values, p.max(0).values
    q = ((p - lo) / (hi - lo) * 1023).to(torch.int64)
    code = torch.zeros(N, dtype=torch.int64, device="cuda")
    for b in range(10):
        for a in range(3):
            code |= ((q[:, a] >> b) & 1) << (3 * b + a)
    p = p[torch.argsort(code, stable=True)]
    src, dst, dist = [], [], []
    for x in range(0, N, 4096):
        dd = torch.cdist(p[x:x + 4096], p, compute_mode="donot_use_mm_for_euclid_dist")
        row = torch.arange(dd.shape[0], device="cuda")
        dd[row, x + row] = math.inf
        for _ in range(k):
            v, i = dd.min(1)
            dd[row, i] = math.inf
            src.append(x + row)
            dst.append(i)
            dist.append(v)
    src, dst, dist = torch.cat(src), torch.cat(dst), torch.cat(dist)
    edges = torch.unique(torch.minimum(src, dst) * N + torch.maximum(src, dst))
    a, b = _symmetric(N, edges)
    w = torch.exp(-((p[a] - p[b]) ** 2).sum(1) / dist.median() ** 2)
    w = w * (0.9 / torch.zeros(N, device="cuda", dtype=torch.float64).scatter_add_(0, a, w.double()).max()).float()
    return _Graph(N, a, b, w)


def _regular(N, gen):
    """Union of four random Hamiltonian cycles."""
    codes = []
    for _ in range(4):
        perm = torch.randperm(N, generator=gen, device="cuda")
        nxt = torch.roll(perm, -1)
        codes.append(torch.minimum(perm, nxt) * N + torch.maximum(perm, nxt))
    a, b = _symmetric(N, torch.unique(torch.cat(codes)))
    return _Graph(N, a, b, torch.full(a.shape, 0.125, device="cuda"))


_contexts = {}


def _context(name):
    """A program makes its context once."""
    if name not in _contexts:
        _contexts[name] = api.Context(0)
    return _contexts[name]


class _State:
    feat = None

    def __del__(self):
        if self.feat is not None and self.feat.handle:
            torch.cuda.synchronize()
            self.feat.free()


def prepare(case, seed):
    s = _State()
    s.case, s.seed = case, seed
    gen = torch.Generator(device="cuda").manual_seed(seed)
    N, G, m, d = case["N"], case["G"], case["m"], case["d"]
    L, route, mode = case["length"], case["route"], case["mode"]
    if case["graph"] == "cloud":
        s.graph = _cloud(N, case["degree"], gen)
    elif case["graph"] == "regular":
        s.graph = _regular(N, gen)
    else:
        s.graph = _grid(N, case["graph"] == "grid", gen)

    alpha = 0.5 ** np.arange(L + 1, dtype=np.float64)
    s.f = B.grf_deconvolve(alpha).astype(np.float32)
    s.f_psi = None
    if route == "asym":
        s.f = alpha.astype(np.float32)
        s.f_psi = np.zeros(L + 1, np.float32)
        s.f_psi[0] = 1.0

    dt = DTYPES[case["dtype"]]
    if mode != "sample":
        s.q = torch.relu(torch.randn(G, N, m, generator=gen, device="cuda")).to(dt)
        s.k = torch.relu(torch.randn(G, N, m, generator=gen, device="cuda")).to(dt)
        s.v = torch.randn(G, N, d, generator=gen, device="cuda").to(dt)
        if case["softmax"]:
            s.q, s.k = s.q * 0.25, s.k * 0.25

    if route == "host":
        s.ctx = _context("host")
        pin = lambda t: t.cpu().pin_memory()  # noqa: E731
        s.host_graph = [pin(t) for t in (s.graph.rowptr, s.graph.col, s.graph.w)]
        s.graph = None
        s.q, s.k, s.v = pin(s.q), pin(s.k), pin(s.v)
        s.out = torch.empty(G, N, d, dtype=dt, pin_memory=True)
        return s

    s.ctx = _context("device")
    s.feat = api.Features(s.ctx, None)
    if route == "linear" and mode != "sample":
        nbytes = B.grf_attn_workspace_bytes(G, N, m, d, B.dtype_code(s.v))
        s.workspace = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    if mode == "sample":
        # Phi, Psi and Psi^T are read into arrays of the largest size they can have (zeros behind the last entry)
        room = N * min(N, case["walks"] * (L + 1))
        s.matrices = [(torch.zeros(N + 1, dtype=torch.int32, device="cuda"),
                       torch.zeros(room, dtype=torch.int32, device="cuda"),
                       torch.zeros(room, dtype=torch.float32, device="cuda")) for _ in range(3)]
    if mode in ("frozen", "remodulated"):
        B.grf_ctx_keep_walks(s.ctx.handle, mode == "remodulated")
        _sample(s)
        B.grf_ctx_keep_walks(s.ctx.handle, False)
        if route == "mask":
            B.grf_features_materialise(s.ctx.handle, s.feat.handle)
    if mode == "remodulated":
        rng = np.random.default_rng(seed)
        s.f = (s.f * (1.0 + 0.2 * rng.random(L + 1))).astype(np.float32)
    return s


# ---------------------------------------------------------------------------------------------------
# One pass

def _sample(s):
    c = s.case
    s.feat.handle = B.grf_sample(s.ctx.handle, c["N"], s.graph.rowptr, s.graph.col, s.graph.w, s.seed, c["walks"],
                                 c["p_halt"], c["length"], s.f, s.f_psi, s.feat.handle)


def _read_features(s):
    for which, (rowptr, col, val) in enumerate(s.matrices):
        B.grf_features_copy(s.ctx.handle, s.feat.handle, which, rowptr, col, val)
    return s.matrices


def run(s):
    c = s.case
    if c["route"] == "host":
        B.grf_step_host(s.ctx.handle, c["N"], *s.host_graph, s.seed, c["walks"], c["p_halt"], c["length"], s.f, s.f_psi,
                        c["G"], c["m"], c["d"], B.dtype_code(s.v), s.q, s.k, s.v, s.out)
        return s.out
    if c["mode"] == "remodulated":
        B.grf_remodulate(s.ctx.handle, s.feat.handle, c["length"], s.f, s.f_psi)
    elif c["mode"] != "frozen":
        _sample(s)
    if c["mode"] == "sample":
        return _read_features(s)
    if c["route"] == "linear":
        return api.masked_linear_attn(s.ctx, s.feat, s.q, s.k, s.v, workspace=s.workspace)
    if c["route"] == "asym":
        return api.masked_attn_asym(s.ctx, s.feat, s.q, s.k, s.v, softmax=c["softmax"])
    if c["mode"] != "frozen":
        B.grf_features_materialise(s.ctx.handle, s.feat.handle)
    return api.masked_attn_mhat(s.ctx, s.feat, s.q, s.k, s.v)


# ---------------------------------------------------------------------------------------------------
# What a pass cannot do without

def work(case):
    """Bytes: every input read once, every output written once.  Flops: the attention's, by the cheaper association of
    Phi Psi^T, from the expected sizes of the features (distinct nodes per row and keys per row of the mask, as fractions
    of the expected deposits and pairs on each kind of graph)."""
    N, G, m, d, keep = case["N"], case["G"], case["m"], case["d"], 1.0 - case["p_halt"]
    size = 4 if case["dtype"] == "fp32" else 2
    deposits = case["walks"] * (1.0 - keep ** (case["length"] + 1)) / case["p_halt"]
    distinct, reach = {"cloud": (0.4, 0.11), "regular": (0.75, 0.9)}.get(case["graph"], (0.5, 0.05))
    per_row = min(N, distinct * deposits)
    keys = min(N, reach * per_row * per_row)
    graph_bytes = 4 * (N + 1) + 8 * N * (case["degree"] * (1.4 if case["graph"] == "cloud" else 1.0))
    feature_bytes = 4 * (N + 1) + 8 * N * per_row
    if case["mode"] == "sample":
        # the deposits' products, the merging sums, and the three matrices
        return {"bytes": graph_bytes + 3 * feature_bytes, "flops": 2 * N * deposits * 5}
    qkv = G * N * (2 * m + 2 * d) * size
    if case["route"] == "asym":
        read = graph_bytes if case["mode"] == "step" else feature_bytes
        return {"bytes": qkv + read, "flops": 2.0 * G * N * per_row * (m + d)}
    read = {"step": graph_bytes, "frozen": 2 * feature_bytes, "remodulated": 2 * 5 * N * deposits}[case["mode"]]
    by_states = 4.0 * G * N * per_row * m * (d + 1)
    by_mask = 2.0 * G * N * keys * (m + d) + 2.0 * N * per_row * per_row
    return {"bytes": qkv + read, "flops": min(by_states, by_mask)}


def tolerance(case):
    if case["mode"] == "sample":
        return "exact"
    if case["dtype"] == "fp32":
        return {"rel": 1e-5, "max": 1e-4}
    return {"rel": 1e-2, "max": 0.1}
