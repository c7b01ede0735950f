"""Key lists, positions and values of the materialised mask at the edges of their kernels: blocks of one row, nodes with
0, 31 ... 200 keys, key lists around whole tiles, and lists longer than a warp's accumulators."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def _csr(lengths, cols, rng):
    c = [np.sort(rng.choice(cols, size=n, replace=False)) for n in lengths]
    rp = np.concatenate([[0], np.cumsum([len(x) for x in c])]).astype(np.int32)
    col = np.concatenate(c).astype(np.int32)
    return oracle.CSR(rp, col, rng.standard_normal(col.size).astype(np.float32), None, (len(lengths), cols))


def _check(N, R, Phi, Psi, rows):
    from paper_2410_03462_b200 import api, binding as B
    ctx = api.Context(0)
    feat = api.features_from_csr(ctx, N, R, (Phi.rowptr, Phi.col, Phi.val), (Psi.rowptr, Psi.col, Psi.val))
    for _ in range(2):                    # the second build finds room in the arrays of the first
        B.grf_features_materialise(ctx.handle, feat.handle)
        out = torch.empty((len(rows), N), dtype=torch.float32, device="cuda")
        B.grf_mask_rows(ctx.handle, feat.handle, len(rows), torch.tensor(rows, dtype=torch.int32, device="cuda"), out)
        want = oracle.mask_rows(Phi, Psi, rows)
        scale = oracle.mask_rows(*(oracle.CSR(m.rowptr, m.col, np.abs(m.val), None, m.shape) for m in (Phi, Psi)), rows)
        got = out.cpu().numpy().astype(np.float64)
        assert (np.abs(got - want) <= 2.0 ** -8 * np.abs(want) + 1e-5 * scale).all()
        assert ((got != 0) <= (scale != 0)).all()
    feat.free()
    ctx.close()


@pytest.mark.parametrize("N", [1, 63, 64, 65, 127, 128, 129, 300])
def test_small_blocks(N):
    rng = np.random.default_rng(N)
    R = 41
    keys_of_node = [min(N, n) for n in (0, 1, 31, 32, 33, 63, 64, 65, 95, 96, 97, 127, 128, 129, 160, 200)] + [min(N, 2)] * (R - 16)
    PsiT = _csr(keys_of_node, N, rng)
    Psi = oracle.transpose(oracle.CSR(PsiT.rowptr, PsiT.col, PsiT.val, None, (R, N)))
    Psi = oracle.CSR(Psi.rowptr, Psi.col, Psi.val, None, (N, R))
    Phi = _csr([(3, 0, 1, 33, 41, 7)[i % 6] for i in range(N)], R, rng)
    _check(N, R, Phi, Psi, list(range(0, N, max(1, N // 40))))


@pytest.mark.parametrize("N", [6784, 6785, 14000])
def test_lists_around_accumulator_segments(N):
    rng = np.random.default_rng(N)
    R = 50
    Psi = _csr([2] * N, R - 1, rng)
    # the last node is reached by every key: lists of N keys
    rp = (Psi.rowptr + np.arange(N + 1)).astype(np.int32)
    col = np.insert(Psi.col, Psi.rowptr[1:], R - 1).astype(np.int32)
    Psi = oracle.CSR(rp, col, rng.standard_normal(col.size).astype(np.float32), None, (N, R))
    Phi = _csr([4] * N, R, rng)
    _check(N, R, Phi, Psi, [0, 1, 127, 128, N // 2, N - 1])


@pytest.mark.parametrize("blocks", [2, 36, 37, 38, 74, 75, 148, 149])
def test_several_ctas_per_block(blocks):
    """A block is built by a cluster of 8, 4 or 2 CTAs, by the number of blocks: nodes with one key, a warp's and
    several warps' shares of nodes, and a last block of one row."""
    N = 128 * (blocks - 1) + 1
    rng = np.random.default_rng(blocks)
    R = N // 4 + 700
    Psi = _csr([(1, 3, 0, 5)[i % 4] for i in range(N)], R, rng)
    Phi = _csr([(3, 0, 9, 1, 40)[i % 5] for i in range(N)], R, rng)
    rows = sorted({0, 1, 2, 127, 128 % N, N // 2, N // 2 + 1, N - 129 if N > 129 else 0, N - 2, N - 1})
    _check(N, R, Phi, Psi, rows)
