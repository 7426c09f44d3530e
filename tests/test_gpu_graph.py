"""Graph preparation where the counting passes can go wrong: numbers of ids at one, two and three digits, edges at a block's
tile, partitions without sources, one long row; whole CSR, CSC, plans and partitions against numpy."""
import numpy as np
import pytest
import torch

from paper_2111_06483_b200 import api

pytestmark = pytest.mark.gpu
DEV = "cuda"


def csr(n_rows, row, col):
    order = np.lexsort((col, row))
    return np.searchsorted(row[order], np.arange(n_rows + 1)).astype(np.int64), col[order]


def plan(indptr, threshold):
    deg = np.diff(indptr)
    rows = np.nonzero(deg > threshold)[0]
    return rows, np.concatenate([[0], np.cumsum(-(-deg[rows] // threshold))])


def check(part, indptr, indices, t_indptr, t_indices, threshold, t_threshold):
    for got, want in ((part.indptr, indptr), (part.indices, indices), (part.t_indptr, t_indptr), (part.t_indices, t_indices)):
        np.testing.assert_array_equal(got.cpu().numpy(), want)
    for s, ip, thr in ((part.split, indptr, threshold), (part.t_split, t_indptr, t_threshold)):
        rows, seg = plan(ip, thr)
        assert (s.threshold, s.n_long, s.n_seg) == (thr, len(rows), seg[-1])
        np.testing.assert_array_equal(s.long_row.cpu().numpy(), rows)
        np.testing.assert_array_equal(s.long_seg.cpu().numpy(), seg)


@pytest.mark.parametrize("n,nnz,k,hub", [
    (1, 3, 1, 0), (7, 0, 9, 0), (2048, 8191, 4, 0), (2049, 8192, 3, 5000), (5000, 8193, 5, 1), (40_000, 700_000, 7, 300_000),
    (1 << 22, 300_001, 2, 0), ((1 << 22) + 1, 1_000_000, 64, 100_000)])
def test_graph_preparation(n, nnz, k, hub):
    rng = np.random.default_rng(n + nnz)
    src, dst = rng.integers(0, n, nnz, dtype=np.int32), rng.integers(0, n, nnz, dtype=np.int32)
    dst[:hub] = n - 1                       # a row of many edges, duplicates among them
    src[hub // 2:hub] = n // 3
    g = api.Graph.from_coo(n, torch.from_numpy(src).to(DEV), torch.from_numpy(dst).to(DEV), k=k, threshold=100,
                           build_parts=True, t_threshold=33)
    check(g.whole, *csr(n, dst, src), *csr(n, src, dst), 100, 33)
    for q, part in enumerate(g.parts):
        s0, s1 = g.bounds[q], g.bounds[q + 1]
        keep = (src >= s0) & (src < s1)
        check(part, *csr(n, dst[keep], src[keep] - s0), *csr(s1 - s0, src[keep] - s0, dst[keep]), 100, 100)
    whole = g.whole
    t = api.graph_from_csr(n, whole.indptr, whole.indices).whole     # the transpose alone
    assert torch.equal(t.t_indptr, whole.t_indptr) and torch.equal(t.t_indices, whole.t_indices)
