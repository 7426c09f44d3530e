"""The iterated propagation as one call: ragged and misaligned rows, one and several partitions, long rows, arrays below and
above the size at which the span kernels take over, an odd and an even number of steps; against float64 sums."""
import numpy as np
import pytest
import torch

from paper_2111_06483_b200 import api

from helpers import allclose_report

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("n,F,dtype,k,iters,scaled,shift", [
    (1, 1, "f32", 1, 1, True, 0), (900, 3, "f32", 1, 3, True, 0), (900, 47, "f32", 4, 2, False, 0), (900, 300, "f32", 1, 1, True, 0),
    (900, 16, "f32", 1, 2, True, 1), (900, 16, "f32", 3, 3, True, 1), (900, 16, "f32", 3, 1, False, 0), (900, 16, "f32", 1, 1, True, 0),
    (900, 16, "f32", 2, 4, False, 0), (900, 16, "f32", 2, 3, True, 0), (900, 9, "bf16", 2, 2, True, 0), (70_000, 47, "f32", 1, 3, True, 0),
    (70_000, 48, "f32", 3, 2, True, 0), (70_000, 100, "bf16", 1, 2, False, 0)])
def test_propagation_in_one_call(n, F, dtype, k, iters, scaled, shift):
    tdt = torch.float32 if dtype == "f32" else torch.bfloat16
    gen = torch.Generator().manual_seed(n + F)
    e = n * 6
    src, dst = (torch.randint(0, max(n - 1, 1), (e,), generator=gen, dtype=torch.int32) for _ in range(2))
    dst[: e // 4] = 0                                     # a long row; the last node has no edge
    g = api.Graph.from_coo(n, src.to(DEV), dst.to(DEV), k=k, build_parts=k > 1, threshold=64)
    x0 = torch.randn((n, F), generator=gen).to(tdt)
    s = torch.rand(n, generator=gen) + 0.5 if scaled else None
    d = 1.0 / torch.bincount(dst.long(), minlength=n).clamp(min=1).float()
    buf = torch.empty(n * F + shift, dtype=tdt, device=DEV)
    x = buf[shift:].view(n, F)
    x.copy_(x0)
    got = api.propagate(g, x, 0.7, iters, s.to(DEV) if scaled else None, d.to(DEV))
    adj = torch.sparse_coo_tensor(torch.stack([dst.long(), src.long()]), torch.ones(e, dtype=torch.float64), (n, n)).to_sparse_csr()
    want, x64 = x0.double(), x0.double()
    for _ in range(iters):
        y = want * s.double()[:, None] if scaled else want
        want = 0.3 * x64 + 0.7 * d.double()[:, None] * (adj @ y)
    tol = dict(rtol=1e-5, atol=1e-5) if dtype == "f32" else dict(rtol=2e-2, atol=2e-2)
    allclose_report(got.double().cpu().numpy(), want.numpy(), what="propagation", **tol)
    assert np.isfinite(got.float().cpu().numpy()).all()


@pytest.mark.parametrize("F,shift_in,shift_out,arrays", [(16, 0, 0, 1), (16, 1, 0, 2), (16, 0, 1, 2), (16, 1, 1, 3), (15, 0, 0, 3)])
@pytest.mark.parametrize("iters,scaled", [(1, True), (2, True), (3, False)])
def test_workspace_for_the_pointers_given(F, shift_in, shift_out, arrays, iters, scaled):
    """The workspace asked for holds no array that the call does not use, and the call stays within it."""
    from paper_2111_06483_b200 import binding as B
    n = 700
    gen = torch.Generator().manual_seed(F)
    src, dst = (torch.randint(0, n, (5 * n,), generator=gen, dtype=torch.int32).to(DEV) for _ in range(2))
    g = api.Graph.from_coo(n, src, dst)
    x, out = (torch.empty(n * F + s, device=DEV)[s:].view(n, F) for s in (shift_in, shift_out))
    x.copy_(torch.randn((n, F), generator=gen))
    s = torch.rand(n, device=DEV) if scaled else None
    nbytes = B.sar_propagate_workspace_bytes_at([g.whole], x, B.SAR_F32, out)
    assert nbytes == arrays * ((n * ((F + 3) // 4) * 16 + 255) // 256 * 256) + 256
    assert B.sar_propagate_workspace_bytes([g.whole], F, B.SAR_F32) >= nbytes
    ws = torch.full((nbytes + 4096,), 0xA5, dtype=torch.uint8, device=DEV)
    B.sar_propagate([g.whole], g.bounds, x, 0.7, iters, s, None, out, ws[:nbytes])
    assert torch.equal(out, api.propagate(g, x.clone(), 0.7, iters, s))
    assert bool((ws[nbytes:] == 0xA5).all())
    with pytest.raises(B.SarError):
        B.sar_propagate([g.whole], g.bounds, x, 0.7, iters, s, None, out, ws[:nbytes - 512])


def test_propagation_takes_one_array_beside_its_result():
    n, F = 200_000, 64
    src, dst = (torch.randint(0, n, (n,), device=DEV, dtype=torch.int32) for _ in range(2))
    g = api.Graph.from_coo(n, src, dst)
    x = torch.randn(n, F, device=DEV)
    api.propagate(g, x, 0.5, 2)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    torch.cuda.reset_peak_memory_stats()
    before = torch.cuda.memory_allocated()
    api.propagate(g, x, 0.5, 3)
    assert torch.cuda.max_memory_allocated() - before < 2.1 * x.nbytes


@pytest.mark.parametrize("n,F", [(1, 1), (37, 3), (1001, 1), (513, 2), (129, 5), (77, 7), (640, 8), (255, 47), (33, 301)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("shift", [0, 1])
def test_rows_of_a_ragged_or_misaligned_result(n, F, dtype, shift):
    """(1 - 0) x0 + 0 sum is x0 to the bit: every element of the result is written, at its place, and none beside it."""
    from paper_2111_06483_b200 import binding as B
    gen = torch.Generator().manual_seed(n)
    src, dst = (torch.randint(0, n, (3 * n,), generator=gen, dtype=torch.int32).to(DEV) for _ in range(2))
    g = api.Graph.from_coo(n, src, dst)
    x = torch.randn((n, F), generator=gen).to(dtype).to(DEV)
    buf = torch.full((shift + n * F + 16,), 7.0, dtype=dtype, device=DEV)
    out = buf[shift:shift + n * F].view(n, F)
    t = B.SAR_F32 if dtype == torch.float32 else B.SAR_BF16
    ws = torch.empty(B.sar_propagate_workspace_bytes([g.whole], F, t), dtype=torch.uint8, device=DEV)
    B.sar_propagate([g.whole], g.bounds, x, 0.0, 2, None, None, out, ws)
    assert torch.equal(out, x)
    assert bool((buf[:shift] == 7.0).all()) and bool((buf[shift + n * F:] == 7.0).all())
