"""The kernels behind the shapes that the lean kernels do not cover, at the sizes where they can go wrong: heads that are no
power of two or no whole number of 16-byte words, rows wider than one lane group, arrays on either side of the size where
the dispatch changes from the row kernels to the span kernels, and calls that get no room for padded copies."""
import numpy as np
import pytest
import torch

import workloads
from helpers import allclose_report
from test_gpu_parity import DEV, Problem, _full_check, check_grad, check_out, hub_graph

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2111_06483_b200 import api, binding as B


class Launches:
    """The names of the gather kernels' launches inside the block."""

    def __enter__(self):
        self.names = []
        B.sar_set_launch_hook(lambda name, phase: self.names.append(name) if phase == 0 else None)
        return self

    def __exit__(self, *exc):
        B.sar_set_launch_hook(None)
        return False

    def only(self, suffix, passes=("gat_fwd", "gat_bwd_dst", "gat_bwd_src")):
        """Every pass over edges was the kernel of that suffix (its merges aside)."""
        seen = [x for x in self.names if x.startswith(tuple(passes)) and not x.endswith(("_merge", "_finalize"))]
        return bool(seen) and all(x.endswith(suffix) for x in seen)


@pytest.mark.parametrize("H,F,dtype", [(1, 47, "bf16"), (3, 33, "f32"), (6, 24, "bf16"), (2, 64, "bf16"), (7, 9, "f32"), (1, 300, "f32"),
                                       (2, 260, "f32"), (1, 520, "bf16"), (12, 8, "f32"), (1, 1030, "bf16")])
@pytest.mark.parametrize("threshold", [0, 24])
def test_attention_on_general_shapes(H, F, dtype, threshold):
    n, src, dst = hub_graph(n=2000, e=24000, d_max=400.0, seed=19)
    p = Problem(n, src, dst, H, F, 70 + H + F, dtype=dtype, k=3, threshold=threshold, build_parts=True)
    # the dot products that cancel in del and der grow with F at worst
    _full_check(p, dtype=dtype, modes=("fused", "stateful"), grad_floor=max(1.0, F / 64))


@pytest.mark.parametrize("H,F,dtype,n", [(2, 64, "bf16", 540_000), (1, 60, "f32", 600_000)])
def test_attention_on_arrays_larger_than_the_l2(H, F, dtype, n):
    spec = workloads.ChungLuSpec(n=n, e=1_500_000, gamma=2.1, d_max=3000.0, seed=5)
    src, dst = workloads.chung_lu_edges(spec)
    p = Problem(n, src, dst, H, F, 7, dtype=dtype, k=2, build_parts=True)
    # a million sums of up to 3000 terms that cancel
    _full_check(p, dtype=dtype, modes=("fused", "stateful"), grad_floor=10.0)


@pytest.mark.parametrize("H,F,dtype,n,deg,d_max", [(4, 8, "f32", 61_000, 3, 200.0), (2, 64, "bf16", 61_000, 2, 400.0), (3, 32, "bf16", 61_000, 4, 900.0),
                                                   (6, 48, "bf16", 21_000, 9, 300.0), (12, 16, "f32", 10_100, 2, 500.0),
                                                   (8, 24, "bf16", 700, 11, 200.0), (4, 48, "f32", 900, 20, 300.0), (3, 64, "f32", 900, 8, 300.0),
                                                   (5, 24, "f32", 20_000, 16, 300.0), (4, 24, "bf16", 20_000, 15, 300.0), (6, 128, "bf16", 900, 6, 100.0),
                                                   (3, 128, "f32", 1_500, 6, 100.0)])
def test_attention_on_short_rows(H, F, dtype, n, deg, d_max):
    """Few edges per row: shapes on either side of the lines between the row, the span and the short-row kernels on small arrays, whole and
    step by step, with long rows among them."""
    n, src, dst = hub_graph(n=n, e=deg * n, d_max=d_max, seed=H + F)
    p = Problem(n, src, dst, H, F, 31, dtype=dtype, k=2, threshold=100, build_parts=True)
    _full_check(p, dtype=dtype, modes=("fused", "stateful"), grad_floor=10.0)


@pytest.mark.parametrize("H,F,dtype", [(1, 5, "f32"), (1, 32, "bf16"), (2, 12, "bf16"), (4, 8, "f32"), (3, 16, "bf16"), (1, 47, "bf16"), (8, 8, "bf16"),
                                       (2, 32, "f32"), (4, 24, "bf16"), (7, 8, "f32"), (8, 24, "bf16"), (3, 24, "f32"),
                                       (2, 32, "bf16"), (2, 16, "f32"), (4, 8, "bf16"), (3, 4, "f32"), (2, 64, "bf16"), (3, 32, "f32")])
@pytest.mark.parametrize("scale", [1.0, 60.0])
def test_attention_of_a_row_per_lane_group(H, F, dtype, scale):
    """Enough rows with few enough edges for the kernel for short rows: rows of 0, 1, 3 to 5, 23 to 25 and 95 to 97 edges (the ends of its
    steps of four, and of what one group keeps to itself), segments of 100 and of 1, and scores that lead a row's first by more than 60."""
    n, gen = 16_100, torch.Generator().manual_seed(H * F)
    # tiles of 16 vectors and two heads, or 32 and four: three edges per row are too many, and the forward pass is another kernel's
    backward_only = (H, F, dtype) in ((2, 32, "f32"), (2, 64, "bf16"), (3, 24, "f32"), (3, 32, "f32"))
    many = 1 if backward_only or (H, F) == (4, 24) else 3
    src, dst = [torch.randint(0, n, (many * n,), generator=gen)], [torch.randint(500, n, (many * n,), generator=gen)]
    for row, deg in enumerate([1, 3, 4, 5, 23, 24, 25, 95, 96, 97, 100, 101, 350]):
        src.append(torch.randint(0, n, (2 * deg,), generator=gen))
        dst.append(torch.tensor([7 * row, 7 * row + 3]).repeat_interleave(deg))
    src, dst = torch.cat(src).int(), torch.cat(dst).int()
    both = torch.cat([src, dst]), torch.cat([dst, src])   # the same lengths among the columns, which the source-major pass walks
    p = Problem(n, both[0], both[1], H, F, 3, dtype=dtype, k=2, threshold=100, build_parts=True, scale=scale)
    if scale == 1.0:
        with Launches() as ran:
            _full_check(p, dtype=dtype, modes=("fused", "stateful"), grad_floor=10.0)
        # (a step has half of the sources, for some tiles too few rows for the source-major pass)
        assert ran.only("_short", ("gat_bwd_dst",) if backward_only else ("gat_fwd", "gat_bwd_dst")) and "gat_bwd_src_short" in ran.names, set(ran.names)
        return
    # d = sum exp(e - m) with |e| up to 500: an ulp of e is 2^-15, and that is the relative error of its exponential
    d, f = p.dev, p.oracle_fwd()
    for mode in ("fused", "stateful"):
        out, m, dd = api.gat_forward(p.graph, d["feat"], d["el"], d["er"], 0.2, mode=mode)[:3]
        has = np.isfinite(f.m)
        assert np.array_equal(np.isfinite(m.cpu().numpy()), has)
        allclose_report(m.cpu().numpy()[has], f.m[has], 2.0 ** -23, 0.0, "m")
        allclose_report(dd.cpu().numpy(), f.d, 2.0 ** -14, 0.0, "d")
        # out is a mean of features of up to 5 with those weights: 2 x 2^-15 x 5, besides the rounding of a stored bf16
        bf16 = dtype == "bf16"
        allclose_report(out.float().cpu().numpy(), f.out, 2.0 ** -7 if bf16 else 1e-5, 2.0 ** -9 if bf16 else 10 * 2.0 ** -15, "out")


def _masked_problem(H, F, dtype, which, threshold, long_rows=()):
    """Rows whose sources' score terms are partly -inf, three random edges per row besides rows of 6 to 96 edges with sources of
    their own.  Every row keeps an edge from the last hundred sources, which are not masked."""
    n, gen = 16_100, torch.Generator().manual_seed(H * F)
    src, dst = [torch.randint(0, n, (2 * n,), generator=gen), n - 1 - torch.arange(n) % 100], [torch.randint(500, n, (2 * n,), generator=gen), torch.arange(n)]
    masked, at = torch.zeros(n, dtype=torch.bool), 1000
    groups = max(1, 32 // (4 if F * (2 if dtype == "bf16" else 4) * H <= 64 else 8))
    for i, deg in enumerate([6, 8, 9, 23, 24, 25, 32, 48, 95, 96, *long_rows]):
        src.append(torch.arange(at, at + deg))     # sources ascend within a row: position p of the row is source at + p
        dst.append(torch.full((deg,), 7 * i))
        pos = torch.arange(deg)
        masked[at:at + deg] = pos < 4 if which == "first" else (pos // 4) % groups == i % groups
        at += deg
    if which == "step":
        masked[:] = torch.arange(n) < n // 2
    elif which == "half":
        masked[:] = torch.rand(n, generator=gen) < 0.5
    masked[n - 100:] = False
    p = Problem(n, torch.cat(src).int(), torch.cat(dst).int(), H, F, 3, dtype=dtype, k=2, threshold=threshold, build_parts=True)
    p.host["er"][masked.numpy()] = -np.inf
    p.dev["er"][masked.to(DEV)] = -float("inf")
    return p


@pytest.mark.parametrize("H,F,dtype", [(1, 32, "bf16"), (1, 47, "bf16"), (1, 16, "f32"), (8, 8, "bf16"), (4, 8, "f32"), (8, 24, "bf16")])
@pytest.mark.parametrize("which", ["first", "group", "step", "half"])
def test_masked_sources_of_short_rows(H, F, dtype, which):
    """er = -inf for a row's first four edges, for all that one group of lanes has of a row the warp shares, for every edge of a
    partition step and for half of all sources: such an edge weighs nothing, and what came before the first other one is 0."""
    p = _masked_problem(H, F, dtype, which, 0)
    with Launches() as ran:
        _full_check(p, dtype=dtype, modes=("fused", "stateful"), grad_floor=10.0)
    assert ran.only("_short", ("gat_fwd",) if (H, F) == (8, 24) else ("gat_fwd", "gat_bwd_dst")), set(ran.names)


@pytest.mark.parametrize("H,F,dtype", [(1, 32, "bf16"), (1, 16, "f32"), (8, 8, "bf16"), (4, 8, "f32")])
@pytest.mark.parametrize("threshold,long_rows", [(100, (101, 350, 800)), (20, (21,) * 300)])
def test_masked_sources_of_long_rows(H, F, dtype, threshold, long_rows):
    """Rows in segments, all of whose edges in the first partition step are masked: their merge (of a block, and of a warp where there
    are many such rows) leaves a state that the second step can go on from."""
    p = _masked_problem(H, F, dtype, "step", threshold, long_rows)
    with Launches() as ran:
        _full_check(p, dtype=dtype, modes=("fused", "stateful"), grad_floor=10.0)
    assert ran.only("_short", ("gat_fwd",)) and "gat_fwd_merge" in ran.names, set(ran.names)
    part = p.graph.parts[0]
    assert part.split.n_long > (296 if threshold == 20 else 0)


@pytest.mark.parametrize("H,F,dtype", [(1, 32, "bf16"), (1, 16, "f32"), (8, 8, "bf16"), (4, 8, "f32")])
@pytest.mark.parametrize("lead,power", [(50.0, 60), (20.0, 100)])
def test_large_features_of_short_rows(H, F, dtype, lead, power):
    """Features of 2^60 (1e18) and 2^100 (1e30) whose scores lead the row's others by 50 and 20: no weight exceeds 1, so that no sum exceeds
    the features' by more than the number of edges.  Features and output gradients are scaled by powers of two, which is exact."""
    p = _masked_problem(H, F, dtype, "none", 0)
    pick = np.random.default_rng(5).random(p.host["er"].shape) < 0.5
    p.host["el"][:] = 0.0
    p.host["er"][:] = np.where(pick, 1.0, 1.0 + lead)
    f = p.oracle_fwd()
    b = p.oracle_bwd(f)
    d = {k: torch.as_tensor(v, device=DEV) for k, v in p.host.items()}
    feat, gout = p.dev["feat"] * 2.0 ** power, p.dev["gout"] * 2.0 ** -power
    for mode in ("fused", "stateful"):
        with Launches() as ran:
            out, m, dd, *acc = api.gat_forward(p.graph, feat, d["el"], d["er"], 0.2, mode=mode, keep_numerator=mode == "stateful")
        assert ran.only("_short"), set(ran.names)
        check_out(out.float() * 2.0 ** -power, f.out, dtype, "out")
        allclose_report(dd.cpu().numpy(), f.d, 1e-5, 1e-6, "d")
        dfeat, del_, der = api.gat_backward(p.graph, feat, d["el"], d["er"], m, dd, gout, 0.2, out=out, mode=mode, acc=acc[0] if acc else None)
        check_grad(dfeat.float() * 2.0 ** power, b.dfeat, dtype, "dfeat", stored=True)
        check_grad(del_, b.del_, dtype, "del", 10.0)
        check_grad(der, b.der, dtype, "der", 10.0)


@pytest.mark.parametrize("H,F,dtype,n,deg,d_max,passes", [(2, 64, "bf16", 61_000, 2, 400.0, ("gat_fwd",)), (6, 48, "bf16", 21_000, 9, 300.0, ("gat_fwd", "gat_bwd_dst", "gat_bwd_src")),
                                                          (12, 16, "f32", 900, 8, 100.0, ("gat_bwd_dst", "gat_bwd_src")), (8, 24, "bf16", 700, 11, 200.0, ("gat_bwd_dst", "gat_bwd_src")),
                                                          (5, 24, "f32", 20_000, 16, 300.0, ("gat_bwd_dst", "gat_bwd_src")), (16, 8, "f32", 1_100, 9, 100.0, ("gat_bwd_dst", "gat_bwd_src")),
                                                          (3, 32, "f32", 40_000, 13, 300.0, ("gat_bwd_dst", "gat_bwd_src"))])
def test_span_kernels_on_small_arrays(H, F, dtype, n, deg, d_max, passes):
    n, src, dst = hub_graph(n=n, e=deg * n, d_max=d_max, seed=H + F)
    p = Problem(n, src, dst, H, F, 31, dtype=dtype, k=2, threshold=100, build_parts=True)
    with Launches() as ran:
        _full_check(p, dtype=dtype, modes=("fused",), grad_floor=10.0)
    assert ran.only("_span", passes), set(ran.names)
    _full_check(p, dtype=dtype, modes=("stateful",), grad_floor=10.0)


def _infinite_last_sources(n):
    """Rows of 1 to 50 edges whose last edge (the highest source) is one of 20 nodes with an infinite feature, and the same transposed.
    Returns src, dst and the nodes; the other rows have three edges each."""
    gen = torch.Generator(device=DEV).manual_seed(n)
    src, dst = [torch.randint(0, n - 20, (3 * n,), generator=gen, device=DEV)], [torch.randint(0, n - 20, (3 * n,), generator=gen, device=DEV)]
    for deg in range(1, 51):
        src += [torch.randint(0, n - 20, (deg,), generator=gen, device=DEV), torch.tensor([n - 1 - deg % 20], device=DEV)]
        dst += [torch.full((deg + 1,), 3 * deg, device=DEV)]
    src, dst = torch.cat(src).int(), torch.cat(dst).int()
    return torch.cat([src, dst]), torch.cat([dst, src]), torch.arange(n - 20, n, device=DEV)


@pytest.mark.parametrize("n,F,dtype", [(1500, 12, "f32"), (1500, 32, "f32"), (1500, 47, "bf16"), (1500, 60, "f32"), (1500, 100, "f32"), (33_000, 16, "f32"),
                                       (33_000, 27, "f32"), (33_000, 32, "bf16"), (33_000, 64, "bf16"), (70_000, 47, "f32"), (90_000, 72, "bf16")])
def test_an_infinity_on_the_last_edge_of_a_sum(n, F, dtype):
    """Whatever a kernel takes for the edges that a row's last step is short of, it is not zero times the last edge's row: a sum with an
    infinite term is infinite in that column and finite in the others."""
    src, dst, nodes = _infinite_last_sources(n)
    if n > 33_000:   # rows of a dozen edges and more in an array that the L2 holds
        gen = torch.Generator(device=DEV).manual_seed(1)
        more = [torch.randint(0, n - 20, (20 * n,), generator=gen, device=DEV, dtype=torch.int32) for _ in range(2)]
        src, dst = torch.cat([src, more[0]]), torch.cat([dst, more[1]])
    g = api.Graph.from_coo(n, src, dst)
    x = (torch.arange(n * F, device=DEV).view(n, F) % 3 == 0).to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    x[nodes, torch.arange(20, device=DEV) % F] = torch.tensor([float("inf"), -float("inf")], device=DEV, dtype=x.dtype).repeat(10)
    scale = 2.0 ** (torch.arange(n, device=DEV) % 3 - 1).float()
    take = lambda y: torch.zeros(n, F, device=DEV).index_add_(0, dst.long(), y[src.long()])
    want = take(x.float())
    assert bool(want.isinf().any()) and not bool(want.isnan().any())
    assert torch.equal(api.spmm_sum(g.whole, x), want.to(x.dtype))
    assert torch.equal(api.spmm_scaled(g.whole, x, src_scale=scale, dst_scale=scale), (take(x.float() * scale[:, None]) * scale[:, None]).to(x.dtype))


@pytest.mark.parametrize("H,F,dtype", [(5, 24, "bf16"), (8, 24, "bf16"), (6, 12, "f32"), (5, 16, "f32")])
@pytest.mark.parametrize("threshold", [0, 100, 256])
@pytest.mark.parametrize("masked", [False, True])
def test_long_rows_that_the_warps_of_a_block_share(H, F, dtype, threshold, masked):
    """Rows that fill a warp, with ones on either side of 96 edges among them: one to four in a block, of lengths that are and are not worth sharing;
    segments of 100, of 256 and of less, a block each; unsplit rows of 1,000.  With half of the sources masked whole warps have nothing to add."""
    n, gen = 16_100, torch.Generator().manual_seed(H * F)
    degs = [(96, 2, 1, 0), (97, 1, 2, 3), (0, 98, 0, 0), (1, 2, 129, 97), (200, 200, 200, 200), (255, 97, 100, 1), (97, 97, 97, 97), (240, 0, 200, 5),
            (300, 0, 0, 1), (1000, 1, 0, 2), (101, 350, 1, 99), (256, 257, 3, 400)]
    deg = torch.tensor(degs).flatten()
    src = [torch.randint(100, n, (n // 2,), generator=gen), torch.randint(100, n, (int(deg.sum()),), generator=gen), n - 1 - torch.arange(n) % 100]
    dst = [torch.randint(100, n, (n // 2,), generator=gen), 200 + torch.arange(deg.numel()).repeat_interleave(deg), torch.arange(n)]
    src, dst = torch.cat(src).int(), torch.cat(dst).int()
    both = torch.cat([src, dst]), torch.cat([dst, src])
    p = Problem(n, both[0], both[1], H, F, 3, dtype=dtype, k=2, threshold=threshold, build_parts=True)
    if masked:
        off = torch.arange(n) < n // 2
        p.host["er"][off.numpy()] = -np.inf
        p.dev["er"][off.to(DEV)] = -float("inf")
    with Launches() as ran:
        _full_check(p, dtype=dtype, modes=("fused", "stateful"), grad_floor=10.0)
    assert ran.only("_short"), set(ran.names)


@pytest.mark.parametrize("H,F,dtype", [(8, 24, "bf16"), (6, 12, "f32"), (8, 8, "f32"), (3, 16, "bf16"), (1, 16, "f32")])
def test_partitions_without_sources(H, F, dtype):
    """More partitions than nodes: steps whose source-major pass has no rows."""
    n, gen = 40, torch.Generator().manual_seed(H)
    src, dst = (torch.randint(0, n, (90,), generator=gen).int() for _ in range(2))
    p = Problem(n, src, dst, H, F, 5, dtype=dtype, k=64, build_parts=True)
    assert any(part.n_src == 0 for part in p.graph.parts)
    _full_check(p, dtype=dtype, modes=("stateful",), grad_floor=1.0)


@pytest.mark.parametrize("H,F,dtype", [(1, 16, "f32"), (1, 32, "f32"), (2, 8, "bf16"), (4, 8, "bf16"), (4, 24, "bf16"), (8, 24, "bf16")])
def test_an_infinity_on_the_last_edge_of_a_short_row(H, F, dtype):
    n = 33_000
    src, dst, nodes = _infinite_last_sources(n)
    g = api.Graph.from_coo(n, src, dst)
    gen = torch.Generator(device=DEV).manual_seed(H * F)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    feat, gout = (torch.randn(n, H, F, generator=gen, device=DEV).to(dt) for _ in range(2))
    el, er = (torch.randn(n, H, generator=gen, device=DEV) for _ in range(2))
    feat_inf, gout_inf = feat.clone(), gout.clone()
    for x in (feat_inf, gout_inf):
        x[nodes, :, torch.arange(20, device=DEV) % F] = float("inf")
    with Launches() as ran:
        out, m, d = api.gat_forward(g, feat_inf, el, er, 0.2)[:3]
        # (with finite features, whose dot products with an infinite gradient do not enter dfeat)
        dfeat = api.gat_backward(g, feat, el, er, m, d, gout_inf, 0.2)[0]
    assert ran.only("_short"), set(ran.names)
    s, t = src.long(), dst.long()
    alpha = torch.exp(torch.nn.functional.leaky_relu(el[t].double() + er[s].double(), 0.2) - m[t].double()) / d[t].double()
    for got, to, x in ((out, t, feat_inf[s]), (dfeat, s, gout_inf[t])):
        want = torch.zeros(n, H, F, device=DEV, dtype=torch.float64).index_add_(0, to, alpha[..., None] * x.double())
        assert bool(want.isinf().any()) and torch.equal(got.double().isinf(), want.isinf()) and not bool(got.isnan().any())
        ok = want.isfinite().cpu().numpy()
        check_grad(got[want.isfinite()], want.cpu().numpy()[ok], dtype, "finite columns", stored=True)


@pytest.mark.parametrize("H,F,dtype", [(1, 64, "bf16"), (5, 8, "f32"), (6, 24, "bf16"), (10, 16, "f32"), (11, 8, "bf16"), (16, 32, "f32"),
                                       (17, 8, "f32"), (1, 1030, "bf16")])
@pytest.mark.parametrize("many", [False, True])
def test_merges_on_either_side_of_what_a_warp_takes(H, F, dtype, many):
    """Rows of 2 to 40 segments next to each other (where there are many long rows a warp merges up to 32, a block more), of a number that does
    not fill the last block, with heads on either side of what one step of the destination-major merge (5 and 10) and a warp (16) take."""
    n, size, gen = 900, 20, torch.Generator().manual_seed(H)
    src, dst = [torch.randint(0, n, (3 * n,), generator=gen)], [torch.randint(100, n, (3 * n,), generator=gen)]
    for i, segs in enumerate([2, 32, 33, 3, 31, 32, 34, 65, 32, 1, 4, 40, 8, 9]):
        for row, deg in ((3 * i, segs * size), (3 * i + 1, segs * size - 1)):
            src.append(torch.randint(100, n, (deg,), generator=gen))
            dst.append(torch.full((deg,), row))
    if many:
        src.append(torch.randint(100, n, (300 * 2 * size,), generator=gen))
        dst.append(torch.arange(500, 800).repeat_interleave(2 * size))
    src, dst = torch.cat(src).int(), torch.cat(dst).int()
    both = torch.cat([src, dst]), torch.cat([dst, src])   # long rows among the columns, which the source-major pass walks
    p = Problem(n, both[0], both[1], H, F, 5, dtype=dtype, k=2, threshold=size, build_parts=True)
    _full_check(p, dtype=dtype, modes=("fused", "stateful"), grad_floor=max(10.0, F / 64))


@pytest.mark.parametrize("H,F,dtype", [(1, 64, "bf16"), (5, 8, "f32"), (8, 24, "bf16"), (10, 16, "f32"), (16, 8, "f32")])
@pytest.mark.parametrize("many", [False, True])
def test_merges_of_hubs(H, F, dtype, many):
    """Rows of 520 segments among short ones, four of them in a block or one after the other, and rows on either side of the 64 that one
    warp sums for the destination-major pass and of the steps in which four warps do."""
    n, size, gen = 1200, 3, torch.Generator().manual_seed(H)
    segs = [520, 2, 519, 64, 65, 521, 63, 66, 520, 127, 128, 129, 130, 512, 3]
    if many:   # of 300 to 303 long rows a block has every 75th or 76th
        segs += [2] * 288
        for at in (75, 76, 150, 152, 225, 228):
            segs[at] = 520
    deg = torch.tensor([s * size - i % 2 for i, s in enumerate(segs)])
    src = [torch.randint(600, n, (n,), generator=gen), torch.randint(600, n, (int(deg.sum()),), generator=gen)]
    dst = [torch.randint(600, n, (n,), generator=gen), torch.arange(len(segs)).repeat_interleave(deg)]
    src, dst = torch.cat(src).int(), torch.cat(dst).int()
    both = torch.cat([src, dst]), torch.cat([dst, src])
    p = Problem(n, both[0], both[1], H, F, 5, dtype=dtype, k=2, threshold=size, build_parts=True)
    _full_check(p, dtype=dtype, modes=("fused", "stateful"), grad_floor=10.0)


@pytest.mark.parametrize("F", [1, 3, 47, 48, 127, 180, 260, 1030])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n", [1500, 40_000])
def test_sums_of_ragged_rows(F, dtype, n):
    """Sums of small whole numbers are exact in float32 and, below 256, in bf16."""
    spec = workloads.ChungLuSpec(n=n, e=6 * n, gamma=2.1, d_max=300.0, seed=8)
    src, dst = (x.to(DEV) for x in workloads.chung_lu_edges(spec))
    g = api.Graph.from_coo(n, src, dst, threshold=64)
    x = (torch.arange(n * F, device=DEV).view(n, F) % 3 == 0).to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    want = torch.zeros(n, F, device=DEV).index_add_(0, dst.long(), x.float()[src.long()])
    got = api.spmm_sum(g.whole, x)
    assert torch.equal(got, want.to(x.dtype))
    scale = torch.full((n,), 2.0, device=DEV)
    out = x.clone()
    api.spmm_scaled(g.whole, x, src_scale=scale, dst_scale=scale, out=out, first=False)   # += 4 * sum
    assert torch.equal(out, (x.float() + 4.0 * want).to(x.dtype))


@pytest.mark.parametrize("F,dtype", [(3, "f32"), (16, "f32"), (32, "f32"), (47, "bf16")])
@pytest.mark.parametrize("k", [1, 3])
@pytest.mark.parametrize("scaled", [False, True])
def test_means_and_propagation_over_short_rows(F, dtype, k, scaled):
    """The ends of the short-row kernel's sum: the mean, factors of sources and rows, what earlier partitions left, the propagation's mix with and
    without the next step's factor; rows without edges, of 25 and more, and split ones."""
    n, tdt = 40_000, torch.bfloat16 if dtype == "bf16" else torch.float32
    gen = torch.Generator().manual_seed(F + k)
    src, dst = [torch.randint(0, n - 5, (2 * n,), generator=gen)], [torch.randint(100, n - 5, (2 * n,), generator=gen)]   # the last five: no edges
    for row, deg in enumerate([1, 4, 24, 25, 26, 63, 64, 65, 200]):
        src.append(torch.randint(0, n - 5, (deg,), generator=gen))
        dst.append(torch.full((deg,), 3 * row))
    src, dst = torch.cat(src), torch.cat(dst)
    e = src.numel()
    g = api.Graph.from_coo(n, src.int().to(DEV), dst.int().to(DEV), k=k, build_parts=k > 1, threshold=64)
    adj = torch.sparse_coo_tensor(torch.stack([dst, src]), torch.ones(e, dtype=torch.float64), (n, n)).to_sparse_csr()
    x0 = torch.randn((n, F), generator=gen).to(tdt)
    deg = torch.bincount(dst, minlength=n)
    s = torch.rand(n, generator=gen) + 0.5 if scaled else None
    d = 1.0 / deg.clamp(min=1).float()
    # sums of up to 200 float32 terms of size 1; a stored bf16 rounds by 2^-9 of its value in every step
    tol = dict(rtol=1e-5, atol=1e-5) if dtype == "f32" else dict(rtol=2e-2, atol=2e-2)
    with Launches() as ran:
        mean = api.spmm_sum(g.whole, x0.to(DEV), mean=True, deg_total=deg.to(DEV))
        got = api.propagate(g, x0.to(DEV), 0.7, 2, s.to(DEV) if scaled else None, d.to(DEV))
    assert ran.only("_short", ("spmm",)), set(ran.names)
    allclose_report(mean.double().cpu().numpy(), ((adj @ x0.double()) * d.double()[:, None]).numpy(), what="mean", **tol)
    want = x0.double()
    for _ in range(2):
        y = want * s.double()[:, None] if scaled else want
        want = 0.3 * x0.double() + 0.7 * d.double()[:, None] * (adj @ y)
    allclose_report(got.double().cpu().numpy(), want.numpy(), what="propagation", **tol)


@pytest.mark.parametrize("F,dtype", [(32, "f32"), (36, "f32"), (47, "f32"), (64, "f32"), (101, "f32"), (128, "f32"), (160, "f32"), (193, "f32"),
                                     (72, "bf16"), (100, "bf16"), (256, "bf16"), (333, "bf16")])
@pytest.mark.parametrize("mb,deg,long", [(13, 11, False), (13, 13, False), (13, 21, True), (39, 21, False), (42, 21, False)])
def test_sums_on_either_side_of_the_span_kernels_line(F, dtype, mb, deg, long):
    """Arrays of 13 to 42 MB and rows of 11 to 21 edges: where the number of edges, the size of the array, weights, long rows and the mix of
    a propagation choose between the row and the span kernels.  Whole numbers, exact in float32: one rounding where the result is bf16."""
    tdt, size = (torch.bfloat16, 2) if dtype == "bf16" else (torch.float32, 4)
    n = mb * 1_000_000 // ((F * size + 15) // 16 * 16)
    gen = torch.Generator(device=DEV).manual_seed(F + deg)
    src, dst = (torch.randint(0, n, (deg * n,), generator=gen, device=DEV, dtype=torch.int32) for _ in range(2))
    if long:
        dst[:300], dst[300:1200] = 5, n - 1
    g = api.Graph.from_coo(n, src, dst, threshold=200)
    x = (torch.arange(n * F, device=DEV).view(n, F) % 3 == 0).to(tdt)
    scale = 2.0 ** (torch.arange(n, device=DEV) % 3 - 1).float()
    take = lambda y: torch.zeros(n, F, device=DEV).index_add_(0, dst.long(), y[src.long()])
    want = take(x.float() * scale[:, None]) * scale[:, None]
    assert torch.equal(api.spmm_sum(g.whole, x), take(x.float()).to(tdt))
    assert torch.equal(api.spmm_scaled(g.whole, x, src_scale=scale, dst_scale=scale), want.to(tdt))
    assert torch.equal(api.propagate(g, x, 0.5, 1, scale, scale), (0.5 * x.float() + 0.5 * want).to(tdt))


def test_row_pointers_that_claim_more_edges_than_there_are():
    """A row of 2^31 + 5 edges by its pointers has the graph's last edges again and again in the short-row kernel's sum, and the sum ends;
    the other rows are what they were."""
    n, row = 33_000, 1234
    gen = torch.Generator(device=DEV).manual_seed(2)
    src, dst = (torch.randint(0, n, (3 * n,), generator=gen, device=DEV, dtype=torch.int32) for _ in range(2))
    g = api.Graph.from_coo(n, src, dst)
    x = torch.randn(n, 16, generator=gen, device=DEV)
    with Launches() as ran:
        want = api.spmm_sum(g.whole, x)
    assert ran.only("_short", ("spmm",)) and g.whole.split.n_long == 0
    g.whole.indptr[row + 1] = g.whole.indptr[row] + 2 ** 31 + 5
    got = api.spmm_sum(g.whole, x)
    others = torch.arange(n, device=DEV) // 2 != row // 2   # (the next row's pointers end before they begin)
    assert torch.equal(got[others], want[others])


def test_ragged_shape_without_room_for_padded_copies():
    """No workspace in the forward call, one that holds the records alone in the backward call: the scalar kernels."""
    n, src, dst = hub_graph(n=500, e=6000, d_max=100.0, seed=3)
    p = Problem(n, src, dst, 2, 7, 4, threshold=512)
    d, f = p.dev, p.oracle_fwd()
    out, m, dd = torch.empty_like(d["feat"]), torch.empty_like(d["el"]), torch.empty_like(d["el"])
    B.sar_gat_fwd(p.graph.whole, d["feat"], d["el"], d["er"], 2, 7, 0.2, B.SAR_FIRST | B.SAR_LAST, None, m, dd, out, None)
    check_out(out, f.out, "f32", "out")
    b = p.oracle_bwd(f)
    dfeat, del_, der = torch.empty_like(d["feat"]), torch.empty_like(m), torch.empty_like(m)
    ws = torch.empty((n * 2 * 16 + 255) // 256 * 256, dtype=torch.uint8, device=DEV)
    B.sar_gat_bwd(p.graph.whole, d["feat"], d["el"], d["er"], m, dd, d["gout"], 2, 7, 0.2, B.SAR_FIRST | B.SAR_LAST, dfeat, del_, der, ws)
    for got, want in ((dfeat, b.dfeat), (del_, b.del_), (der, b.der)):
        allclose_report(got.cpu().numpy(), np.asarray(want), 1e-4, 1e-5, "gradients")


@pytest.mark.parametrize("H,F,dtype", [(1, 47, "bf16"), (2, 7, "f32")])
def test_ragged_steps_with_a_workspace_each(H, F, dtype):
    """A step of the backward pass needs of its workspace what sar_gat_bwd_prepare wrote and nothing that an earlier step left."""
    n, src, dst = hub_graph(n=1200, e=15000, d_max=300.0, seed=23)
    p = Problem(n, src, dst, H, F, 12, dtype=dtype, k=3, threshold=24, build_parts=True)
    d, g = p.dev, p.graph
    out, m, dd, acc = api.gat_forward(g, d["feat"], d["el"], d["er"], 0.2, mode="stateful", keep_numerator=True)
    want = api.gat_backward(g, d["feat"], d["el"], d["er"], m, dd, d["gout"], 0.2, mode="stateful", acc=acc)
    dfeat, del_, der = torch.empty_like(d["feat"]), torch.empty_like(m), torch.empty_like(m)
    for q, part in enumerate(g.parts):
        nbytes = B.sar_gat_workspace_bytes(part, H, F, B.SAR_BF16 if dtype == "bf16" else B.SAR_F32)
        ws = torch.full((nbytes,), 0x7f, dtype=torch.uint8, device=DEV)
        B.sar_gat_bwd_prepare(n, H, F, acc, True, d["gout"], d["el"], m, dd, None, ws)
        s0, s1 = g.bounds[q], g.bounds[q + 1]
        B.sar_gat_bwd(part, d["feat"][s0:s1], d["el"], d["er"][s0:s1], m, dd, d["gout"], H, F, 0.2,
                      (B.SAR_FIRST if q == 0 else 0) | (B.SAR_LAST if q == 2 else 0), dfeat[s0:s1], del_, der[s0:s1], ws)
    for got, ref in zip((dfeat, del_, der), want):
        assert torch.equal(got, ref)


@pytest.mark.parametrize("H,F,dtype", [(4, 16, "f32"), (4, 32, "f32"), (8, 32, "bf16"), (4, 64, "f32")])
@pytest.mark.parametrize("threshold,many", [(3, True), (100, False)])
def test_segments_of_the_lean_kernels(H, F, dtype, threshold, many):
    """Few segments run as the first blocks of the rows' grid, from 148 * 256 on in a launch of their own."""
    n, src, dst = hub_graph(n=9000, e=300_000, d_max=1500.0, seed=H * F)
    p = Problem(n, src, dst, H, F, 5, dtype=dtype, k=2, threshold=threshold, build_parts=True)
    for part in [p.graph.whole] + p.graph.parts:
        for split in (part.split, part.t_split):
            assert split.n_seg >= 148 * 256 if many else 0 < split.n_seg < 148 * 256
    _full_check(p, dtype=dtype, modes=("fused", "stateful"), grad_floor=10.0)


@pytest.mark.parametrize("H,F,dtype", [(6, 48, "bf16"), (12, 16, "f32")])
@pytest.mark.parametrize("threshold", [7, 150, 230, 600])
def test_segments_of_the_span_kernels(H, F, dtype, threshold):
    """Segments shorter and longer than the chunks a span kernel stages (192 and 256 edges), whole and step by step.
    Heavier hubs than these leave the fixed tolerance: an element of dfeat sums D terms alpha * gout whose alpha carries about
    2^-21 (an exponential of an argument of up to 16), that is an error of 2^-21 sqrt(D sum alpha^2 / D): 1e-5 for D = 1500 and
    mean alpha^2 = 0.3, the tolerance's floor, and 2e-5 for D = 5000 (seen there: 5e-5, one element in four million)."""
    n, src, dst = hub_graph(n=20_500, e=170_000, d_max=1500.0, seed=H + F)
    p = Problem(n, src, dst, H, F, 9, dtype=dtype, k=2, threshold=threshold, build_parts=True)
    assert p.graph.whole.split.n_seg > 0 and p.graph.whole.t_split.n_seg > 0
    _full_check(p, dtype=dtype, modes=("fused", "stateful"), grad_floor=10.0)
