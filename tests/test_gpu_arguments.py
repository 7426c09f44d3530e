"""Arguments of the wrong type or size are refused by the native side of api.py: the library sees pointers only and would read
past the end of a smaller array (or take a float32 array's place for a bf16 one's)."""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"
N, H, F, D_IN = 64, 4, 8, 16

if torch.cuda.is_available():
    from paper_2111_06483_b200 import api


def graph(k=1):
    i = torch.arange(N, dtype=torch.int32, device=DEV)
    return api.Graph.from_coo(N, i, (i + 1) % N, k=k, build_parts=k > 1)


def f32(*shape):
    return torch.zeros(*shape, device=DEV)


def bf16(*shape):
    return torch.zeros(*shape, device=DEV, dtype=torch.bfloat16)


def refused(call, good, **bad):
    """call(**good) runs; with any one of the arguments replaced it is refused."""
    call(**good)
    for name, values in bad.items():
        for v in values:
            with pytest.raises(AssertionError):
                call(**{**good, name: v})


@pytest.mark.parametrize("k", [1, 3])
def test_attention(k):
    g = graph(k)
    mode = "stateful" if k > 1 else "fused"
    refused(lambda feat, el, er: api.gat_forward(g, feat, el, er, 0.2, mode=mode), dict(feat=f32(N, H, F), el=f32(N, H), er=f32(N, H)),
            feat=[f32(N - 1, H, F)], el=[bf16(N, H), f32(N - 1, H)], er=[bf16(N, H), f32(N - 1, H)])
    refused(lambda feat, el, er, m, d, gout, out: api.gat_backward(g, feat, el, er, m, d, gout, 0.2, out=out, mode=mode),
            dict(feat=f32(N, H, F), el=f32(N, H), er=f32(N, H), m=f32(N, H), d=f32(N, H), gout=f32(N, H, F), out=f32(N, H, F)),
            feat=[f32(N - 1, H, F)], el=[bf16(N, H)], er=[f32(N - 1, H)], m=[f32(N, H - 1)], d=[bf16(N, H)],
            gout=[bf16(N, H, F), f32(N - 1, H, F)], **(dict(out=[bf16(N, H, F), f32(N, H)]) if k > 1 else {}))


def test_sums():
    g = graph()
    deg = torch.ones(N, dtype=torch.int64, device=DEV)
    refused(lambda x, deg: api.spmm_sum(g.whole, x, mean=True, deg_total=deg), dict(x=f32(N, F), deg=deg),
            x=[f32(N - 1, F)], deg=[deg.int(), deg[1:]])
    refused(lambda x, s, d, out: api.spmm_scaled(g.whole, x, s, d, out), dict(x=f32(N, F), s=f32(N), d=f32(N), out=f32(N, F)),
            x=[f32(N - 1, F)], s=[bf16(N), f32(N - 1)], d=[bf16(N), f32(N - 1)], out=[bf16(N, F), f32(N - 1, F)])
    for k in (1, 2):
        gk = graph(k)
        refused(lambda x, s, d: api.propagate(gk, x, 0.5, 2, s, d), dict(x=f32(N, F), s=f32(N), d=f32(N)),
                x=[f32(N - 1, F)], s=[bf16(N), f32(N - 1)], d=[bf16(N), f32(N - 1)])


@pytest.mark.parametrize("feat", [F, 12])   # the scores from the projection's epilogue, and from a pass of their own
def test_attention_layer(feat):
    g = graph()
    good = dict(h=bf16(N, D_IN), W=bf16(D_IN, H * feat), a_l=f32(H, feat), a_r=f32(H, feat))
    bad = dict(W=[bf16(D_IN, H * feat - 8), bf16(D_IN - 8, H * feat), bf16(D_IN, H, feat), f32(D_IN, H * feat)], a_l=[bf16(H, feat)],
               a_r=[bf16(H, feat), f32(H - 1, feat)])
    refused(lambda **a: api.full_layer_forward(g, slope=0.2, **a), good, h=[bf16(N - 1, D_IN)], **bad)
    out, saved = api.full_layer_forward(g, slope=0.2, **good)
    for relu in (False, True):
        refused(lambda z, gout, **a: api.full_layer_backward(g, saved=(z, *saved[1:]), gout=gout, slope=0.2, relu_input=relu, **a),
                dict(z=saved[0], gout=out, **good), z=[saved[0][1:], saved[0].float()], gout=[out[1:], out.float()], **bad)


def test_sage_layer():
    g = graph()
    good = dict(h=bf16(N, D_IN), W=bf16(D_IN, 24), W_res=bf16(D_IN, 24))
    bad = dict(W=[bf16(D_IN - 8, 24), f32(D_IN, 24)], W_res=[bf16(D_IN, 16), f32(D_IN, 24)])
    refused(lambda inv, **a: api.sage_layer_forward(g, inv=inv, **a), dict(inv=f32(N), **good), h=[bf16(N - 1, D_IN)],
            inv=[bf16(N), f32(N - 1)], **bad)
    refused(lambda agg, inv, gpre, **a: api.sage_layer_backward(g, saved=(agg, inv), gpre=gpre, **a),
            dict(agg=bf16(N, D_IN), inv=f32(N), gpre=bf16(N, 24), **good), agg=[bf16(N - 1, D_IN), f32(N, D_IN)],
            inv=[bf16(N), f32(N - 1)], gpre=[f32(N, 24), bf16(N - 1, 24)], **bad)


def test_batch_normalisation():
    x = torch.randn(N, F, device=DEV)
    refused(lambda gamma, beta: api.bn_forward(x, gamma=gamma, beta=beta), dict(gamma=f32(F), beta=f32(F)),
            gamma=[bf16(F), f32(F - 1)], beta=[bf16(F), f32(F - 1)])
    _, (mean, rstd, n) = api.bn_forward(x)
    refused(lambda gy, mean, rstd, gamma: api.bn_backward(x, gy, (mean, rstd, n), gamma=gamma),
            dict(gy=x, mean=mean, rstd=rstd, gamma=f32(F)), gy=[x.bfloat16(), x[1:]], mean=[mean[1:]], rstd=[rstd.bfloat16()],
            gamma=[f32(F - 1)])
