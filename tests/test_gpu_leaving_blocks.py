"""Launches whose blocks agree on a bit-width need not be resident as a whole: a block that runs out of patience leaves its
share in memory and another one finishes it.  With engine 6 no block has any patience, so every kernel and form takes that
path; results equal those of the waiting form.  Graphs of four contexts on four streams then run against each other."""
import pytest
import torch

from test_gpu_general_shapes import CASES
from test_gpu_ops import POOL_SHAPES

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def niti():
    from paper_2009_13108_b200 import Niti
    n = Niti(0)
    yield n
    n.check()
    n.close()


def _i8(seed, *shape):
    g = torch.Generator(device="cpu").manual_seed(seed)
    return torch.randint(-127, 128, shape, dtype=torch.int8, generator=g).cuda()


def _left(n):
    """Blocks that left in the last call (upper half of the second word of the header that unprepared calls use)."""
    torch.cuda.synchronize()
    return int(n._ws[63 * 4096 + 4:63 * 4096 + 8].view(torch.int32)) >> 16


def _both(n, call):
    """The call's tensors with patience and without; blocks that left without."""
    outs, left = [], 0
    for engine in (0, 6):
        assert n.set_engine(engine) in (0, 6)
        try:
            outs.append([t.clone() for t in call() if t is not None])
            left = _left(n)
        finally:
            assert n.set_engine(0) == engine
    assert len(outs[0]) == len(outs[1]) and all(torch.equal(a, b) for a, b in zip(*outs))
    return left


@pytest.mark.parametrize("M,N,K", [(33, 10, 257), (64, 256, 784), (256, 256, 256), (1000, 500, 250), (96, 64, 1023), (128, 10, 6000),
                                   (300, 3000, 200), (512, 1024, 2048), (64, 1024, 4096), (96, 768, 1056), (500, 1000, 3000)])
def test_linear(niti, M, N, K):
    n = niti
    a, w, e = _i8(M, M, K).clamp_(min=0), _i8(N, N, K), _i8(K, M, N)
    sa, sw = n.scalar(-7), n.scalar(-9)
    left = _both(n, lambda: n.linear_fwd(a, sa, w, sw, relu=True))
    left += _both(n, lambda: n.linear_bwd(a, e, w, relu_mask_src=a))

    def update(need):
        wt = w.clone()
        return list(n.linear_bwd_update(a, e, wt, need_e_prev=need, relu_mask_src=a if need else None)) + [wt]
    left += _both(n, lambda: update(True)) + _both(n, lambda: update(False))
    assert left > 0


@pytest.mark.parametrize("s_a", [-8, -5])
@pytest.mark.parametrize("B,N", [(9, 63), (64, 1000), (40, 1028), (1185, 68), (4737, 72), (2400, 33), (4096, 1000)])
def test_int_xent(niti, B, N, s_a):
    n = niti
    a, labels = _i8(B, B, N), (torch.arange(B, dtype=torch.int32) % N).cuda()
    assert _both(n, lambda: n.int_xent(a, n.scalar(s_a), labels)) > 0


@pytest.mark.parametrize("B,H,W,Ci,Co,R,pad,stride", CASES + [(256, 4, 4, 512, 512, 3, 1, 1), (100, 9, 9, 96, 160, 3, 1, 1),
                                                             (16, 14, 14, 256, 256, 3, 1, 1), (8, 28, 28, 128, 128, 3, 1, 1)])
def test_convolutions(niti, B, H, W, Ci, Co, R, pad, stride):
    n = niti
    Ho, Wo = (H + 2 * pad - R) // stride + 1, (W + 2 * pad - R) // stride + 1
    x, w, e = _i8(B + H, B, H, W, Ci).clamp_(min=0), _i8(Co, Co, R, R, Ci), _i8(W, B, Ho, Wo, Co)
    _both(n, lambda: n.conv_fwd(x, n.scalar(-7), w, n.scalar(-9), pad=pad, relu=True, stride=stride))
    _both(n, lambda: n.conv_dgrad(e, w, (H, W), relu_mask_src=x, pad=pad, stride=stride))
    _both(n, lambda: n.conv_wgrad(x, e, (R, R), pad=pad, stride=stride))
    if stride == 1:
        def update():
            wt = w.clone()
            return [n.conv_wgrad_update(x, e, wt, pad=pad)[-1], wt]
        _both(n, update)


@pytest.mark.parametrize("B,H,W,Ci,Co", POOL_SHAPES)
def test_pooled_convolutions(niti, B, H, W, Ci, Co):
    n = niti
    x, w = _i8(B + H, B, H, W, Ci), _i8(Co, Co, 3, 3, Ci)
    _both(n, lambda: n.conv_fwd_pool(x, n.scalar(-7), w, n.scalar(-9), relu=True))


def test_four_streams_at_once():
    """Every launch of these chains wants most of the SMs for blocks that wait for each other."""
    from paper_2009_13108_b200 import Niti
    ctxs, graphs, wants, outs = [], [], [], []
    for i, (M, N, K) in enumerate([(256, 256, 256), (512, 1024, 1024), (300, 500, 700), (64, 1000, 4096)]):
        n = Niti(0)
        x, w, labels = _i8(i, M, K).clamp_(min=0), _i8(10 + i, N, K), (torch.arange(M, dtype=torch.int32) % N).cuda()
        img, f, e = _i8(20 + i, 32, 8, 8, 128).clamp_(min=0), _i8(30 + i, 128, 3, 3, 128), _i8(40 + i, 32, 8, 8, 128)
        sx, sw, sl = n.scalar(-7), n.scalar(-9), n.scalar(-6)
        bufs = [torch.empty((M, N), dtype=torch.int8, device="cuda"), torch.empty((M, N), dtype=torch.int8, device="cuda"),
                torch.empty((M, K), dtype=torch.int8, device="cuda"), torch.empty((N, K), dtype=torch.int8, device="cuda"),
                torch.empty_like(e), torch.empty_like(img), torch.empty_like(f)]
        scal = [n.scalar() for _ in range(8)]

        def chain(n=n, x=x, w=w, labels=labels, img=img, f=f, e=e, sx=sx, sw=sw, sl=sl, b=bufs, s=scal):
            for _ in range(8):
                n.linear_fwd(x, sx, w, sw, out=b[0], s_out=s[0], b_out=s[1])
                n.int_xent(b[0], sl, labels, e=b[1], b_e=s[2], n_correct=s[3])
                n.linear_bwd(x, b[1], w, relu_mask_src=x, e_prev=b[2], g=b[3], b_e=s[4], b_g=s[5])
                n.conv_fwd(img, sx, f, sw, y=b[4], s_y=s[0], b_y=s[1], relu=True)
                n.conv_dgrad(e, f, (8, 8), e_prev=b[5], relu_mask_src=img, b_e=s[6])
                n.conv_wgrad(img, e, g=b[6], b_g=s[7])
        chain()
        torch.cuda.synchronize()
        wants.append([t.clone() for t in bufs])
        stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            chain()
        ctxs.append((n, chain))                     # (the chain holds the graph's inputs)
        graphs.append((stream, graph))
        outs.append(bufs)
    for _ in range(10):
        for b in outs:
            for t in b:
                t.fill_(77)
        torch.cuda.synchronize()
        for _ in range(3):
            for stream, graph in graphs:
                with torch.cuda.stream(stream):
                    graph.replay()
        torch.cuda.synchronize()
        for b, want in zip(outs, wants):
            assert all(torch.equal(t, u) for t, u in zip(b, want))
    for n, _ in ctxs:
        n.check()                                   # (no wait ran out)
        n.close()
