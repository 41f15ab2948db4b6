"""Outputs in the storage of an operand or of the ReLU gate, in multiplies of several waves whose bit-width shows only outside
the tiles that the guess is made from: nothing that is read again has been overwritten (bit-exact against separate buffers)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def niti():
    from paper_2009_13108_b200 import Niti
    n = Niti(0)
    yield n
    n.check()
    n.close()


def _i8(seed, *shape):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randint(-127, 128, shape, generator=g, dtype=torch.int8, device="cuda")


@pytest.mark.parametrize("M,N,K", [(8192, 256, 2048), (8000, 2048, 1000)])        # single CTAs, pairs
def test_error_in_place_of_the_gate(niti, M, N, K):
    n = niti
    e, w, gate = torch.zeros((M, N), dtype=torch.int8, device=n.device), _i8(1, N, K), _i8(2, M, K)
    e[M - 200:] = _i8(3, 200, N)                  # (the rows before them round to zeros)
    a = gate.clone()
    want, _, b, _ = n.linear_bwd(a, e, w, relu_mask_src=gate)
    assert int((want != 0).sum()) > 0
    for _ in range(3):
        at = gate.clone()
        got, _, b_e, _ = n.linear_bwd(a, e, w, relu_mask_src=at, e_prev=at)
        assert torch.equal(got, want) and int(b_e) == int(b)


@pytest.mark.parametrize("M,K", [(8192, 1024), (300001, 64)])                      # pairs, the row-batched mode's shape
def test_output_in_place_of_an_operand(niti, M, K):
    n = niti
    a, w, sa = _i8(4, M, K), _i8(5, K, K), n.scalar(-7)
    want, _, b = n.linear_fwd(a, sa, w, sa, relu=True)
    for _ in range(3):
        at = a.clone()
        _, _, b_out = n.linear_fwd(at, sa, w, sa, out=at, relu=True)
        assert torch.equal(at, want) and int(b_out) == int(b)


@pytest.mark.parametrize("B,S,Ci,Co,R,pad,stride", [(64, 56, 64, 64, 3, 1, 1), (64, 56, 128, 256, 3, 1, 2), (64, 56, 64, 64, 1, 0, 2)])
def test_convolution_errors_in_place_of_the_gate(niti, B, S, Ci, Co, R, pad, stride):
    n = niti
    So = (S + 2 * pad - R) // stride + 1
    e, w, gate = torch.zeros((B, So, So, Co), dtype=torch.int8, device=n.device), _i8(6, Co, R, R, Ci), _i8(7, B, S, S, Ci)
    e[-1, So // 2:] = _i8(8, So - So // 2, So, Co)
    want, b = n.conv_dgrad(e, w, (S, S), relu_mask_src=gate, pad=pad, stride=stride)
    assert int((want != 0).sum()) > 0
    for _ in range(3):
        gt = gate.clone()
        got, b_e = n.conv_dgrad(e, w, (S, S), e_prev=gt, relu_mask_src=gt, pad=pad, stride=stride)
        assert torch.equal(got, want) and int(b_e) == int(b)


@pytest.mark.parametrize("M,N,K", [(64, 100, 256), (96, 768, 1056), (8192, 256, 2048), (500, 1000, 3000)])
def test_update_with_the_error_in_place_of_the_input(niti, M, N, K):
    """The gradient is that of the input as it was, the error that of the weights as they were."""
    n = niti
    a, e, w = _i8(9, M, K).clamp_(min=0), _i8(10, M, N), _i8(11, N, K)
    w_want = w.clone()
    want, b, b_g = n.linear_bwd_update(a, e, w_want, relu_mask_src=a)
    for _ in range(2):
        at, wt = a.clone(), w.clone()
        got, b_e, b_gt = n.linear_bwd_update(at, e, wt, relu_mask_src=at, e_prev=at)
        assert torch.equal(got, want) and torch.equal(wt, w_want) and (int(b_e), int(b_gt)) == (int(b), int(b_g))


@pytest.mark.parametrize("M,N", [(64, 96), (512, 1024), (8192, 1024)])
def test_error_in_place_of_the_error_above(niti, M, N):
    n = niti
    a, e, w = _i8(12, M, N).clamp_(min=0), _i8(13, M, N), _i8(14, N, N)
    w_want = w.clone()
    want, g, b, b_g = n.linear_bwd(a, e, w, relu_mask_src=a)
    n.linear_bwd_update(a, e, w_want, relu_mask_src=a)
    for _ in range(2):
        et = e.clone()
        got, g_t, b_e, b_gt = n.linear_bwd(a, et, w, relu_mask_src=a, e_prev=et)
        assert torch.equal(got, want) and torch.equal(g_t, g) and (int(b_e), int(b_gt)) == (int(b), int(b_g))
        et, wt = e.clone(), w.clone()
        got, _, _ = n.linear_bwd_update(a, et, wt, relu_mask_src=a, e_prev=et)
        assert torch.equal(got, want) and torch.equal(wt, w_want)


@pytest.mark.parametrize("engine", [0, 1, 2, 4, 5])
@pytest.mark.parametrize("B,S,C,R", [(64, 56, 64, 3), (20, 45, 72, 5), (40, 64, 200, 1), (100, 9, 160, 3)])
def test_convolution_in_place_of_its_input(niti, B, S, C, R, engine):
    n = niti
    x, w, sx = _i8(15, B, S, S, C), _i8(16, C, R, R, C), n.scalar(-7)
    want, _, b = n.conv_fwd(x, sx, w, sx, pad=R // 2, relu=True)
    n.set_engine(engine)
    try:
        xt = x.clone()
        _, _, b_y = n.conv_fwd(xt, sx, w, sx, y=xt, pad=R // 2, relu=True)
    finally:
        n.set_engine(0)
    assert torch.equal(xt, want) and int(b_y) == int(b)
