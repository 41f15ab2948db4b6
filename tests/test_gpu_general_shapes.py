"""Shapes of the tensor-core engine's general forms, against the CPU oracle (bit-exact): im2col copies (image
sides and strides no pixel box tiles), short channel chunks, operands padded to 16-byte rows, output rows of
any pitch, the phases of a strided error, gathered first layers of more than 32 taps."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

CASES = [
    # B, H, W, Ci, Co, R, pad, stride
    (3, 27, 27, 96, 64, 5, 2, 1),       # chunk of 96 channels, rows of a tile across images
    (2, 7, 7, 192, 160, 3, 1, 1),       # two chunks, the second short; 98 output rows
    (5, 13, 9, 48, 96, 3, 1, 1),        # 16 of 32 elements of the last MMA are fill
    (2, 15, 11, 24, 72, 3, 1, 1),       # pixels padded to 16-byte pitches, 8-byte output units
    (4, 12, 12, 20, 50, 5, 0, 1),       # 4- and 2-byte output units
    (2, 9, 14, 33, 37, 3, 1, 1),        # odd channel counts: single bytes
    (2, 16, 16, 96, 96, 5, 2, 1),       # exact pixel boxes with short channel chunks
    (2, 16, 16, 256, 96, 3, 1, 1), (4, 16, 8, 160, 256, 3, 1, 1), (2, 16, 32, 48, 128, 3, 1, 1),
    (128, 3, 5, 96, 256, 3, 1, 1),      # pixel boxes of one pixel in 128 images
    (2, 36, 36, 48, 96, 3, 1, 1),       # resident weights with short channel chunks (48 of 64, 96 of 128)
    (3, 19, 26, 24, 40, 3, 1, 1), (2, 32, 24, 16, 72, 3, 1, 1), (2, 20, 11, 112, 24, 3, 1, 1),
    (3, 16, 8, 64, 64, 3, 1, 1), (2, 15, 15, 32, 64, 3, 1, 1), (4, 14, 16, 64, 128, 3, 1, 1),   # one patch high
    (90, 17, 15, 24, 72, 3, 1, 1), (90, 16, 16, 48, 96, 3, 1, 1), (40, 24, 24, 96, 256, 3, 1, 1),   # tap groups
    (40, 23, 24, 112, 288, 3, 1, 1), (90, 16, 16, 32, 40, 5, 2, 1), (90, 33, 31, 64, 128, 3, 1, 2),
    (3, 16, 16, 64, 64, 3, 1, 2),       # strided error: four phases of 4, 2, 2 and 1 taps
    (2, 17, 23, 32, 96, 3, 1, 2),
    (2, 19, 13, 64, 32, 5, 2, 3),
    (2, 21, 18, 32, 64, 1, 0, 2),       # filter smaller than the stride: untouched phases are zero
    (1, 40, 33, 16, 48, 3, 0, 4),
    (2, 30, 30, 32, 32, 4, 1, 2),       # even filter, no phase is shorter
    (2, 31, 31, 64, 64, 7, 5, 2),       # padding larger than (R - 1) / 2
    (2, 3, 9, 32, 32, 1, 1, 4), (2, 1, 7, 32, 32, 1, 1, 2),     # strided error without a single position: zeros
    (3, 29, 31, 3, 40, 11, 2, 4),       # gathered rows of 384 bytes
    (2, 33, 20, 3, 24, 7, 3, 2),
    (2, 21, 300, 1, 17, 5, 2, 1),       # two row segments
    (2, 18, 26, 4, 64, 5, 2, 1),
]


@pytest.fixture(scope="module")
def niti():
    from paper_2009_13108_b200 import Niti
    n = Niti(0)
    yield n
    n.check()
    n.close()


@pytest.mark.parametrize("B,H,W,Ci,Co,R,pad,stride", CASES)
def test_general_convolutions(niti, oref, B, H, W, Ci, Co, R, pad, stride):
    rng = np.random.default_rng(B + 3 * H + 5 * W + 7 * Ci + 11 * Co + 13 * R + stride)
    i8 = lambda *s: rng.integers(-127, 128, size=s, dtype=np.int8)  # noqa: E731
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(niti.device)  # noqa: E731
    Ho, Wo = oref.conv_out_hw(H, W, R, R, pad, stride)
    x, w, e = np.maximum(i8(B, H, W, Ci), 0), i8(Co, R, R, Ci), i8(B, Ho, Wo, Co)
    for relu in (False, True):
        wy, s, b = oref.conv_fwd(x, -7, w, -9, pad, relu, stride=stride)
        y, s_y, b_y = niti.conv_fwd(T(x), niti.scalar(-7), T(w), niti.scalar(-9), pad=pad, relu=relu, stride=stride)
        assert np.array_equal(y.cpu().numpy(), wy) and (int(s_y), int(b_y)) == (s, b)
    for mask in (None, x):
        wd, bd = oref.conv_dgrad(e, w, (H, W), pad, mask, stride=stride)
        ep, b_e = niti.conv_dgrad(T(e), T(w), (H, W), e_prev=torch.full((B, H, W, Ci), 99, dtype=torch.int8, device=niti.device),
                                  relu_mask_src=None if mask is None else T(mask), pad=pad, stride=stride)
        assert np.array_equal(ep.cpu().numpy(), wd) and int(b_e) == bd
    wg, bg = oref.conv_wgrad(x, e, (R, R), pad, 5, stride=stride)
    g, b_g = niti.conv_wgrad(T(x), T(e), (R, R), pad=pad, stride=stride)
    assert np.array_equal(g.cpu().numpy(), wg) and int(b_g) == bg
    if stride == 1:
        wt = T(w)
        niti.conv_wgrad_update(T(x), T(e), wt, pad=pad)
        assert np.array_equal(wt.cpu().numpy(), oref.sgd_update(w, wg))


@pytest.mark.parametrize("M,N,K", [(300, 257, 100), (1, 33, 47), (129, 1000, 515), (640, 37, 1030), (77, 250, 4098)])
def test_general_matrices(niti, oref, M, N, K):
    rng = np.random.default_rng(M + N + K)
    i8 = lambda *s: rng.integers(-127, 128, size=s, dtype=np.int8)  # noqa: E731
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(niti.device)  # noqa: E731
    a, w, e = np.maximum(i8(M, K), 0), i8(N, K), i8(M, N)
    want, s, b = oref.linear_fwd(a, -7, w, -9, True)
    out, s_out, b_out = niti.linear_fwd(T(a), niti.scalar(-7), T(w), niti.scalar(-9), relu=True)
    assert np.array_equal(out.cpu().numpy(), want) and (int(s_out), int(b_out)) == (s, b)
    we, wg, be, bg = oref.linear_bwd(a, e, w, True, a, 5)
    ep, g, b_e, b_g = niti.linear_bwd(T(a), T(e), T(w), True, T(a))
    assert np.array_equal(ep.cpu().numpy(), we) and np.array_equal(g.cpu().numpy(), wg)
    assert (int(b_e), int(b_g)) == (be, bg)
