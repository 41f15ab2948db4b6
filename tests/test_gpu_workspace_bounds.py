"""Few-channel convolutions on a workspace of exactly the queried size, with guard bytes behind it: no call writes past its
end, and results equal the CPU oracle's (bit-exact).  Strides above 8 and layers that a forced engine refuses take the
CUDA-core engine; gathered and widened ones stay beside them as controls."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
GUARD = 8 << 20


@pytest.mark.parametrize("engine,B,H,W,Ci,Co,R,pad,stride", [
    (0, 4, 96, 96, 3, 40, 16, 0, 16), (0, 2, 63, 70, 3, 24, 14, 0, 14), (0, 3, 50, 41, 1, 32, 9, 2, 9),
    (0, 2, 60, 60, 4, 17, 12, 3, 12), (0, 2, 41, 40, 3, 20, 3, 1, 10), (0, 2, 40, 33, 20, 24, 3, 1, 9),
    (3, 2, 32, 32, 3, 64, 7, 3, 2), (3, 2, 30, 30, 3, 24, 5, 2, 1), (3, 2, 20, 20, 3, 24, 3, 1, 1),
    (0, 2, 33, 20, 3, 24, 7, 3, 2), (0, 2, 12, 12, 20, 50, 5, 0, 1)])
def test_calls_stay_inside_the_workspace(oref, engine, B, H, W, Ci, Co, R, pad, stride):
    from paper_2009_13108_b200 import Niti
    from paper_2009_13108_b200.api import OP_CONV_FWD, OP_CONV_DGRAD, OP_CONV_WGRAD, OP_CONV_WGRAD_UPDATE
    n = Niti(0)
    n.set_engine(engine)
    rng = np.random.default_rng(B + 3 * H + 5 * W + 7 * Ci + 11 * Co + 13 * R + stride)
    i8 = lambda *s: rng.integers(-127, 128, size=s, dtype=np.int8)  # noqa: E731
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(n.device)  # noqa: E731
    Ho, Wo = oref.conv_out_hw(H, W, R, R, pad, stride)
    x, w, e = i8(B, H, W, Ci), i8(Co, R, R, Ci), i8(B, Ho, Wo, Co)

    def guarded(op, call):
        need = n.workspace_bytes(op, [B, H, W, Ci, Co, R, R, pad, stride])
        mem = torch.full((need + GUARD,), 0x5A, dtype=torch.uint8, device=n.device)
        n._ws = mem[:need]
        out = call()
        assert n._ws.data_ptr() == mem.data_ptr()                 # (the workspace was not replaced by a larger one)
        assert bool((mem[need:] == 0x5A).all()), "bytes behind the workspace were written"
        return out

    y, s_y, b_y = guarded(OP_CONV_FWD, lambda: n.conv_fwd(T(x), n.scalar(-7), T(w), n.scalar(-9), pad=pad, relu=True,
                                                          stride=stride))
    wy, s, b = oref.conv_fwd(x, -7, w, -9, pad, True, stride=stride)
    assert np.array_equal(y.cpu().numpy(), wy) and (int(s_y), int(b_y)) == (s, b)
    ep, b_e = guarded(OP_CONV_DGRAD, lambda: n.conv_dgrad(T(e), T(w), (H, W), pad=pad, stride=stride))
    wd, bd = oref.conv_dgrad(e, w, (H, W), pad, None, stride=stride)
    assert np.array_equal(ep.cpu().numpy(), wd) and int(b_e) == bd
    g, b_g = guarded(OP_CONV_WGRAD, lambda: n.conv_wgrad(T(x), T(e), (R, R), pad=pad, stride=stride))
    wg, bg = oref.conv_wgrad(x, e, (R, R), pad, 5, stride=stride)
    assert np.array_equal(g.cpu().numpy(), wg) and int(b_g) == bg
    if stride == 1:
        wt = T(w)
        guarded(OP_CONV_WGRAD_UPDATE, lambda: n.conv_wgrad_update(T(x), T(e), wt, pad=pad))
        assert np.array_equal(wt.cpu().numpy(), oref.sgd_update(w, wg))
    n.check()
    n.close()
