"""Launches overlap the tail of the one before them; the order of their memory accesses stays the stream's.  A chain in
which every call reads what the one before it wrote (weights updated in place, dirty workspaces, scratch of odd size that
is cleared in between) gives the same bytes as with a synchronisation after every call."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _chain(n, sync, M, K, N, steps=12):
    g = torch.Generator(device="cpu").manual_seed(M + K + N)
    r = lambda *s: torch.randint(-127, 128, s, dtype=torch.int8, generator=g).cuda()
    x, w, w2, labels = r(M, K), r(N, K), r(10, N), torch.randint(0, 10, (M,), dtype=torch.int32, generator=g).cuda()
    sx, sw = n.scalar(-7), n.scalar(-9)
    img, f = r(4, 20, 20, 32), r(32, 3, 3, 32)
    done = torch.cuda.synchronize if sync else (lambda: None)
    for _ in range(steps):
        h, sh, _ = n.linear_fwd(x, sx, w, sw, relu=True)
        done()
        z, sz, _ = n.linear_fwd(h, sh, w2, sw)
        done()
        e, _, _ = n.int_xent(z, n.scalar(-6), labels)
        done()
        eh = torch.empty_like(h)
        n.linear_bwd_update(h, e, w2, relu_mask_src=h, e_prev=eh)
        done()
        ex = torch.empty_like(x)
        n.linear_bwd_update(x, eh, w, relu_mask_src=x, e_prev=ex)
        done()
        y, _, _ = n.conv_fwd(img, sx, f, sw, relu=True, pad=1)
        done()
        n.conv_wgrad_update(img, y, f, pad=1)
        done()
        x = ex
    return [t.cpu() for t in (x, w, w2, f, z)]


@pytest.mark.parametrize("M,K,N", [(64, 784, 256), (300, 1029, 515), (512, 4096, 96)])
def test_overlapped_chain_is_ordered(M, K, N):
    from paper_2009_13108_b200 import Niti
    n = Niti(0)
    want = _chain(n, True, M, K, N)
    for _ in range(3):
        got = _chain(n, False, M, K, N)
        assert all(torch.equal(a, b) for a, b in zip(want, got))
    n.check()
    n.close()
