"""niti_int_xent at the edges of its forms: rows kept in registers or re-read (64 bytes, 1024 packed logits), one or
several rows per warp, one block, and both launch widths; labels outside the row stay zeros beside good rows."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s_a", [-8, -5, 17])
@pytest.mark.parametrize("B,N", [(1, 1), (8, 2), (9, 63), (5, 65), (40, 1024), (40, 1028), (1185, 68), (2369, 64), (4737, 72),
                                 (2400, 33), (4800, 5)])
def test_int_xent_edges(oref, s_a, B, N):
    from paper_2009_13108_b200 import Niti
    n = Niti(0)
    rng = np.random.default_rng(B * 7 + N + s_a)
    a = rng.integers(-127, 128, size=(B, N)).astype(np.int8)
    a[B // 2] = np.clip(a[B // 2] // 32, -2, 2)
    labels = rng.integers(0, N, size=B).astype(np.int32)
    labels[0], labels[-1] = 0, N - 1
    want, b, hits = oref.int_xent(a, s_a, labels, 0)
    e, b_e, n_correct = n.int_xent(torch.from_numpy(a).cuda(), n.scalar(s_a), torch.from_numpy(labels).cuda())
    assert np.array_equal(e.cpu().numpy(), want)
    assert (int(b_e), int(n_correct)) == (b, hits)
    n.check()
    n.close()
