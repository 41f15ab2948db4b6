"""niti_int_xent at the edges of its forms: rows kept in registers or re-read (64 bytes, 1024 packed logits), one or
several rows per warp, one block, and all launch widths; both rounding modes and the ends of the exponent's ranges; labels
outside the row give zeros there and nothing to the rest."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

BAD_LABEL = 8                       # NITI_DEV_BAD_LABEL


@pytest.fixture(scope="module")
def niti():
    from paper_2009_13108_b200 import Niti
    n = Niti(0)
    yield n
    n.check()
    n.close()


def _case(B, N, s_a):
    rng = np.random.default_rng(B * 7 + N + s_a + 22)
    a = rng.integers(-127, 128, size=(B, N)).astype(np.int8)
    a[B // 2] = np.clip(a[B // 2] // 32, -2, 2)
    labels = rng.integers(0, N, size=B).astype(np.int32)
    labels[0], labels[-1] = 0, N - 1
    return a, labels


@pytest.mark.parametrize("round_mode", [0, 1])
@pytest.mark.parametrize("s_a", [-22, -8, -7, -6, -5, 14, 15, 17, 24])
@pytest.mark.parametrize("B,N", [(1, 1), (8, 2), (9, 63), (5, 65), (40, 1024), (40, 1028), (1185, 68), (2369, 64), (4737, 72),
                                 (2400, 33), (4800, 5)])
def test_int_xent_edges(niti, oref, s_a, B, N, round_mode):
    n = niti
    a, labels = _case(B, N, s_a)
    want, b, hits = oref.int_xent(a, s_a, labels, round_mode)
    e, b_e, n_correct = n.int_xent(torch.from_numpy(a).cuda(), n.scalar(s_a), torch.from_numpy(labels).cuda(), round_mode=round_mode)
    assert np.array_equal(e.cpu().numpy(), want)
    assert (int(b_e), int(n_correct)) == (b, hits)
    n.check()


@pytest.mark.parametrize("s_a", [-8, -5])
@pytest.mark.parametrize("B,N", [(9, 63), (40, 1024), (40, 1028), (12, 70), (4737, 72), (2400, 33)])
def test_labels_outside_the_row(niti, oref, s_a, B, N):
    from paper_2009_13108_b200 import NitiError
    n = niti
    a, labels = _case(B, N, s_a)
    bad = np.array([1, B // 3, B // 2, B - 2])
    labels[bad] = [-1, N, -(1 << 31), (1 << 31) - 1]
    good = np.setdiff1d(np.arange(B), bad)
    want, b, hits = oref.int_xent(a[good], s_a, labels[good], 0)
    e, b_e, n_correct = n.int_xent(torch.from_numpy(a).cuda(), n.scalar(s_a), torch.from_numpy(labels).cuda(),
                                   e=torch.full((B, N), 99, dtype=torch.int8, device="cuda"))
    got = e.cpu().numpy()
    assert np.array_equal(got[good], want) and not got[bad].any()
    assert (int(b_e), int(n_correct)) == (b, hits)
    with pytest.raises(NitiError, match=hex(BAD_LABEL)):
        n.check()
    n.check()                       # (reported once)
