"""The one-launch kernel of small fully connected multiplies against the CPU oracle (bit-exact): region edges,
contraction remainders and chunks, operand rows of every alignment, both multiplies of a backward call, the update."""
import numpy as np
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


@pytest.mark.parametrize("M,N,K", [
    (1, 1, 1), (31, 33, 65), (33, 10, 257), (64, 31, 64), (65, 97, 130),       # remainders of tiles and steps
    (7, 129, 36), (40, 50, 72), (96, 64, 1023),                                # row pitches of 4, 8 and odd bytes
    (16, 48, 20000), (128, 10, 6000), (4096, 10, 70), (5000, 31, 33),          # contractions staged in chunks
    (33, 20, 511), (500, 300, 99), (64, 33, 3137), (96, 512, 4000),            # rows at any byte, on both sides of the line
    (3000, 300, 200), (300, 3000, 200), (64, 1400, 2200)])                     # near the size limit
def test_small_multiplies(niti, oref, M, N, K):
    rng = np.random.default_rng(M + 3 * N + 7 * K)
    i8 = lambda *s: rng.integers(-127, 128, size=s, dtype=np.int8)  # noqa: E731
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(niti.device)  # noqa: E731
    a, w, e = np.maximum(i8(M, K), 0), i8(N, K), i8(M, N)
    for relu, mode in ((True, 0), (False, 1)):
        want, s, b = oref.linear_fwd(a, -7, w, -9, relu, mode)
        out, s_out, b_out = niti.linear_fwd(T(a), niti.scalar(-7), T(w), niti.scalar(-9), relu=relu, round_mode=mode)
        assert np.array_equal(out.cpu().numpy(), want) and (int(s_out), int(b_out)) == (s, b)
    we, wg, be, bg = oref.linear_bwd(a, e, w, True, a, 5)
    ep, g, b_e, b_g = niti.linear_bwd(T(a), T(e), T(w), True, T(a))
    assert np.array_equal(ep.cpu().numpy(), we) and np.array_equal(g.cpu().numpy(), wg)
    assert (int(b_e), int(b_g)) == (be, bg)
    wt = T(w)
    eu, b_e, b_g = niti.linear_bwd_update(T(a), T(e), wt, True, T(a))
    assert np.array_equal(eu.cpu().numpy(), we) and np.array_equal(wt.cpu().numpy(), oref.sgd_update(w, wg))
    niti.linear_bwd_update(T(a), T(e), wt, need_e_prev=False)
    assert np.array_equal(wt.cpu().numpy(), oref.sgd_update(oref.sgd_update(w, wg), wg))


@pytest.mark.parametrize("M,N,K", [(64, 256, 784), (256, 10, 512), (300, 100, 90)])
def test_error_in_place_of_the_input(niti, oref, M, N, K):
    """niti_linear_bwd with e_prev in the storage of a: the weight gradient still sees the input."""
    rng = np.random.default_rng(M + N + K)
    i8 = lambda *s: rng.integers(-127, 128, size=s, dtype=np.int8)  # noqa: E731
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(niti.device)  # noqa: E731
    a, w, e = i8(M, K), i8(N, K), i8(M, N)
    we, wg, be, bg = oref.linear_bwd(a, e, w, True, None, 5)
    for _ in range(5):
        at = T(a)
        ep, g, b_e, b_g = niti.linear_bwd(at, T(e), T(w), True, e_prev=at)
        assert np.array_equal(ep.cpu().numpy(), we) and np.array_equal(g.cpu().numpy(), wg)
        assert (int(b_e), int(b_g)) == (be, bg)
