"""Forms of the fused rounding that the layers of the networks do not reach (bit-exact against the CPU oracle's rounding):
binary points above 24, and row-batched first layers whose rows are not whole 32-byte chunks."""
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


@pytest.mark.parametrize("engine,N,K", [(2, 1280, 4096), (2, 1250, 4100), (0, 512, 1024)])   # many tiles, odd rows, one wave
def test_binary_points_above_24(niti, oref, engine, N, K):
    M = 4096
    g = torch.Generator(device=niti.device)
    g.manual_seed(N)
    a = torch.full((M, K), 127, dtype=torch.int8, device=niti.device)
    a[::3] = torch.randint(-127, 128, a[::3].shape, generator=g, dtype=torch.int8, device=niti.device)
    e = torch.full((M, N), 127, dtype=torch.int8, device=niti.device)
    e[:, 1::2] = torch.randint(-127, 128, e[:, 1::2].shape, generator=g, dtype=torch.int8, device=niti.device)
    e[:, 2::4] = -127
    w = torch.randint(-127, 128, (N, K), generator=g, dtype=torch.int8, device=niti.device)
    acc = (e.double().T @ a.double()).cpu().numpy().astype(np.int32)       # (sums below 2^27: exact)
    niti.set_engine(engine)
    try:
        for mode in (0, 1):
            want, b, _ = oref.shift_round(acc, 1, mode)
            assert b > 25
            _, got, _, b_g = niti.linear_bwd(a, e, w, False, m_u=1, round_mode=mode)
            assert int(b_g) == b and np.array_equal(got.cpu().numpy(), want)
            wt = w.clone()
            niti.linear_bwd_update(a, e, wt, need_e_prev=False, m_u=1, round_mode=mode)
            assert np.array_equal(wt.cpu().numpy(), oref.sgd_update(w.cpu().numpy(), want))
    finally:
        niti.set_engine(0)


@pytest.mark.parametrize("cout,cin", [(10, 3), (40, 1), (97, 3)])
def test_row_batched_first_layers_with_odd_rows(niti, oref, cout, cin):
    rng = np.random.default_rng(cout)
    x = rng.integers(-127, 128, size=(48, 60, 64, cin), dtype=np.int8)
    w = rng.integers(-127, 128, size=(cout, 3, 3, cin), dtype=np.int8)
    for relu, mode in ((True, 0), (False, 1)):
        want, s, b = oref.conv_fwd(x, -7, w, -9, 1, relu, mode)
        y, s_y, b_y = niti.conv_fwd(torch.from_numpy(x).to(niti.device), niti.scalar(-7), torch.from_numpy(w).to(niti.device),
                                    niti.scalar(-9), pad=1, relu=relu, round_mode=mode)
        assert np.array_equal(y.cpu().numpy(), want) and (int(s_y), int(b_y)) == (s, b)


@pytest.mark.parametrize("M,N", [(1024, 1024), (500, 736)])
def test_outputs_in_the_storage_of_an_operand(niti, oref, M, N):
    """One-wave multiplies read all operands before they store: outputs may replace an operand or the gate."""
    rng = np.random.default_rng(M)
    i8 = lambda *s: rng.integers(-127, 128, size=s, dtype=np.int8)  # noqa: E731
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(niti.device)  # noqa: E731
    a, w, e = np.maximum(i8(M, N), 0), i8(N, N), i8(M, N)
    want, s, b = oref.linear_fwd(a, -7, w, -9, True)
    we, wg, be, bg = oref.linear_bwd(a, e, w, True, a, 5)
    for _ in range(3):
        at = T(a)
        _, s_out, b_out = niti.linear_fwd(at, niti.scalar(-7), T(w), niti.scalar(-9), out=at, relu=True)
        assert np.array_equal(at.cpu().numpy(), want) and (int(s_out), int(b_out)) == (s, b)
        at = T(a)
        _, g, b_e, b_g = niti.linear_bwd(at, T(e), T(w), True, at, e_prev=at)
        assert np.array_equal(at.cpu().numpy(), we) and np.array_equal(g.cpu().numpy(), wg)
        assert (int(b_e), int(b_g)) == (be, bg)


def test_headers_of_an_own_workspace(oref):
    """Calls outside a step leave a clean header for the next one, whatever the path of either, a captured call (whose replays
    repeat) and a step between them, and a buffer put in the workspace's place."""
    from paper_2009_13108_b200 import Niti
    n = Niti(0)
    rng = np.random.default_rng(5)
    i8 = lambda *s: rng.integers(-127, 128, size=s, dtype=np.int8)  # noqa: E731
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(n.device)  # noqa: E731
    x, w, e, lab = i8(4, 20, 20, 64), i8(64, 3, 3, 64), i8(4, 20, 20, 64), rng.integers(0, 64, 33).astype(np.int32)
    a, wl = i8(33, 70), i8(64, 70)
    xt, wt, et, at, wlt, labt = T(x), T(w), T(e), T(a), T(wl), T(lab)
    sx, sw = n.scalar(-7), n.scalar(-9)
    want = [oref.conv_fwd(x, -7, w, -9, 1, True)[0], oref.conv_dgrad(e, w, (20, 20), 1, None)[0], oref.conv_wgrad(x, e, (3, 3), 1, 5)[0],
            oref.linear_fwd(a, -7, wl, -9, False)[0]]
    want.append(oref.int_xent(want[3], -3, lab)[0])
    logits, s3 = T(want[3]), n.scalar(-3)
    calls = [lambda: n.conv_fwd(xt, sx, wt, sw, relu=True)[0], lambda: n.conv_dgrad(et, wt, (20, 20))[0],
             lambda: n.conv_wgrad(xt, et, (3, 3))[0], lambda: n.linear_fwd(at, sx, wlt, sw)[0],
             lambda: n.int_xent(logits, s3, labt)[0]]

    def check(order):
        for k in order:
            assert np.array_equal(calls[k]().cpu().numpy(), want[k]), k

    def all_pairs():
        for engine in (0, 6, 2, 4, 1):                       # (one wave, leaving CTAs on a header of their own, single CTAs, ...)
            n.set_engine(engine)
            check([i for p in range(5) for q in range(5) for i in (p, q)])
        n.set_engine(0)

    all_pairs()
    launches = []
    for _ in range(3):
        l0 = n.launch_count()
        calls[3]()
        launches.append(n.launch_count() - l0)
    assert launches == [1, 1, 1]                             # no clear of its own
    y = torch.empty((4, 20, 20, 64), dtype=torch.int8, device=n.device)
    st = torch.cuda.Stream(device=n.device)
    st.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    s_y, b_y = n.scalar(), n.scalar()
    with torch.cuda.graph(graph, stream=st):
        n.conv_fwd(xt, sx, wt, sw, y=y, s_y=s_y, b_y=b_y, relu=True)
    for k in (3, 0, 4, 2):
        y.zero_()
        graph.replay()
        graph.replay()
        check([k])
        assert np.array_equal(y.cpu().numpy(), want[0])
    n.begin_step()
    check(list(range(5)) * 14)                               # (70 calls: past the step's headers)
    n._ck(n.lib.niti_begin_step(n.h, None, None, 0))
    check(range(5))
    n._ws = torch.full((n._ws.numel(),), 0x5A, dtype=torch.uint8, device=n.device)
    check(list(range(5)) * 2)
    n.reserve_workspace(2 * n._ws.numel())
    all_pairs()
    n.check()
    n.close()


@pytest.mark.parametrize("B,S,Ci,Co,R,pad,stride,resident", [
    (60, 32, 72, 40, 1, 0, 1, True), (64, 61, 64, 100, 3, 1, 2, True), (15, 64, 130, 64, 1, 0, 1, True),
    # windows of few channels: 444 row tiles and more, and 439, which are copied tile by tile
    (70, 119, 3, 96, 11, 2, 4, True), (16, 60, 3, 40, 5, 2, 1, True), (60, 66, 1, 33, 7, 2, 2, True), (20, 111, 3, 96, 11, 2, 2, False)])
def test_weights_resident_over_many_tiles(niti, oref, B, S, Ci, Co, R, pad, stride, resident):
    """One column tile and three row tiles per CTA or more: short chunks, odd rows, windows, errors."""
    rng = np.random.default_rng(S + Ci)
    i8 = lambda *s: rng.integers(-127, 128, size=s, dtype=np.int8)  # noqa: E731
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(niti.device)  # noqa: E731
    x, w = i8(B, S, S, Ci), i8(Co, R, R, Ci)
    want, s, b = oref.conv_fwd(x, -7, w, -9, pad, True, stride=stride)
    before = niti.tc_resident_launch_count()
    y, s_y, b_y = niti.conv_fwd(T(x), niti.scalar(-7), T(w), niti.scalar(-9), pad=pad, relu=True, stride=stride)
    assert (niti.tc_resident_launch_count() > before) == resident
    assert np.array_equal(y.cpu().numpy(), want) and (int(s_y), int(b_y)) == (s, b)
    if stride == 1 and Ci >= 32:
        e = i8(*want.shape)
        wd, bd = oref.conv_dgrad(e, w, (S, S), pad, x)
        before = niti.tc_resident_launch_count()
        ep, b_e = niti.conv_dgrad(T(e), T(w), (S, S), relu_mask_src=T(x), pad=pad)
        assert niti.tc_resident_launch_count() > before
        assert np.array_equal(ep.cpu().numpy(), wd) and int(b_e) == bd


def test_fully_connected_weights_resident(niti, oref):
    rng = np.random.default_rng(3)
    a, w = rng.integers(-127, 128, size=(60000, 130), dtype=np.int8), rng.integers(-127, 128, size=(200, 130), dtype=np.int8)
    want, s, b = oref.linear_fwd(a, -7, w, -9, False)
    before = niti.tc_resident_launch_count()
    out, s_out, b_out = niti.linear_fwd(torch.from_numpy(a).to(niti.device), niti.scalar(-7), torch.from_numpy(w).to(niti.device),
                                        niti.scalar(-9))
    assert niti.tc_resident_launch_count() > before
    assert np.array_equal(out.cpu().numpy(), want) and (int(s_out), int(b_out)) == (s, b)
