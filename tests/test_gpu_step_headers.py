"""Calls between and after steps take zeroed headers, whatever came before them on the workspace: a captured step that has not
been replayed yet, replays of a step of another network, a capture of their own; and they clear none in front of every call."""
import pytest
import torch

from synth.workloads import config_net, make_net_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture
def niti():
    from paper_2009_13108_b200 import Niti
    n = Niti(0)
    n.reserve_workspace(128 << 20)
    yield n
    n.check()
    n.close()


class Multiply:
    """A multiply of several waves of `value`s; its bit-width is exact, so that a maximum left in the header shows."""

    def __init__(self, n, M=4096, N=4096, K=256):
        self.n, self.K = n, K
        self.a, self.w = torch.empty((M, K), dtype=torch.int8, device=n.device), torch.ones((N, K), dtype=torch.int8, device=n.device)
        self.out, self.s, self.b, self.sa = torch.empty((M, N), dtype=torch.int8, device=n.device), n.scalar(), n.scalar(), n.scalar(-7)

    def call(self):
        self.n.linear_fwd(self.a, self.sa, self.w, self.sa, out=self.out, s_out=self.s, b_out=self.b)

    def check(self):
        top = abs(int(self.a[0, 0])) * self.K
        b = top.bit_length()
        assert int(self.b) == b and bool((self.out == top >> max(0, b - 7)).all())

    def __call__(self, value):
        self.a.fill_(value)
        self.call()
        self.check()


def _trainer(n, cfg, batch):
    from paper_2009_13108_b200 import NitiTrainer
    net = config_net(cfg, batch=batch)
    x, labels, weights = make_net_inputs(net)
    tr = NitiTrainer(n, net, weights)
    tr.load_batch(x, labels)
    tr.snapshot_weights()
    return tr


def _capture(n, fn):
    stream, graph = torch.cuda.Stream(device=n.device), torch.cuda.CUDAGraph()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(graph, stream=stream):
        fn()
    return graph


def test_calls_after_a_captured_begin(niti):
    m, other = Multiply(niti), Multiply(niti)
    m(1)
    niti.begin_step()
    m(1)
    m(127)
    other.a.fill_(1)

    def step():
        niti.begin_step()
        other.call()
    graph = _capture(niti, step)
    for value in (1, 3, 1):                       # (nothing has been replayed: the recorded clear has cleared nothing)
        m(value)
    graph.replay()
    other.check()
    m(1)


def test_captured_calls_after_a_begin_in_front_of_the_capture(niti):
    m, other = Multiply(niti), Multiply(niti)
    m(1)
    niti.begin_step()
    m(1)
    other.a.fill_(127)
    graph = _capture(niti, other.call)
    for value in (127, 1, 5):
        other.a.fill_(value)
        graph.replay()
        other.check()
        m(1)


def test_calls_between_the_steps_of_two_networks(niti):
    big, small, m = _trainer(niti, 2, 64), _trainer(niti, 0, 64), Multiply(niti)
    big.step()
    replay = big.capture(with_reset=True)
    replay()
    want = [t.clone() for t in big.weights]
    small.step()
    replay()
    for _ in range(40):
        m(1)
    small.reset_weights()
    small.step()
    replay()
    m(1)
    assert all(torch.equal(t, u) for t, u in zip(big.weights, want))


@pytest.mark.parametrize("calls", [1, 64])
def test_no_clears_after_a_step(niti, calls):
    """After a step, whether it used all headers or not, at most the first call clears anything."""
    a, w, sa = torch.ones((64, 64), dtype=torch.int8, device=niti.device), torch.ones((64, 64), dtype=torch.int8, device=niti.device), niti.scalar(-7)

    def launches():
        l0 = niti.launch_count()
        out, _, b = niti.linear_fwd(a, sa, w, sa)
        assert int(b) == 7 and bool((out == 64).all())
        return niti.launch_count() - l0
    niti.begin_step()
    for _ in range(calls):
        launches()
    niti.end_step()
    launches()
    assert [launches() for _ in range(70)] == [1] * 70


def test_no_clears_after_a_training_step(niti):
    tr = _trainer(niti, 0, 64)
    tr.step()
    a, w, sa = torch.ones((64, 64), dtype=torch.int8, device=niti.device), torch.ones((64, 64), dtype=torch.int8, device=niti.device), niti.scalar(-7)
    counts = []
    for _ in range(80):
        l0 = niti.launch_count()
        niti.linear_fwd(a, sa, w, sa)
        counts.append(niti.launch_count() - l0)
    assert counts[1:] == [1] * 79
