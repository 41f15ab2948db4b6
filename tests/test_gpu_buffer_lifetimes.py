"""A workspace or tap cache that is replaced by a larger one is not given back while something still uses it: replays of a step
captured with it, or calls enqueued on another stream than the one it was allocated on."""
import pytest
import torch

from synth.workloads import config_net, make_net_inputs

pytestmark = pytest.mark.gpu


def _patterns(sizes):
    """Tensors of the sizes given, which the allocator takes from blocks that were freed."""
    return [torch.full((size,), 0x5A, dtype=torch.uint8, device="cuda") for size in sizes for _ in range(3)]


def _trainer(n, batch):
    from paper_2009_13108_b200 import NitiTrainer
    net = config_net(2, batch=batch)
    x, labels, weights = make_net_inputs(net)
    tr = NitiTrainer(n, net, weights)
    tr.load_batch(x, labels)
    tr.snapshot_weights()
    return tr


def test_a_captured_step_keeps_its_buffers():
    from paper_2009_13108_b200 import Niti
    n = Niti(0)
    tr = _trainer(n, 64)
    tr.step()
    replay = tr.capture(with_reset=True)
    replay()
    torch.cuda.synchronize()
    want = [w.clone() for w in tr.weights]
    sizes = [n._ws.numel(), n._tap.numel()]
    bigger = _trainer(n, 200)                     # (a larger tap cache; its step needs a larger workspace)
    bigger.step()
    assert n._ws.numel() > sizes[0] and n._tap.numel() > sizes[1]
    torch.cuda.synchronize()
    held = _patterns(sizes)
    replay()
    torch.cuda.synchronize()
    assert all(bool((t == 0x5A).all()) for t in held)
    assert all(torch.equal(w, u) for w, u in zip(tr.weights, want))
    n.check()
    n.close()


def test_a_workspace_replaced_behind_calls_of_another_stream():
    from paper_2009_13108_b200 import Niti
    n = Niti(0)
    size = n._ws.numel()
    ones, sa = torch.ones((64, 64), dtype=torch.int8, device=n.device), n.scalar(-7)
    n.linear_fwd(ones, sa, ones, sa)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        torch.cuda._sleep(20_000_000)             # about 10 ms
        out, _, b = n.linear_fwd(ones, sa, ones, sa)
        n.reserve_workspace(64 << 20)
    held = _patterns([size])                      # written while the call still waits
    torch.cuda.synchronize()
    assert all(bool((t == 0x5A).all()) for t in held)
    assert int(b) == 7 and bool((out == 64).all())
    n.check()
    n.close()
