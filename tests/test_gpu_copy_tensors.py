"""niti_copy_tensors: whole and partial 32 KB blocks, byte tails, more tensors than one launch takes."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[1], [15, 16, 17], [32768, 32767, 32769, 100000], [1 << 20] * 3 + [5] * 40])
def test_copy_tensors(sizes):
    from paper_2009_13108_b200 import Niti
    n = Niti(0)
    src = [torch.randint(-128, 128, (s,), dtype=torch.int8, device=n.device) for s in sizes]
    pad = [torch.full((s + 64,), 7, dtype=torch.int8, device=n.device) for s in sizes]
    n.copy_tensors([p[:s] for p, s in zip(pad, sizes)], src)
    for p, s, x in zip(pad, sizes, src):
        assert torch.equal(p[:s], x) and bool((p[s:] == 7).all())
    n.close()
