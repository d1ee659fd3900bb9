"""A workspace between the least and the queried size counts in full: the Slater matrices, which need more
of it than an evaluation, come in one chunk of walkers where it has the room (the FP32 sums of the
gradients go with the walkers that share a tile, so one chunk is one set of bits)."""
import pytest
import torch

from synth import config_system, make_walkers

pytestmark = pytest.mark.gpu
dev = torch.device("cuda", 0)


@pytest.mark.parametrize("W", [129, 200])
def test_slater_below_the_queried_size(W):
    from paper_1209_6630_gb300 import QmcSystem
    s = config_system("434e")
    q = QmcSystem(s, 0)
    R = torch.from_numpy(make_walkers(s, W, first=97000)).to(dev)
    need = q.workspace_size(W, "mixed")
    whole = q.slater(R, precision="mixed", ws=torch.empty(4 * need, dtype=torch.uint8, device=dev))
    below = q.slater(R, precision="mixed", ws=torch.empty(need - 256, dtype=torch.uint8, device=dev))
    for a, b in zip(whole, below):
        assert torch.equal(a, b)
