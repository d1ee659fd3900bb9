"""The largest matrices that the FP64 elimination's 32-column panels take (their shared memory ends at
855 rows): the mixed path with gj_panel = 32, which runs k_gj for flagged matrices beyond the list,
against gj_panel = 8."""
import pytest
import torch

from synth import make_system, make_walkers

pytestmark = pytest.mark.gpu
dev = torch.device("cuda", 0)


@pytest.mark.parametrize("n", [852, 853, 855])
def test_widest_panel_at_its_largest_matrix(n):
    from paper_1209_6630_gb300 import QmcSystem
    heavy = (2 * n) // 9
    s = make_system(heavy, 0, 0, 2 * n - 6 * heavy, seed=100 + n)
    assert s.n_up == n
    q = QmcSystem(s, 0)
    R = torch.from_numpy(make_walkers(s, 2, first=98000)).to(dev)
    q.set_tiles(gj_panel=8)
    ref = q.eval(R, precision="mixed")
    q.set_tiles(gj_panel=32)
    got = q.eval(R, precision="mixed")
    assert (got["status"] == 0).all() and torch.equal(got["sign"], ref["sign"])
    assert (got["logpsi"] - ref["logpsi"]).abs().max().item() < 1e-6
