"""The largest matrices that the eliminations take.  FP64 with 32-column panels (their shared memory ends at
855 rows): the mixed path with gj_panel = 32, which runs k_gj for flagged matrices beyond the list,
against gj_panel = 8.  Tensor-core a4: 896 rows, a thread each in the panel."""
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


def test_tensor_a4_at_its_largest_matrix():
    from paper_1209_6630_gb300 import QmcSystem
    from paper_1209_6630_gb300._lib import QmcError
    for n in (896, 897):
        heavy = (2 * n) // 9
        s = make_system(heavy, 0, 0, 2 * n - 6 * heavy, seed=100 + n)
        q = QmcSystem(s, 0)
        assert s.n_up == n and q.tiles()["a4_mode"] == ("tensor" if n == 896 else "float_float")
        if n == 897:
            with pytest.raises(QmcError):
                q.set_tiles(a4_mode="tensor")
            continue
        R = torch.from_numpy(make_walkers(s, 2, first=98000)).to(dev)
        got = q.eval(R, precision="mixed")
        q.set_tiles(a4_mode="float_float")
        ref = q.eval(R, precision="mixed")
        assert (got["status"] == 0).all() and torch.equal(got["sign"], ref["sign"])
        assert (got["logpsi"] - ref["logpsi"]).abs().max().item() < 1e-6
