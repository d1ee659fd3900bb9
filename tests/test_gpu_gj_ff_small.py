"""The float-float elimination of small matrices in blocks of 64 threads (more than 304 matrices of up to 64
rows) against blocks of 256 (fewer): the same arithmetic, so one walker repeated gives the same bits; and
against the FP64 elimination of the same C1 within the mixed path's 1e-6."""
import pytest
import torch

from synth import make_system, make_walkers, tiny_system

pytestmark = pytest.mark.gpu
dev = torch.device("cuda", 0)


@pytest.mark.parametrize("n", [5, 8, 17, 31, 33, 48, 63, 64])
@pytest.mark.parametrize("panel", [8, 16, 32])
def test_blocks_of_64_equal_blocks_of_256(n, panel):
    from paper_1209_6630_gb300 import QmcSystem, det_inverse
    heavy = max(2, 2 * n // 9)
    s = tiny_system("h2o_like") if n == 5 else make_system(heavy, 0, 0, 2 * n - 6 * heavy, seed=700 + n)
    assert s.n_up == n
    q = QmcSystem(s, 0)
    q.set_tiles(a4_mode="float_float", gj_panel=panel)
    R = torch.from_numpy(make_walkers(s, 1, first=93000)).to(dev)
    few = q.eval(R.expand(128, -1, -1).contiguous(), precision="mixed", want_dinv=True)
    many = q.eval(R.expand(384, -1, -1).contiguous(), precision="mixed", want_dinv=True)
    assert (few["status"] == 0).all()
    for k in ("logabs", "dinv", "sign"):
        assert (many[k] == few[k][:1]).all() and (few[k] == few[k][:1]).all()
    C = q.slater(R, precision="mixed")[0][:, 0].contiguous()
    logabs, _, D, _ = det_inverse(C.clone())
    assert (few["logabs"][0, 0] - logabs[0]).abs().item() < 1e-6
    E = few["dinv"][0, : n * n].reshape(n, n).mT @ C[0] - torch.eye(n, dtype=torch.float64, device=dev)
    assert E.abs().max().item() < 1e-6
