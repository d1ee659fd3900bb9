"""The FP64 elimination spread over many CTAs against one CTA per matrix (k_gj) at the sizes where a call
always spreads, and with two spins of different sizes: bit for bit.  k_gj is reached through the
recomputation pass of QMC_PREC_F64_TCA4 with a threshold that flags every matrix, on the same FP64 C1."""
import pytest
import torch

from synth import make_system, make_walkers

pytestmark = pytest.mark.gpu
dev = torch.device("cuda", 0)


@pytest.mark.parametrize("n,panel", [(60, 16), (217, 32), (512, 16), (545, 8), (640, 16), (866, 8)])
def test_spread_equals_one_cta_per_matrix(n, panel):
    from paper_1209_6630_gb300 import QmcSystem
    heavy = max(2, (2 * n) // 9)
    s = make_system(heavy, 0, 0, 2 * n - 1 - 6 * heavy, seed=500 + n)      # n and n - 1 electrons
    assert (s.n_up, s.n_dn) == (n, n - 1)
    q = QmcSystem(s, 0)
    q.set_tiles(gj_panel=panel, f64_kappa_max=1e-300)
    R = torch.from_numpy(make_walkers(s, 2, first=96000)).to(dev)
    few = q.eval(R, precision="f64", want_dinv=True)
    one = q.eval(R, precision="f64_tca4", want_dinv=True)
    assert (few["status"] == 0).all()
    for k in ("logabs", "sign", "dinv"):
        assert torch.equal(few[k], one[k]), k
