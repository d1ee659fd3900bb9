"""The energy kernel with a walker on 1, 2, 4 or 8 CTAs, and the Jastrow pairs
evaluated once for both electrons: walker counts on both sides of each split,
odd and even electron counts, more electrons than a block has threads, against
the oracle at the FP64 path's bars (1e-10 relative).  Two electrons at the same
point stay a status, not an error."""
import numpy as np
import pytest
import torch

from oracle import Oracle
from synth import config_system, make_system, make_walkers, tiny_system

pytestmark = pytest.mark.gpu
dev = torch.device("cuda", 0)
SYSTEMS = {"tiny": lambda: tiny_system("h2o_like"), "119e": lambda: make_system(9, 3, 3, 20, seed=21),
           "434e": lambda: config_system("434e")}


def _jas(s):
    return dict(a_par=0.25, a_anti=0.5, b_ee=1.1, a_en=np.linspace(0.4, 1.2, s.n_atom),
                b_en=np.linspace(1.5, 2.5, s.n_atom))


@pytest.mark.parametrize("key,W", [("tiny", 1), ("tiny", 700), ("119e", 2), ("119e", 76), ("119e", 152), ("119e", 700),
                                   ("434e", 1), ("434e", 77), ("434e", 153)])
@pytest.mark.parametrize("jastrow", [False, True])
def test_energy_split_vs_oracle(key, W, jastrow):
    from paper_1209_6630_gb300 import QmcSystem
    s = SYSTEMS[key]()
    q = QmcSystem(s, 0)
    jas = _jas(s) if jastrow else None
    if jastrow:
        q.set_jastrow(jas)
    R = make_walkers(s, W, first=81000)
    sample = np.unique(np.linspace(0, W - 1, 5).astype(int))
    ref = Oracle(s, jastrow=jas).eval(R[sample], nthreads=8)
    for precision in ("f64", "mixed"):
        got = {k: v.cpu().numpy()[sample] for k, v in q.eval(torch.from_numpy(R).to(dev), precision=precision).items()}
        np.testing.assert_array_equal(got["status"], ref["status"])
        bar = 1e-10 if precision == "f64" else 1e-5
        scale = np.abs(ref["e_parts"]).max(1)
        assert (np.abs(got["e_loc"] - ref["e_loc"]) / scale).max() < bar
        assert (np.abs(got["e_parts"] - ref["e_parts"]).max(1) / scale).max() < bar
        assert np.abs(got["logpsi"] - ref["logpsi"]).max() < (1e-9 if precision == "f64" else 1e-6)
        d = np.abs(got["drift"] - ref["drift"]).max((1, 2)) / np.abs(ref["drift"]).max((1, 2))
        assert d.max() < bar


@pytest.mark.parametrize("jastrow", [False, True])
def test_coincident_and_distant_electrons(jastrow):
    from paper_1209_6630_gb300 import QmcSystem
    s = tiny_system("mini_chain")
    q = QmcSystem(s, 0)
    jas = _jas(s) if jastrow else None
    if jastrow:
        q.set_jastrow(jas)
    R = make_walkers(s, 3, first=82000)
    R[1, s.n_up] = R[1, 0]                       # an up and a down electron at one point
    ref = Oracle(s, jastrow=jas).eval(R, nthreads=1)
    for precision in ("f64", "mixed"):
        got = q.eval(torch.from_numpy(R).to(dev), precision=precision)
        np.testing.assert_array_equal(got["status"].cpu().numpy(), ref["status"])
        assert np.abs(got["logpsi"].cpu().numpy() - ref["logpsi"]).max() < 1e-6
