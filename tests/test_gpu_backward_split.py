"""The FP64 adjoint with its (walker, electron) pairs split over a cluster of
1, 2, 4 or 8 CTAs: walker counts on both sides of each split, an open shell, a
walker with weight zero, and atoms of up to 32 AOs (s, p, d, f shells), against
the oracle.  Both sides sum the same terms in FP64 in different orders: at most
8192 terms, so 8192 x 2^-53 = 1e-12 of the largest sum of magnitudes; those sums
are within 100 of the gradient's scale here, hence 1e-10 of it."""
import numpy as np
import pytest
import torch

from helpers import one_atom_system
from oracle import Oracle
from synth import config_system, make_system, make_walkers

pytestmark = pytest.mark.gpu
dev = torch.device("cuda", 0)


def _check(s, R, g):
    from paper_1209_6630_gb300 import QmcSystem
    q = QmcSystem(s, 0)
    Rd = torch.from_numpy(R).to(dev)
    dinv = q.eval(Rd, precision="f64", want_dinv=True)["dinv"]
    got = q.backward(Rd, dinv, torch.from_numpy(g).to(dev), precision="f64")
    for a, b in zip(got, Oracle(s).logpsi_grad(R, g, nthreads=8)):
        if b.size:
            assert np.abs(a.cpu().numpy() - b).max() <= 1e-10 * np.abs(b).max()


@pytest.mark.parametrize("W", [1, 6, 7, 13, 26, 40])
@pytest.mark.parametrize("open_shell", [False, True])
def test_backward_split_vs_oracle(W, open_shell):
    s = make_system(9, 3, 3, 20, seed=21) if open_shell else config_system("158e")
    g = np.random.default_rng(W).normal(size=W)
    if W > 1:
        g[W // 2] = 0.0
    _check(s, make_walkers(s, W, first=61000), g)


def test_backward_split_wide_atom():
    rng = np.random.default_rng(3)
    shells = [(L, [0.5 + 0.2 * L, 1.7], [0.8, 0.5]) for L in (0, 1, 2, 3)] + [(0, [0.3], [1.0])]
    n_ao = 1 + 3 + 6 + 10 + 1
    s = one_atom_system(5, shells, 3, 2, rng.normal(size=(n_ao, 3)), rng.normal(size=(n_ao, 2)))
    R = rng.normal(size=(1500, 5, 3))
    _check(s, R, rng.normal(size=1500))
