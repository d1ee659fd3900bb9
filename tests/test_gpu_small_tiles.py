"""Mixed-path products and the C-free drift with few walkers: a single tile of
1 .. 128 walkers stages only its own rows (rounded up to 8) and spreads a
row's AOs over the threads that have no row (the power of two that holds the
rows), so the walker counts here sit at the edges of both, and one past a
tile.  Against the FP64 path at the mixed path's bars; the walkers of a call
must not depend on the others beyond the grouping's rounding."""
import numpy as np
import pytest
import torch

from helpers import one_atom_system
from synth import config_system, make_system, make_walkers

pytestmark = pytest.mark.gpu
dev = torch.device("cuda", 0)
COUNTS = [1, 2, 3, 7, 8, 9, 17, 33, 63, 64, 65, 100, 127, 128, 129]


def _q(s):
    from paper_1209_6630_gb300 import QmcSystem
    return QmcSystem(s, 0)


@pytest.mark.parametrize("W", COUNTS)
@pytest.mark.parametrize("open_shell", [False, True])
def test_eval_few_walkers(W, open_shell):
    s = make_system(9, 3, 3, 20, seed=21) if open_shell else config_system("158e")
    q = _q(s)
    R = torch.from_numpy(make_walkers(s, W, first=52000)).to(dev)
    ref = q.eval(R, precision="f64")
    for mode in ("cfree", "tensor"):
        q.set_tiles(c15_mode=mode)
        got = q.eval(R, precision="mixed")
        assert torch.equal(got["status"], ref["status"])
        assert torch.equal(got["sign"], ref["sign"])
        assert (got["logpsi"] - ref["logpsi"]).abs().max().item() < 1e-6
        # E_L against the size of its terms (T and V cancel for some walkers)
        scale = ref["e_parts"].abs().amax(1)
        assert ((got["e_loc"] - ref["e_loc"]).abs() / scale).max().item() < 1e-5
        d = (got["drift"] - ref["drift"]).abs().amax((1, 2)) / ref["drift"].abs().amax((1, 2))
        assert d.max().item() < (1e-5 if mode == "cfree" else 1e-4)


@pytest.mark.parametrize("W", [1, 5, 32, 70, 129])
def test_slater_few_walkers(W):
    s = config_system("158e")
    q = _q(s)
    R = torch.from_numpy(make_walkers(s, W, first=53000)).to(dev)
    got, ref = q.slater(R, precision="mixed"), q.slater(R, precision="f64")
    for g, r in zip(got, ref):
        err = (g - r).abs().amax(-1) / r.abs().amax(-1)          # row-normwise, [W, 5, n]
        assert err[:, [0, 4]].max().item() < 1e-9
        assert err[:, 1:4].max().item() < 1e-5


def test_small_workspace_gives_the_same_walkers():
    """A workspace below the queried size takes smaller electron batches (and chunks of walkers)."""
    s = config_system("158e")
    q = _q(s)
    R = torch.from_numpy(make_walkers(s, 96, first=54000)).to(dev)
    full = {k: v.clone() for k, v in q.eval(R, precision="mixed").items()}
    need = q.workspace_size(96, "mixed")
    for part in (0.75, 0.4):
        ws = torch.empty(int(need * part), dtype=torch.uint8, device=dev)
        got = q.eval(R, precision="mixed", ws=ws)
        assert torch.equal(got["status"], full["status"])
        assert (got["logpsi"] - full["logpsi"]).abs().max().item() < 1e-6
        assert ((got["e_loc"] - full["e_loc"]).abs() / full["e_parts"].abs().amax(1)).max().item() < 1e-5


@pytest.mark.parametrize("degrees", [(0, 1, 2), (0, 1, 3, 4)])
def test_every_degree(degrees):
    """Shells of degree 0 to 2 (written out) and above (general expressions), every component, in the
    mixed products and the C-free drift against the FP64 path."""
    rng = np.random.default_rng(7)
    shells = [(L, [0.4 + 0.1 * L, 1.3, 2.0][: 1 + L % 3], [0.7, 0.4, 0.3][: 1 + L % 3]) for L in degrees]
    n_ao = sum((L + 1) * (L + 2) // 2 for L in degrees)
    n_up, n_dn = min(n_ao, 9), min(n_ao, 7)
    Qa, _ = np.linalg.qr(rng.normal(size=(n_ao, n_up)))
    Qb, _ = np.linalg.qr(rng.normal(size=(n_ao, n_dn)))
    s = one_atom_system(8, shells, n_up, n_dn, Qa, Qb)
    q = _q(s)
    R = torch.from_numpy(rng.normal(size=(70, n_up + n_dn, 3))).to(dev)
    (gu, gd), (ru, rd) = q.slater(R, precision="mixed"), q.slater(R, precision="f64")
    for g, r in ((gu, ru), (gd, rd)):
        err = (g - r).abs().amax(-1) / r.abs().amax(-1)
        assert err[:, [0, 4]].max().item() < 1e-9
        assert err[:, 1:4].max().item() < 1e-5
    ref, got = q.eval(R, precision="f64"), q.eval(R, precision="mixed")
    assert torch.equal(got["status"], ref["status"]) and torch.equal(got["sign"], ref["sign"])
    d = (got["drift"] - ref["drift"]).abs().amax((1, 2)) / ref["drift"].abs().amax((1, 2))
    assert d.max().item() < 1e-5
    T, Tr = got["e_parts"][:, 0], ref["e_parts"][:, 0]
    assert ((T - Tr).abs() / ref["e_parts"].abs().amax(1)).max().item() < 1e-5
