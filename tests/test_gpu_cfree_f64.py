"""FP64 path without C2..C5: C1 bit-identical to qmc_slater_matrices' (log|Psi| and
D^-1 follow), drift and Laplacian from v = D^-1 A^T.  Reference: the same sums
in torch from the library's own AO derivatives (qmc_screen_ao) and D^-1, with
the rounding bound of the sums as the tolerance: terms x 2^-53 x the sum of
magnitudes, for both sides, and twice that for the AO derivatives' own last bits."""
import numpy as np
import pytest
import torch

from helpers import one_atom_system
from synth import config_system, make_system, make_walkers, tiny_system

pytestmark = pytest.mark.gpu
dev = torch.device("cuda", 0)


def _wide():
    rng = np.random.default_rng(5)
    shells = [(L, [0.4 + 0.1 * i, 2.0], [0.7, 0.4]) for i, L in enumerate((0, 1, 3, 4))]
    return one_atom_system(7, shells, 4, 3, rng.normal(size=(29, 4)), rng.normal(size=(29, 3)))


SYSTEMS = {"h2o": lambda: tiny_system("h2o_like"), "wide": _wide,
           "open": lambda: make_system(9, 3, 3, 20, seed=21),      # n_up, n_dn around one slot of 128 MOs
           "158e": lambda: config_system("158e"), "434e": lambda: config_system("434e"),
           "1056e": lambda: config_system("1056e"), "1731e": lambda: config_system("1731e")}


@pytest.mark.parametrize("key", sorted(SYSTEMS))
def test_f64_drift_from_v(key):
    from paper_1209_6630_gb300 import QmcSystem
    s = SYSTEMS[key]()
    q = QmcSystem(s, 0)
    R = torch.from_numpy(make_walkers(s, 2, first=71000)).to(dev)
    out = q.eval(R, precision="f64", want_dinv=True)
    assert (out["status"] == 0).all()
    cnt, idx, B = q.screen_ao(R, s.n_ao)
    for w in range(2):
        lap_tot, lap_tol = 0.0, 0.0
        for spin, (lo, hi, A) in enumerate(((0, s.n_up, s.A_up), (s.n_up, s.n_elec, s.A_dn))):
            n = hi - lo
            if n == 0:
                continue
            off = s.n_up ** 2 if spin else 0
            D = out["dinv"][w, off: off + n * n].reshape(n, n)
            At = torch.from_numpy(np.asarray(A, np.float64)).to(dev)
            dB = torch.zeros(n, 5, s.n_ao, dtype=torch.float64, device=dev)
            for e in range(n):
                c = int(cnt[w, lo + e])
                dB[e][:, idx[w, lo + e, :c].long()] = B[w, lo + e, :, :c]
            v, va = D @ At.T, D.abs() @ At.abs().T
            eps = 2.0 ** -53 * 4 * (n + s.n_ao)
            for c in range(3):
                ref = (v * dB[:, 1 + c]).sum(1)
                tol = eps * (va * dB[:, 1 + c].abs()).sum(1)
                assert ((out["drift"][w, lo:hi, c] - ref).abs() <= tol + 1e-300).all()
            lap_tot += (v * dB[:, 4]).sum().item()
            lap_tol += eps * (va * dB[:, 4].abs()).sum().item()
        assert abs(out["e_parts"][w, 0].item() + 0.5 * lap_tot) <= 0.5 * lap_tol


def test_f64_c1_is_the_slater_matrix_and_bad_walkers():
    """log|det| of the C1 that qmc_slater_matrices returns is the evaluation's, bit for bit; an
    electron out of every shell's reach makes its matrix singular and the drift NaN."""
    from paper_1209_6630_gb300 import QmcSystem, det_inverse
    s = config_system("434e")
    q = QmcSystem(s, 0)
    R = torch.from_numpy(make_walkers(s, 3, first=72000)).to(dev)
    R[2, 5] = 1.0e3
    out = q.eval(R, precision="f64")
    up, dn = q.slater(R, precision="f64")
    for sp, C in enumerate((up, dn)):
        logabs = det_inverse(C[:2, 0].contiguous())[0]
        assert torch.equal(logabs, out["logabs"][:2, sp])
    assert out["status"][:2].tolist() == [0, 0] and out["status"][2].item() != 0
    assert torch.isnan(out["drift"][2, : s.n_up]).all() and torch.isinf(out["logpsi"][2])
