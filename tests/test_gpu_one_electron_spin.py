"""Systems whose spins differ widely, a spin of one or two electrons beside 32 and more: the spread FP64
elimination keeps a matrix's state in its own D^-1, which has 8 bytes at one electron.  Against the
oracle, with and without the caller's own D^-1 (whose neighbouring memory must stay as it was), at
few walkers, at many (one CTA per matrix) and from 512 rows on (always spread).  The default mixed path on the
same systems (float-float and tensor-core a4)."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import Oracle
from synth import make_system, make_walkers

pytestmark = pytest.mark.gpu
dev = torch.device("cuda", 0)


def _spins(n_up, n_dn):
    """A chain with its electrons dealt to the spins as asked."""
    n = max(n_up, n_dn)
    heavy = max(2, (2 * n) // 9)
    s = make_system(heavy, 0, 0, max(2 * n - 6 * heavy, 4), seed=300 + n)
    Q, _ = np.linalg.qr(np.random.default_rng(n).normal(size=(s.n_ao, n)))
    full = np.repeat(np.arange(len(s.Z)), s.Z.astype(int))
    at = lambda k: full[np.linspace(0, len(full) - 1, k).astype(int)]   # noqa: E731
    return dataclasses.replace(s, n_up=n_up, n_dn=n_dn, A_up=np.ascontiguousarray(Q[:, :n_up]),
                               A_dn=np.ascontiguousarray(Q[:, :n_dn]),
                               elec_atom=np.concatenate([at(n_up), at(n_dn)]).astype(np.int32))


@pytest.mark.parametrize("n_up,n_dn", [(40, 1), (1, 40), (33, 2), (2, 33), (100, 7), (520, 1)])
@pytest.mark.parametrize("W", [1, 3, 160])
@pytest.mark.parametrize("mode", ["f64", "fp64_a4", "mixed"])
def test_small_spin_beside_a_large_one(n_up, n_dn, W, mode):
    from paper_1209_6630_gb300 import QmcSystem
    if max(n_up, n_dn) > 500 and W > 3:
        W = 5
    s = _spins(n_up, n_dn)
    q = QmcSystem(s, 0)
    precision = "f64" if mode == "f64" else "mixed"
    if mode == "fp64_a4":
        q.set_tiles(a4_mode="fp64")
    R = make_walkers(s, W, first=41000)
    sample = np.unique([0, W // 2, W - 1])
    ref = Oracle(s).eval(R[sample], nthreads=8)
    Rd = torch.from_numpy(R).to(dev)
    # the FP64 path's bars, and the mixed path's; the inverse's residual: kappa <= 1e8 times 2^-40 (mixed
    # C1) or n 2^-53 (FP64)
    bar, lbar, res = (1e-5, 1e-6, 1e-4) if precision == "mixed" else (1e-10, 1e-9, 1e-5)
    for own_dinv in (False, True):
        out = q.alloc_out(W)
        msz, pad = n_up ** 2 + n_dn ** 2, 64
        if own_dinv:
            room = torch.full((W * msz + pad,), 7.25, dtype=torch.float64, device=dev)
            out["dinv"] = room[: W * msz].view(W, msz)
        q.eval(Rd, precision=precision, out=out)
        assert (out["status"] == 0).all() and torch.isfinite(out["logpsi"]).all()
        got = {k: v.cpu().numpy()[sample] for k, v in out.items()}
        np.testing.assert_array_equal(got["sign"], ref["sign"])
        assert np.abs(got["logpsi"] - ref["logpsi"]).max() < lbar
        scale = np.abs(ref["e_parts"]).max(1)
        assert (np.abs(got["e_loc"] - ref["e_loc"]) / scale).max() < bar
        d = np.abs(got["drift"] - ref["drift"]).max((1, 2)) / np.abs(ref["drift"]).max((1, 2))
        assert d.max() < bar
        if own_dinv:
            assert (room[W * msz:] == 7.25).all()
            C = q.slater(Rd, precision="f64")
            for sp, n in enumerate((n_up, n_dn)):
                D = out["dinv"][:, (n_up ** 2 if sp else 0):][:, : n * n].reshape(W, n, n)
                E = D.mT @ C[sp][:, 0] - torch.eye(n, dtype=torch.float64, device=dev)
                assert E.abs().max().item() < res


def test_wide_small_spin_is_the_inverse_alone():
    """The D^-1 of an evaluation with spins of 40 and 7 electrons, spread, is bit for bit that of the same
    matrices alone: 7 rows go one CTA per matrix there."""
    from paper_1209_6630_gb300 import QmcSystem, det_inverse
    s = _spins(40, 7)
    q = QmcSystem(s, 0)
    R = torch.from_numpy(make_walkers(s, 3, first=42000)).to(dev)
    out = q.eval(R, precision="f64", want_dinv=True)
    for sp, C in enumerate(q.slater(R, precision="f64")):
        n = C.shape[-1]
        la, sg, D, _ = det_inverse(C[:, 0].contiguous())
        assert torch.equal(la, out["logabs"][:, sp])
        assert torch.equal(D.reshape(3, -1), out["dinv"][:, (1600 if sp else 0):][:, : n * n])
