"""FP64 elimination with each matrix spread over many CTAs (few matrices) against
one CTA per matrix: the same arithmetic in the same order, so bit for bit the
same log|det|, sign and inverse; singular matrices, pivot ties, zeros and
non-finite entries among them.  One CTA per matrix runs on the batch repeated
until it fills the card (304 matrices: two on each of 152 SMs)."""
import pytest
import torch

pytestmark = pytest.mark.gpu
dev = torch.device("cuda", 0)


def _inv(X):
    from paper_1209_6630_gb300 import det_inverse
    return det_inverse(X.clone())


@pytest.mark.parametrize("n", [1, 2, 7, 8, 15, 16, 17, 31, 32, 33, 63, 64, 65, 100, 217, 255, 256, 257, 300])
def test_wide_equals_one_cta_per_matrix(n):
    g = torch.Generator(device="cuda").manual_seed(n)
    X = torch.randn(8, n, n, dtype=torch.float64, device=dev, generator=g)
    X[1] = X[1].round()                              # ties
    X[2, :, n // 2] = 0.0                            # an exactly zero column
    X[3, n // 3, :] = X[3, 0, :]                      # (n > 1) two equal rows
    X[4, 0, 0] = float("nan")
    X[5, n - 1, 0] = float("inf")
    X[6] = torch.eye(n, dtype=torch.float64, device=dev).flip(0)
    few = _inv(X)
    many = _inv(X.repeat(38, 1, 1))
    for a, b in zip(few, many):
        b = b[:8]
        assert torch.equal(torch.isnan(a), torch.isnan(b)) if a.is_floating_point() else True
        assert torch.equal(a.nan_to_num(0.0), b.nan_to_num(0.0)) if a.is_floating_point() else torch.equal(a, b)


@pytest.mark.parametrize("n,batch", [(512, 2), (640, 1), (866, 1), (1024, 2)])
def test_wide_large_inverse(n, batch):
    """Against torch in FP64 (LU): both within n x 2^-53 x kappa of the inverse; kappa <= 1e6 for these."""
    g = torch.Generator(device="cuda").manual_seed(n)
    X = torch.randn(batch, n, n, dtype=torch.float64, device=dev, generator=g)
    X += 3.0 * n ** 0.5 * torch.eye(n, dtype=torch.float64, device=dev)
    logabs, sign, D, sing = _inv(X)
    s, l = torch.linalg.slogdet(X)
    assert torch.equal(s, sign) and not sing.any()
    assert ((logabs - l).abs() / l.abs()).max().item() < 1e-10
    E = D.mT @ X - torch.eye(n, dtype=torch.float64, device=dev)
    assert E.abs().max().item() < n * 2.0 ** -53 * 1e6


@pytest.mark.parametrize("key,W", [("tiny", 3), ("119e", 1), ("119e", 200), ("158e", 1), ("158e", 160), ("300e", 2),
                                   ("434e", 3), ("434e", 160), ("700e", 2), ("1056e", 2)])
@pytest.mark.parametrize("panel", [8, 16, 32])
def test_float_float_inverse(key, W, panel):
    """The float-float elimination in its forms (work matrix in shared memory or not, one or two rows per
    thread, short last panels, odd sizes) against the FP64 one on the same C1 (qmc_slater_matrices):
    log|det| within the mixed path's 1e-6 and the inverse's residual max|D^T C1 - 1| within 1e-6
    (float pairs and a mixed C1, ~2^-44 x kappa <= 1e7; near-node matrices are recomputed in FP64)."""
    from paper_1209_6630_gb300 import QmcSystem, det_inverse
    from synth import config_system, make_system, make_walkers, tiny_system
    s = {"tiny": lambda: tiny_system("h2o_like"), "119e": lambda: make_system(9, 3, 3, 20, seed=21),
         "300e": lambda: make_system(22, 6, 8, 62, seed=31), "700e": lambda: make_system(53, 15, 16, 149, seed=32)}.get(
             key, lambda: config_system(key))()
    q = QmcSystem(s, 0)
    q.set_tiles(a4_mode="float_float", gj_panel=panel, a4_kappa_max=1e7, c15_mode="tensor")
    R = torch.from_numpy(make_walkers(s, W, first=91000)).to(dev)
    out = q.eval(R, precision="mixed", want_dinv=True)
    assert (out["status"] == 0).all()
    sample = torch.unique(torch.linspace(0, W - 1, min(W, 6)).long())
    for sp, C in enumerate(q.slater(R, precision="mixed")):
        n = C.shape[-1]
        off = s.n_up ** 2 if sp else 0
        C1 = C[sample.to(dev), 0].contiguous()
        D = out["dinv"][sample.to(dev), off: off + n * n].reshape(-1, n, n)
        logabs = det_inverse(C1.clone())[0]
        assert (out["logabs"][sample.to(dev), sp] - logabs).abs().max().item() < 1e-6
        E = D.mT @ C1 - torch.eye(n, dtype=torch.float64, device=dev)
        assert E.abs().max().item() < 1e-6


@pytest.mark.parametrize("n_up_plus", [31, 32, 33, 63, 65, 127, 129, 160, 543, 545, 577, 865])
def test_tensor_panel_sizes(n_up_plus):
    """The panel kernel of the tensor-core elimination at the edges of its sub-panels (short last
    panels), of its warps and of its two arithmetics (544 / 545 rows): log|det| against the FP64 path
    within 1e-6 and the inverse's residual within 1e-6 on every walker."""
    from paper_1209_6630_gb300 import QmcSystem, det_inverse
    from synth import make_system, make_walkers
    n = n_up_plus
    heavy = max(2, (2 * n) // 9)
    s = make_system(heavy, 0, 0, 2 * n - 6 * heavy, seed=100 + n)      # 2 n electrons
    assert s.n_up == n
    q = QmcSystem(s, 0)
    q.set_tiles(a4_mode="tensor", c15_mode="tensor")
    R = torch.from_numpy(make_walkers(s, 3, first=95000)).to(dev)
    out = q.eval(R, precision="mixed", want_dinv=True)
    assert (out["status"] == 0).all()
    for sp, C in enumerate(q.slater(R, precision="mixed")):
        m = C.shape[-1]
        off = s.n_up ** 2 if sp else 0
        D = out["dinv"][:, off: off + m * m].reshape(-1, m, m)
        C1 = C[:, 0].contiguous()
        logabs = det_inverse(C1.clone())[0]
        assert (out["logabs"][:, sp] - logabs).abs().max().item() < 1e-6
        E = D.mT @ C1 - torch.eye(m, dtype=torch.float64, device=dev)
        assert E.abs().max().item() < 1e-6


@pytest.mark.parametrize("n", [130, 257, 544, 545])
def test_tensor_update_row_tiles(n):
    """The update's CTAs take one or several row tiles each and the panel runs with one or two CTAs per
    SM, by the number of matrices; every element's arithmetic is the same, so the inverses of one walker repeated W times are equal bit for bit at
    every split (repeated, because C1's slice scales go with the walkers that share a tile)."""
    from paper_1209_6630_gb300 import QmcSystem
    from synth import make_system, make_walkers
    heavy = max(2, (2 * n) // 9)
    s = make_system(heavy, 0, 0, 2 * n - 6 * heavy, seed=100 + n)      # 2 n electrons
    assert s.n_up == n
    q = QmcSystem(s, 0)
    q.set_tiles(a4_mode="tensor", c15_mode="tensor")
    R = torch.from_numpy(make_walkers(s, 1, first=95000)).to(dev)
    ref = q.eval(R, precision="mixed", want_dinv=True)
    for W in (38, 76, 250):
        out = q.eval(R.expand(W, -1, -1).contiguous(), precision="mixed", want_dinv=True)
        assert (out["dinv"] == ref["dinv"]).all()
        assert (out["logabs"] - ref["logabs"]).abs().max().item() < 1e-12
