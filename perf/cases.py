"""The work that a quantum Monte Carlo program hands to this library, as cases that can be timed.

A program loads one molecule (basis set, nuclei, MO coefficients: a `QmcSystem`, kept for the whole run) and then
evaluates walkers: positions in; log|Psi|, sign, drift and local energy out.  A population has from one walker (a
starting point that is looked at by hand) over tens (what one rank of a large job holds) to a few thousand walkers
(what fills the card).  Around the evaluation there are the DMC step, the gradient for optimising the MO
coefficients, and the single stages.  The molecules are chains of C, N, O and H with 3s2p1d / 2s1p Cartesian
Gaussians; the four sizes are those of the repository's own configurations.

The molecule depends on its composition alone, as a program's input file does; walkers (and the matrices of
`det_inverse`) are drawn from the seed.
"""
from __future__ import annotations

import functools
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1209_6630_gb300 import LogPsi, QmcBatch, QmcSystem, det_inverse

# The repository's configurations: atoms of the chains with 158, 434, 1056 and 1731 electrons.
E158, E434 = dict(n_C=12, n_N=3, n_O=4, n_H=33), dict(n_C=32, n_N=9, n_O=10, n_H=99)
E1056, E1731 = dict(n_C=80, n_N=22, n_O=24, n_H=230), dict(n_C=130, n_N=36, n_O=40, n_H=379)
BASIS_SEED = 2                  # 208, 248, 318 unscreened AOs an electron at 158, 434, 1056 electrons
EPS = 1e-8                      # screening threshold on a shell's radial part
JASTROW = dict(a_par=0.25, a_anti=0.5, b_ee=1.0, a_en=0.8, b_en=2.0)
MOST_WORK = 2048 * 4 * 528**3   # of the largest listed case: walkers x sum over spins of 2 n^3


def listed():
    return [
        # One walker of the smallest molecule: a trial position, a restart check.  Launches and latency.
        dict(name="eval_158e_1w", kind="eval", precision="mixed", walkers=1, **E158),
        # The smallest molecule with the population that its configuration names.
        dict(name="eval_158e_100w", kind="eval", precision="mixed", walkers=100, **E158),
        # What one of many ranges of a large job holds: a large molecule and a few walkers, not a multiple of anything.
        dict(name="eval_1056e_37w", kind="eval", precision="mixed", walkers=37, **E1056),
        # A medium molecule with a full population.
        dict(name="eval_434e_4096w", kind="eval", precision="mixed", walkers=4096, **E434),
        # The headline workload of the repository's benchmark.
        dict(name="eval_1056e_2048w", kind="eval", precision="mixed", walkers=2048, **E1056),
        # A double-precision evaluation: equilibration checks, reference energies.
        dict(name="eval_f64_434e_96w", kind="eval", precision="f64", walkers=96, **E434),
        # One DMC step (move, evaluation, weights, reconfiguration) with a Jastrow factor; ragged population.
        dict(name="dmc_434e_601w", kind="dmc", precision="mixed", walkers=601, **E434),
        # Wave-function optimisation: log|Psi| and its gradient in the MO coefficients, the largest molecule
        # (single-precision coefficients, as its configuration has them).
        dict(name="logpsi_1731e_512w", kind="logpsi", precision="mixed", walkers=512, a_f32=True, **E1731),
        # The same in double precision on the smallest molecule.
        dict(name="logpsi_f64_158e_100w", kind="logpsi", precision="f64", walkers=100, **E158),
        # The five Slater matrices alone (values, gradients, Laplacians), one walker more than a tile of 128.
        dict(name="slater_434e_129w", kind="slater", precision="mixed", walkers=129, **E434),
        # Determinants and inverses alone, a batch of odd size.
        dict(name="det_inverse_217x300", kind="det_inverse", n=217, batch=300),
        # A job that holds several molecules at once: all four, one CUDA graph launch per step.
        dict(name="batch_4x64w", kind="batch", precision="mixed", walkers=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _composition(rng, lo, hi):
    heavy = _log_int(rng, lo, hi)
    n_N, n_O = round(heavy * rng.uniform(0.13, 0.21)), round(heavy * rng.uniform(0.16, 0.24))
    return dict(n_C=heavy - n_N - n_O, n_N=n_N, n_O=n_O, n_H=round(heavy * rng.uniform(1.6, 2.0)))


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "eval_f64", "dmc", "logpsi", "logpsi_f64", "slater", "det_inverse", "batch"])
    if kind == "det_inverse":
        n = _log_int(rng, 79, 866)
        return dict(kind=kind, n=n, batch=_log_int(rng, 1, max(2, min(2000, 2 * 10**11 // (2 * n**3)))))
    if kind == "batch":
        return dict(kind=kind, precision="mixed", walkers=_log_int(rng, 1, 96))
    f64 = kind.endswith("_f64")
    comp = _composition(rng, 19, 206 if not f64 and kind != "slater" else 51)
    n_s = (6 * comp["n_C"] + 7 * comp["n_N"] + 8 * comp["n_O"] + comp["n_H"] + 1) // 2
    most = MOST_WORK // (4 * n_s**3)
    walkers = {"eval": min(4096, most), "dmc": min(2048, most // 2), "logpsi": min(512, most // 4), "slater": 300,
               "eval_f64": min(256, most // 16), "logpsi_f64": min(128, most // 16)}[kind]
    return dict(kind=kind.removesuffix("_f64"), precision="f64" if f64 else "mixed",
                walkers=_log_int(rng, 2 if "logpsi" in kind else 1, max(3, walkers)), **comp)


# --- the molecules ------------------------------------------------------------------------------------------

HEAVY, HYDROGEN = [(0, 8), (0, 0), (0, 0), (1, 0), (1, 0), (2, 0)], [(0, 0), (0, 0), (1, 0)]   # (L, primitives; 0: 1..3)


def _dfact(n):
    return math.prod(range(n, 0, -2)) if n > 0 else 1


def _far(p, others, least):
    return not len(others) or np.min(np.linalg.norm(np.asarray(others) - p, axis=1)) >= least


def _geometry(rng, n_heavy, n_H):
    """A self-avoiding chain with 2.8 bohr bonds and angles of 110 +- 5 degrees, and hydrogens 2 bohr from its atoms."""
    pos = [np.zeros(3), np.array([2.8, 0.0, 0.0])][:n_heavy]
    while len(pos) < n_heavy:
        b, c = pos[-2], pos[-1]
        u = (c - b) / np.linalg.norm(c - b)
        side = np.cross(u, rng.normal(size=3))          # a uniform dihedral
        th = math.radians(180.0 - 110.0 + rng.uniform(-5.0, 5.0))
        p = c + 2.8 * (math.cos(th) * u + math.sin(th) * side / np.linalg.norm(side))
        if _far(p, pos[:-1], 2.5):
            pos.append(p)
    every = list(pos)
    while len(every) < n_heavy + n_H:
        k, v = int(rng.integers(n_heavy)), rng.normal(size=3)
        p = pos[k] + 2.0 * v / np.linalg.norm(v)
        if _far(p, every[:k] + every[k + 1:], 1.8):
            every.append(p)
    return np.array(every)


def _shells(rng, kinds):
    """(L, exponents, coefficients with unit self-overlap of the x^L component) of one element."""
    out = []
    for L, n in kinds:
        n = n or int(rng.integers(1, 4))
        g = np.sort(np.exp(rng.uniform(math.log(0.1), math.log(30.0), n)))[::-1]
        c = rng.uniform(0.1, 1.0, n)
        norm = (2 * g / math.pi) ** 0.75 * (4 * g) ** (L / 2) / math.sqrt(_dfact(2 * L - 1))
        overlap = (2 * np.sqrt(np.outer(g, g)) / (g[:, None] + g)) ** (L + 1.5)
        out.append((L, g, c * norm / math.sqrt(c @ overlap @ c)))
    return out


@functools.lru_cache(maxsize=8)
def _molecule(n_C, n_N, n_O, n_H, a_f32=False):
    rng = np.random.default_rng([n_C, n_N, n_O, n_H])
    heavy = rng.permutation([6.0] * n_C + [7.0] * n_N + [8.0] * n_O)
    Z = np.concatenate([heavy, np.ones(n_H)])
    Q = _geometry(rng, len(heavy), n_H)
    basis_rng = np.random.default_rng(BASIS_SEED)           # one basis set for every molecule
    basis = {z: _shells(basis_rng, HYDROGEN if z == 1 else HEAVY) for z in (1.0, 6.0, 7.0, 8.0)}
    sh, prim, ao = [], [], []                            # (atom, L, primitives, first), (exponent, coefficient), (shell, powers, scale)
    for a, z in enumerate(Z):
        for L, g, c in basis[z]:
            for nx in range(L, -1, -1):
                for ny in range(L - nx, -1, -1):
                    nz = L - nx - ny
                    scale = math.sqrt(_dfact(2 * L - 1) / (_dfact(2 * nx - 1) * _dfact(2 * ny - 1) * _dfact(2 * nz - 1)))
                    ao.append((len(sh), (nx, ny, nz), scale))
            sh.append((a, L, len(g), len(prim)))
            prim += list(zip(g, c))
    electrons = np.repeat(np.arange(len(Z)), Z.astype(int))   # Z electrons at each nucleus, dealt to the spins in turn
    where = np.concatenate([electrons[0::2], electrons[1::2]])
    n_up, n_dn = len(electrons[0::2]), len(electrons[1::2])
    A = np.linalg.qr(rng.normal(size=(len(ao), n_up)))[0]
    dt = np.float32 if a_f32 else np.float64
    i32 = functools.partial(np.array, dtype=np.int32)
    return SimpleNamespace(
        n_atom=len(Z), Z=Z, Q=Q, n_shell=len(sh), shell_atom=i32([s[0] for s in sh]), shell_L=i32([s[1] for s in sh]),
        shell_nprim=i32([s[2] for s in sh]), shell_pstart=i32([s[3] for s in sh]),
        prim_gamma=np.array([p[0] for p in prim]), prim_coef=np.array([p[1] for p in prim]), n_ao=len(ao),
        ao_shell=i32([x[0] for x in ao]), ao_pow=i32([x[1] for x in ao]), ao_scale=np.array([x[2] for x in ao]),
        n_up=n_up, n_dn=n_dn, A_up=np.ascontiguousarray(A, dtype=dt), A_dn=np.ascontiguousarray(A[:, :n_dn], dtype=dt),
        eps=EPS, where=where)


def _of(case):
    """The molecules of a case."""
    if case["kind"] == "batch":
        return [_molecule(**E158), _molecule(**E434), _molecule(**E1056), _molecule(**E1731, a_f32=True)]
    return [_molecule(case["n_C"], case["n_N"], case["n_O"], case["n_H"], case.get("a_f32", False))]


@functools.lru_cache(maxsize=1)
def _loaded(key):
    """The loaded systems that a program keeps (one case's at a time: a system keeps its workspace)."""
    case = dict(key)
    systems = [QmcSystem(m) for m in _of(case)]
    if case["kind"] == "dmc":
        systems[0].set_jastrow(JASTROW)
    return systems


def _systems(case):
    return _loaded(tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "walkers", "precision"))))


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _walkers(m, W, g):
    """Every electron at its nucleus + N(0, 1 bohr^2) per component."""
    at = torch.from_numpy(m.Q[m.where]).cuda()
    return (at + torch.randn(W, len(m.where), 3, dtype=torch.float64, device="cuda", generator=g)).contiguous()


def _matrices(case, seed):
    """Matrices like Slater matrices: a row's scale is set by how near its electron is to a nucleus."""
    g, b, n = _generator(seed), case["batch"], case["n"]
    X = torch.randn(b, n, n, dtype=torch.float64, device="cuda", generator=g)
    return X * torch.exp(0.7 * torch.randn(b, n, 1, dtype=torch.float64, device="cuda", generator=g)) * (n**-0.5)


# --- one pass -----------------------------------------------------------------------------------------------

def prepare(case, seed):
    st = SimpleNamespace(case=case)
    if case["kind"] == "det_inverse":
        st.X = _matrices(case, seed)
        return st
    st.q, g = _systems(case), _generator(seed)
    st.R = [_walkers(m, case["walkers"], g) for m in _of(case)]
    if case["kind"] == "batch":
        st.batch = QmcBatch(list(zip(st.q, st.R)), precision=case["precision"])
    if case["kind"] == "dmc":
        st.a = st.q[0].init_state(st.R[0], precision=case["precision"])
        st.b = st.q[0].walker_state(case["walkers"])
        st.stats = torch.zeros(4, dtype=torch.float64, device="cuda")
        st.e_trial, st.step_seed = -500.0, seed
    if case["kind"] == "logpsi":
        m = _of(case)[0]
        st.A = [torch.from_numpy(x).cuda().requires_grad_() for x in (m.A_up, m.A_dn)]
    return st


def run(st):
    case = st.case
    if case["kind"] == "det_inverse":
        return det_inverse(st.X.clone())                 # the call consumes its matrices
    q, R = st.q[0], st.R[0]
    if case["kind"] == "eval":
        return q.eval(R, precision=case["precision"])
    if case["kind"] == "slater":
        return q.slater(R, precision=case["precision"])
    if case["kind"] == "batch":
        return st.batch.launch()
    if case["kind"] == "dmc":
        # the same step from the same population each time
        st.stats.zero_()
        out = q.dmc_step(st.a, st.b, tau=1e-4, e_trial=st.e_trial, seed=st.step_seed, step=1, precision=case["precision"],
                         stats=st.stats)
        return dict(out, stats=st.stats)
    logpsi, e_loc = LogPsi.apply(*st.A, R, q, case["precision"])
    with torch.no_grad():
        g = 2.0 * (e_loc - e_loc.mean()) / len(e_loc)    # the energy gradient's weights
    dA_up, dA_dn = torch.autograd.grad(logpsi, st.A, g)
    return dict(logpsi=logpsi.detach(), e_loc=e_loc, dA_up=dA_up, dA_dn=dA_dn)


# --- what a pass cannot do without -----------------------------------------------------------------------------

@functools.lru_cache(maxsize=64)
def _active(*comp):
    """Mean number of unscreened AOs of an electron, from one walker."""
    m = _molecule(*comp)
    r = m.Q[m.where] + np.random.default_rng(1).normal(size=(len(m.where), 3))
    d2 = ((r[:, None, :] - m.Q[None]) ** 2).sum(-1)[:, m.shell_atom]
    g = np.zeros_like(d2)
    for p in range(int(m.shell_nprim.max())):
        has = p < m.shell_nprim
        k = np.where(has, m.shell_pstart + p, 0)
        g += np.where(has, m.prim_coef[k], 0.0) * np.exp(-m.prim_gamma[k] * d2)
    width = np.bincount(m.ao_shell, minlength=m.n_shell)
    return float(((g >= EPS) * width).sum(1).mean())


def _eval_work(case, m, comp):
    W, N, K = case["walkers"], m.n_up + m.n_dn, _active(*comp)
    n2, n3 = m.n_up**2 + m.n_dn**2, m.n_up**3 + m.n_dn**3
    products = 2.0 * n2 * K                              # one of the products with the MO coefficients
    a_bytes = m.A_up.nbytes + m.A_dn.nbytes
    kind = case["kind"]
    if kind == "slater":
        return dict(flops=W * 5 * products, bytes=W * (24 * N + 40 * n2) + a_bytes)
    # C1; determinant and inverse; drift and Laplacian from D^-1 A^T; the pairs of electrons
    w = dict(flops=W * (2 * products + 2 * n3 + 10.0 * N * (N / 2 + m.n_atom)), bytes=W * (48 * N + 80) + a_bytes)
    if kind == "dmc":
        w["bytes"] += W * 96 * N                         # the population before and after
    if kind == "logpsi":
        w["flops"] += W * products
        w["bytes"] += a_bytes
    return w


def work(case):
    if case["kind"] == "det_inverse":
        return dict(flops=2.0 * case["batch"] * case["n"] ** 3, bytes=16.0 * case["batch"] * case["n"] ** 2)
    if case["kind"] == "batch":
        comps = [tuple(c.values()) for c in (E158, E434, E1056)] + [(*E1731.values(), True)]
        every = [_eval_work(case, _molecule(*c), c) for c in comps]
        return dict(flops=sum(w["flops"] for w in every), bytes=sum(w["bytes"] for w in every))
    comp = (case["n_C"], case["n_N"], case["n_O"], case["n_H"], case.get("a_f32", False))
    return _eval_work(case, _molecule(*comp), comp)


# --- the same in 64 bits, by definition ---------------------------------------------------------------------------

class _Basis:
    """A molecule's AOs in plain torch."""

    def __init__(self, m):
        t = lambda x: torch.as_tensor(x, device="cuda")   # noqa: E731
        self.m, self.Q, self.Z = m, t(m.Q), t(m.Z)
        self.sh_atom, self.ao_shell, self.ao_scale = t(m.shell_atom).long(), t(m.ao_shell).long(), t(m.ao_scale)
        self.pow = t(m.ao_pow).long()
        most, k = int(m.shell_nprim.max()), np.arange(int(m.shell_nprim.max()))
        at = np.minimum(m.shell_pstart[:, None] + k, len(m.prim_coef) - 1)
        has = k < m.shell_nprim[:, None]
        self.gamma, self.coef, self.most = t(np.where(has, m.prim_gamma[at], 0.0)), t(np.where(has, m.prim_coef[at], 0.0)), most
        self.A = [t(np.asarray(x, np.float64)) for x in (m.A_up, m.A_dn)]

    def aos(self, r):
        """chi, its gradient (3) and Laplacian at positions r [n, 3]: five [n, n_ao]; zero where the shell is screened out."""
        d = r[:, None, :] - self.Q[None]
        d2 = (d * d).sum(-1)[:, self.sh_atom]
        g, gd, gdd = torch.zeros_like(d2), torch.zeros_like(d2), torch.zeros_like(d2)
        for p in range(self.most):
            e = self.coef[:, p] * torch.exp(-self.gamma[:, p] * d2)
            g += e
            gd += self.gamma[:, p] * e
            gdd += self.gamma[:, p] ** 2 * e
        on = (g >= EPS).to(g.dtype)
        g, gd, gdd = ((x * on)[:, self.ao_shell] for x in (g, gd, gdd))
        dx, n = d[:, self.sh_atom[self.ao_shell]], self.pow[None]
        pw = torch.where(n == 0, 1.0, torch.where(n == 1, dx, dx * dx))
        d1 = torch.where(n == 0, 0.0, torch.where(n == 1, 1.0, 2.0 * dx))
        c2 = torch.where(n == 2, 2.0, 0.0).to(g.dtype)
        P = pw.prod(-1)
        chi, grad, lap = P * g, [], 0.0
        L = n.sum(-1)
        for a in range(3):
            o = pw[..., (a + 1) % 3] * pw[..., (a + 2) % 3]
            grad.append((d1[..., a] * g - 2.0 * dx[..., a] * pw[..., a] * gd) * o)
            lap = lap + c2[..., a] * o * g
        lap = lap - (4.0 * L + 6.0) * P * gd + 4.0 * d2[:, self.ao_shell] * P * gdd
        return [x * self.ao_scale for x in (chi, *grad, lap)]


def _exact_eval(m, R, with_grad=False):
    B, W, N = _Basis(m), R.shape[0], R.shape[1]
    split = [(0, m.n_up), (m.n_up, N)]
    f64 = dict(dtype=torch.float64, device="cuda")
    drift, lap, la, sg = torch.empty(W, N, 3, **f64), torch.empty(W, N, **f64), torch.empty(W, 2, **f64), torch.empty(W, 2, **f64)
    keep = []
    for w in range(W):
        B5 = B.aos(R[w])
        for s, (lo, hi) in enumerate(split):
            X = B5[0][lo:hi] @ B.A[s]
            sg[w, s], la[w, s] = torch.linalg.slogdet(X)
            D = torch.linalg.inv(X).T                     # D[e, k]: the weight of MO k for electron e
            v = D @ B.A[s].T
            for a in range(3):
                drift[w, lo:hi, a] = (v * B5[1 + a][lo:hi]).sum(1)
            lap[w, lo:hi] = (v * B5[4][lo:hi]).sum(1)
            if with_grad:
                keep.append(B5[0][lo:hi].T @ D)
    kin = -0.5 * lap.sum(1)
    ven = torch.stack([-(B.Z / torch.cdist(r[None], B.Q[None], compute_mode="donot_use_mm_for_euclid_dist")[0]).sum() for r in R])
    vee = torch.stack([(1.0 / torch.pdist(r)).sum() for r in R])
    vnn = (torch.outer(B.Z, B.Z) / torch.cdist(B.Q, B.Q).fill_diagonal_(math.inf)).sum() / 2
    parts = torch.stack([kin, ven, vee, vnn.expand(W)], 1)
    out = dict(logpsi=la.sum(1), sign=sg.prod(1), logabs=la, drift=drift, e_loc=parts.sum(1), e_parts=parts,
               status=torch.zeros(W, dtype=torch.int32, device="cuda"))
    return out, keep


def exact(case, seed):
    if case["kind"] == "det_inverse":
        X = _matrices(case, seed)
        sign, logabs = torch.linalg.slogdet(X)
        return logabs, sign, torch.linalg.inv(X).mT.contiguous(), torch.zeros(len(X), dtype=torch.int32, device="cuda")
    if case["kind"] == "dmc":
        return None                                      # the step's random numbers are the library's own
    ms, g = _of(case), _generator(seed)
    dense = sum((m.n_up**2 + m.n_dn**2) * 6.0 * m.n_ao + 12.0 * (m.n_up**3 + m.n_dn**3) for m in ms)
    if case["walkers"] * (dense / 1e12 + 0.008 * len(ms)) > 15.0:
        return None                                      # double precision would take too long
    Rs = [_walkers(m, case["walkers"], g) for m in ms]
    if case["kind"] == "batch":
        return [_exact_eval(m, R)[0] for m, R in zip(ms, Rs)]
    m, R = ms[0], Rs[0]
    if case["kind"] == "eval":
        return _exact_eval(m, R)[0]
    if case["kind"] == "slater":
        B, up, dn = _Basis(m), [], []
        for r in R:
            B5 = B.aos(r)
            up.append(torch.stack([b[:m.n_up] @ B.A[0] for b in B5]))
            dn.append(torch.stack([b[m.n_up:] @ B.A[1] for b in B5]))
        return torch.stack(up), torch.stack(dn)
    out, keep = _exact_eval(m, R, with_grad=True)
    wg = 2.0 * (out["e_loc"] - out["e_loc"].mean()) / len(R)
    dA = [sum(wg[w] * keep[2 * w + s] for w in range(len(R))) for s in range(2)]
    return dict(logpsi=out["logpsi"], e_loc=out["e_loc"], dA_up=dA[0], dA_dn=dA[1])
