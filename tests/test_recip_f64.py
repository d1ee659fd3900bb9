"""The FP64 reciprocals of the energy kernel (csrc/recip_f64.cuh) against long double.

CPU: the header compiled for the host, its FP32 seeds off by up to 2 units of their last place (what
CUDA documents for rsqrtf).  1/sqrt is one rounding: 0.5 ulp, and 2^-10 for the third-order remainder.  The
Jastrow term's mean errors are no larger than those of the same formulas from correctly rounded sqrt
and divisions (1% for the sampling of 400000 arguments; lap U, whose terms cancel, by its larger term).
GPU: 1/r of two electrons on a line, which is V_ee itself, and J of two electrons."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include <math.h>
#include <string.h>
static int g_off;
static float off(float x) { for (int k = 0; k < (g_off < 0 ? -g_off : g_off); ++k) x = nextafterf(x, g_off > 0 ? INFINITY : 0.f); return x; }
static float seed_rsqrt(float x) { return off((float)(1.0 / sqrt((double)x))); }
static float seed_rcp(float x) { return (float)(1.0 / (double)x); }
static double plain_rsqrt(double x) { return 1.0 / sqrt(x); }
static int hiint(double x) { long long v; memcpy(&v, &x, 8); return (int)(v >> 32); }
static int loint(double x) { long long v; memcpy(&v, &x, 8); return (int)v; }
static double hilo(int h, int l) { long long v = (long long)((unsigned long long)(unsigned)h << 32 | (unsigned)l); double x; memcpy(&x, &v, 8); return x; }
#define __double2hiint hiint
#define __double2loint loint
#define __hiloint2double hilo
#define rsqrtf seed_rsqrt
#define __frcp_rn seed_rcp
#define rsqrt plain_rsqrt
#define __device__
#define __forceinline__ inline
#include "recip_f64.cuh"
static double ulps(double x, long double ref, long double of)
{
    int e; frexpl(of, &e);
    return (double)(fabsl((long double)x - ref) / ldexpl(1.0L, e - 53));
}
// mean[0..3], most[0..3]: 1/sqrt, U, U'/r, lap U; plain[0..3]: means from sqrt and division
extern "C" void errors(long n, const double *x, const double *a, const double *b, double *mean, double *most, double *plain)
{
    for (int q = 0; q < 4; ++q) mean[q] = most[q] = plain[q] = 0.0;
    for (long i = 0; i < n; ++i) {
        g_off = (int)(i % 5) - 2;
        const long double r = sqrtl((long double)x[i]), q = 1.0L + (long double)b[i] * r, u1 = (long double)a[i] / (q * q);
        const long double u = (long double)a[i] * r / q, f = u1 / r, u2 = -2.0L * (long double)b[i] * u1 / q, lap = u2 + 2.0L * f;
        const long double big = fabsl(u2) > fabsl(2.0L * f) ? u2 : 2.0L * f;
        double jf, jl, ju;
        qmc::jastrow_term(x[i], a[i], b[i], jf, jl, ju);
        const double e[4] = {ulps(qmc::rsqrt_f64(x[i]), 1.0L / r, 1.0L / r), ulps(ju, u, u), ulps(jf, f, f), ulps(jl, lap, big)};
        const double R = sqrt(x[i]), Q = 1.0 + b[i] * R, iq = 1.0 / Q, U1 = a[i] * iq * iq, F = U1 / R;
        const double p[4] = {ulps(1.0 / R, 1.0L / r, 1.0L / r), ulps(a[i] * R * iq, u, u), ulps(F, f, f),
                             ulps(-2.0 * a[i] * b[i] * iq * iq * iq + 2.0 * F, lap, big)};
        for (int k = 0; k < 4; ++k) {
            mean[k] += e[k] / n;
            plain[k] += p[k] / n;
            if (e[k] > most[k]) most[k] = e[k];
        }
    }
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("recip")
    (d / "h.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_1209_6630_gb300", "csrc"), "-o", str(d / "h.so"), str(d / "h.cpp"), "-lm"],
                   check=True)
    return ctypes.CDLL(str(d / "h.so"))


@pytest.mark.parametrize("lo,hi", [(1e-4, 1e3), (1e-29, 1e29)])
def test_errors_in_ulp(host, lo, hi):
    rng = np.random.default_rng(17)
    n = 400000
    x = np.exp(rng.uniform(np.log(lo), np.log(hi), n))
    a, b = rng.uniform(-1.0, 1.0, n), rng.uniform(0.2, 3.0, n)
    p = lambda v: v.ctypes.data_as(ctypes.POINTER(ctypes.c_double))   # noqa: E731
    mean, most, plain = np.zeros(4), np.zeros(4), np.zeros(4)
    host.errors(ctypes.c_long(n), p(x), p(a), p(b), p(mean), p(most), p(plain))
    assert most[0] <= 0.5 + 2.0 ** -10
    assert (mean <= 1.01 * plain).all(), (mean, plain)


@pytest.mark.gpu
def test_two_electrons_on_the_gpu():
    """One electron of each spin on the x axis: r^2 = (x1 - x2)^2 in one rounding, V_ee = 1/r at 0.5 ulp and 2^-10
    for the remainder; with a = 10^6, log|Psi| is J but for a rounding of 0.5 ulp: 4 ulp with U's own 3.1."""
    import torch
    from helpers import one_atom_system
    from paper_1209_6630_gb300 import QmcSystem
    s = one_atom_system(2, [(0, [0.5], [1.0])], 1, 1, np.ones((1, 1)), np.ones((1, 1)))
    q = QmcSystem(s, 0)
    W = 20000
    rng = np.random.default_rng(18)
    R = np.zeros((W, 2, 3))
    R[:, :, 0] = rng.uniform(-2.0, 2.0, (W, 2))
    R[:, 1, 0] = np.where(np.arange(W) % 4 == 0, R[:, 0, 0] + 10.0 ** rng.uniform(-6, 0, W), R[:, 1, 0])
    Rd = torch.from_numpy(R).cuda()
    out = q.eval(Rd, precision="f64")
    assert (out["status"] == 0).all()
    dx = R[:, 0, 0] - R[:, 1, 0]
    r = np.sqrt((dx * dx).astype(np.longdouble))
    ref = 1.0 / r
    err = np.abs(out["e_parts"][:, 2].cpu().numpy() - ref) / np.spacing(ref.astype(np.float64))
    assert err.max() <= 0.5 + 2.0 ** -10
    a, b = 1e6, 1.25
    la = out["logpsi"].cpu().numpy()
    q.set_jastrow(dict(a_par=0.0, a_anti=a, b_ee=b, a_en=0.0, b_en=1.0))
    got = q.eval(Rd, precision="f64")["logpsi"].cpu().numpy()
    big = dx * dx > 1e-4                                  # (J above 10^4: log|Det| is a small addend)
    J = a * r / (1.0 + b * r) + la
    err = np.abs(got - J)[big] / np.spacing(np.abs(J).astype(np.float64))[big]
    assert err.max() <= 4.0
