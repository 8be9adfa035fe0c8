"""The float-pair refinement of a float temperature root (step::refine_quartic)
against the double Newton step (step::refine_root) that it stands in for: wherever
it accepts, both give the same float, bit for bit, and it declines only where it
says it does.  The probe is compiled from the kernels' own header.

Equations over the whole range of the guards, beta rounding up and down to float,
one of the two terms dominant or both alike, temperatures near and far from the
root, roots laid next to the midpoint of two floats, where it must decline, and onto
powers of two, whose neighbour below is half as far as the one above."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2002_08377_gb300 import build as rtbuild

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("refine") / "refine_probe.so")
    subprocess.run([rtbuild.nvcc(), *rtbuild.ARCH, *rtbuild.FLAGS, "-I", rtbuild.CSRC, "-I",
                    rtbuild.INCLUDE, "-shared", os.path.join(HERE, "refine_probe.cu"), "-o", so],
                   check=True)
    fn = ctypes.CDLL(so).probe
    fn.argtypes = [ctypes.c_void_p] * 4 + [ctypes.c_int64, ctypes.c_float] + [ctypes.c_void_p] * 3

    def run(alpha, beta, g, T0, tol):
        dev = lambda x, t: torch.tensor(np.ascontiguousarray(x, t), device="cuda")
        a, b, gg, T = (dev(alpha, np.float32), dev(beta, np.float64), dev(g, np.float32),
                       dev(T0, np.float32))
        n = a.numel()
        quick, full = torch.empty_like(a), torch.empty_like(a)
        took = torch.empty(n, dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        p = lambda x: ctypes.c_void_p(x.data_ptr())
        assert fn(p(a), p(b), p(gg), p(T), n, tol, p(quick), p(took), p(full)) == 0
        return quick.cpu().numpy(), took.cpu().numpy().astype(bool), full.cpu().numpy()

    return run


def _equations(n, rng, spread):
    """alpha, beta, g with a root T and alpha T^3 / beta spread over 2^(+-spread)."""
    T = np.exp2(rng.uniform(-12, 12, n))
    beta = np.exp2(rng.uniform(-20, 20, n)) * (1 + rng.uniform(-1, 1, n) * 2.0 ** -24)
    alpha = (beta / T ** 3 * np.exp2(rng.uniform(-spread, spread, n))).astype(np.float32)
    g = (alpha.astype(np.float64) * T ** 4 + beta * T).astype(np.float32)
    return alpha, beta, g, T


@pytest.mark.parametrize("tol", [1e-4, 1e-7])
@pytest.mark.parametrize("spread", [2, 30])
def test_accepted_roots_equal_the_double_step(probe, spread, tol):
    rng = np.random.default_rng(int(spread))
    n = 1 << 23
    alpha, beta, g, T = _equations(n, rng, spread)
    T0 = T * np.where(rng.uniform(size=n) < 0.5, 1 + 0.1 * rng.uniform(-1, 1, n),
                      np.exp2(rng.uniform(-4, 4, n)))
    quick, took, full = probe(alpha, beta, g, T0, tol)
    assert np.array_equal(quick[took].view(np.uint32), full[took].view(np.uint32))
    # it declines within 2^-40 of a midpoint (2^-15 of the floats at most)
    # and for steps above 3e-7 of T; the latter are few from a converged root
    assert (~took).mean() < 1e-4


@pytest.mark.parametrize("off", [0.0, 2.0 ** -30, -2.0 ** -30, 2.0 ** -25, -2.0 ** -25,
                                 -2.0 ** -25 * (1 - 2.0 ** -13), -2.0 ** -25 * (1 + 2.0 ** -13),
                                 2.0 ** -24 * (1 - 2.0 ** -13), 2.0 ** -24 * (1 + 2.0 ** -13),
                                 -2.0 ** -24])
def test_roots_at_powers_of_two(probe, off):
    """The root a power of two (uniform gas at T = 1) times (1 + off): accepted unless it
    lies next to a midpoint, 2^-24 above and 2^-25 below."""
    rng = np.random.default_rng(11)
    n = 1 << 18
    two = np.exp2(rng.integers(-8, 9, n).astype(np.float64))
    T = two * (1 + off)
    alpha = (np.exp2(rng.uniform(-4, 4, n)) / T ** 3).astype(np.float32)
    g = (alpha.astype(np.float64) * T ** 4 * rng.uniform(1.5, 8.0, n)).astype(np.float32)
    beta = (g - alpha.astype(np.float64) * T ** 4) / T
    T0 = two.astype(np.float32)
    T0 = np.where(rng.uniform(size=n) < 0.3, np.nextafter(T0, np.float32(0)), T0)
    quick, took, full = probe(alpha, beta, g, T0, 0.0)
    assert np.array_equal(quick[took].view(np.uint32), full[took].view(np.uint32))
    if off == -2.0 ** -25:
        assert not took.any()
    else:
        assert took.all()


@pytest.mark.parametrize("off", [0.0, 2.0 ** -44, -2.0 ** -44, 2.0 ** -41, -2.0 ** -41,
                                 2.0 ** -39, -2.0 ** -39, 2.0 ** -30])
def test_roots_near_a_midpoint(probe, off):
    """beta chosen so that the equation's root is a midpoint of two floats times
    (1 + off), the start one float off."""
    rng = np.random.default_rng(7)
    n = 1 << 20
    lo = np.exp2(rng.uniform(-8, 8, n)).astype(np.float32)
    mid = 0.5 * (lo.astype(np.float64) + np.nextafter(lo, np.float32(np.inf)).astype(np.float64))
    T = mid * (1 + off)
    alpha = (np.exp2(rng.uniform(-4, 4, n)) / T ** 3).astype(np.float32)
    g = (alpha.astype(np.float64) * T ** 4 * rng.uniform(1.5, 8.0, n)).astype(np.float32)
    beta = (g - alpha.astype(np.float64) * T ** 4) / T
    T0 = np.where(rng.uniform(size=n) < 0.5, lo, np.nextafter(lo, np.float32(np.inf)))
    quick, took, full = probe(alpha, beta, g, T0, 0.0)
    assert np.array_equal(quick[took].view(np.uint32), full[took].view(np.uint32))
    if abs(off) < 2.0 ** -42:
        assert not took.any()
    if abs(off) > 2.0 ** -31:
        assert took.mean() > 0.99


@pytest.mark.parametrize("shift", [0, 40, 55, 65, 80])
def test_small_energy_densities(probe, shift):
    """The same equations in units of energy density 2^shift times larger: accepted down
    to g = 2^-98 and beta = 2^-100, with the same floats as the double step."""
    rng = np.random.default_rng(3)
    n = 1 << 21
    T = np.exp2(rng.uniform(0, 12, n))
    beta = np.exp2(rng.uniform(-17.9, 0, n)) * (1 + rng.uniform(-1, 1, n) * 2.0 ** -24)
    alpha = (beta / T ** 3 * np.exp2(rng.uniform(-10, 10, n))).astype(np.float32)
    beta = beta * 2.0 ** -shift
    alpha = (alpha * np.float32(2.0 ** -(shift // 2))) * np.float32(2.0 ** -(shift - shift // 2))
    g = (alpha.astype(np.float64) * T ** 4 + beta * T).astype(np.float32)
    T0 = T * (1 + 0.1 * rng.uniform(-1, 1, n))
    quick, took, full = probe(alpha, beta, g, T0, 1e-4)
    assert np.array_equal(quick[took].view(np.uint32), full[took].view(np.uint32))
    assert (~took).mean() < 1e-4


def test_vacuum(probe):
    """The root 0 of a dark cell without energy, opaque or not."""
    rng = np.random.default_rng(13)
    n = 1 << 12
    alpha, beta = np.exp2(rng.uniform(-20, 20, n)), np.exp2(rng.uniform(-90, 20, n))
    alpha[::2] = 0.0
    zero = np.zeros(n)
    quick, took, full = probe(alpha, beta, zero, zero, 0.0)
    assert took.all() and not quick.any() and not full.any()


def test_guard_limits(probe):
    """Powers of two as roots, and scales at and past the guards' limits."""
    rng = np.random.default_rng(9)
    e = rng.integers(-60, 60, 1 << 20)
    T = np.exp2(e.astype(np.float64))
    T = np.where(rng.uniform(size=T.size) < 0.5, T, T * (1 + rng.uniform(0, 1, T.size)))
    with np.errstate(over="ignore", under="ignore"):
        beta = np.exp2(rng.integers(-70, 104, T.size).astype(np.float64)) * \
            (1 + rng.uniform(0, 1, T.size))
        alpha = np.exp2(rng.uniform(-120, 120, T.size)).astype(np.float32)
        g = (alpha.astype(np.float64) * T ** 4 + beta * T).astype(np.float32)
    ok = np.isfinite(g) & (g > 0) & (T < 2.0 ** 60)
    quick, took, full = probe(alpha[ok], beta[ok], g[ok], T[ok].astype(np.float32), 0.0)
    assert took.any() and not took.all()
    assert np.array_equal(quick[took].view(np.uint32), full[took].view(np.uint32))
