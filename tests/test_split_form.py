"""The split products' arithmetic (csrc/split.cuh), emulated in integers on the CPU with the segments
of csrc/split_layout.h, against the exact product of the stored FP64 values: reaction tables up to
the admission limit (a layer's k below k_max, evanescent growth along the rows), within a layer and
across an interface, multipoles of sources in the inner part of their cell, potentials over the
target cell.  The error must be that of a product in FP64, not of one in fewer bits."""

import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest
from scipy.special import jv

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WORK = os.path.join(ROOT, "tests", "_build")   # git-ignored
CSRC = os.path.join(ROOT, "paper_2511_12450_gb300", "csrc")


@pytest.fixture(scope="module")
def segment_size():
    cxx = shutil.which("g++") or shutil.which("c++")
    inc = [d for d in (os.environ.get("CUDA_HOME", ""), "/usr/local/cuda")
           if d and os.path.exists(os.path.join(d, "include", "cuda_runtime.h"))]
    if cxx is None or not inc:
        pytest.skip("needs a C++ compiler and the CUDA headers")
    os.makedirs(WORK, exist_ok=True)
    exe = os.path.join(WORK, "split_harness")
    res = subprocess.run([cxx, "-std=c++17", "-I", os.path.join(inc[0], "include"), "-I", CSRC,
                          os.path.join(ROOT, "tests", "split_harness.cpp"), "-o", exe], capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    return lambda *a: int(subprocess.run([exe, *map(repr, a)], capture_output=True, text=True, check=True).stdout)


def ky(k, lam):
    s = np.sqrt(k * k - lam * lam + 0j)
    return np.where(s.imag < 0, -s, s)


def reaction_table(ks, kt, k2, hS, hT, X, p, T):
    """I_mn of waves from the layer ks to itself (kt None) off a half space k2, or into the layer kt
    (density 2 in the second layer), summed over the nodes in a form that stays in range"""
    out = np.zeros((2 * p + 1, 2 * p + 1), complex)
    n = np.arange(-p, p + 1)[:, None]

    def add(lam, w, signs):
        a, b = ky(ks, lam), ky(k2 if kt is None else kt, lam)
        dens = 1j / (2 * a) * (a - 2 * b) / (a + 2 * b) if kt is None else 1j / (a + 2 * b)
        kyt, kk = (a, ks) if kt is None else (b, kt)
        for sg in signs:
            half = 0.5 * (np.log(dens * w / (2 * np.pi)) + 1j * a * hS + 1j * kyt * hT + sg * 1j * lam * X)
            U = sg * n * np.log((a + 1j * lam) / ks) + half
            V = -sg * n * np.log((kyt + 1j * lam) / kk) + half
            u, v = U.real.max(0), V.real.max(0)
            q = u + v > (u + v).max() - 700
            out[:] += (np.exp(V[:, q] - v[q]) * np.exp(u[q] + v[q])) @ np.exp(U[:, q] - u[q]).T

    h = min(0.5, 1 / X)
    gx, gw = np.polynomial.legendre.leggauss(16)
    panels = 300
    t = ((np.arange(panels)[:, None] + 0.5 * (1 + gx)) * (T / panels)).ravel()
    w = np.tile(0.5 * T / panels * gw, panels)
    add(t - 1j * h * np.sin(0.5 * np.pi * t / T), w * (1 - 1j * h * 0.5 * np.pi / T * np.cos(0.5 * np.pi * t / T)), (1, -1))
    v = np.linspace(-4.2, 3.4, 500)
    e = np.exp(np.pi / 2 * np.sinh(v))
    de = e * np.pi / 2 * np.cosh(v) * (v[1] - v[0])
    D = hS + hT
    for sg in (1, -1):
        u = (D + 1j * sg * X) / np.hypot(D, X)
        add(T - 1j * h + e / np.hypot(D, X) * u, de / np.hypot(D, X) * u, (sg,))
    return out


def cut(x, shift):
    """x 2^shift towards zero, as Python integers"""
    out = np.empty(x.shape, dtype=object)
    for i in np.ndindex(x.shape):
        m, e = np.frexp(x[i])
        q, s = abs(int(m * 2.0 ** 53)), int(e - 53 + shift[i])
        q = q << s if s >= 0 else q >> -s
        out[i] = q if m >= 0 else -q
    return out


def digits(ints):
    """eight signed digits of base 256, the largest first"""
    u = ints + 0x8080808080808080
    return [np.array((u >> (8 * (7 - j))) & 255, dtype=np.int64) - 128 for j in range(8)]


def split_product(A, v, d, size, p):
    n = np.abs(np.arange(-p, p + 1))

    def expo(z, off):
        m = np.maximum(np.abs(z.real), np.abs(z.imag))
        return np.where(m > 0, np.frexp(np.where(m > 0, m, 1.0))[1], -100000) + off

    total = np.zeros(2 * p + 1, complex)
    for seg in range(p // size + 1):
        c = np.where((n >= seg * size) & (n < (seg + 1) * size))[0]
        dd, As, vs = d[n[c]], A[:, c], v[c]
        ea, ev = expo(As, -dd[None, :]).max(1), expo(vs, dd).max()
        sa, sv = 62 - ea[:, None] - dd[None, :], 62 - ev + dd
        ar, ai, vr, vi = (digits(cut(x, s)) for x, s in ((As.real, sa), (As.imag, sa), (vs.real, sv), (vs.imag, sv)))
        y = [0, 0]
        for i in range(8):
            for j in range(8 - i):
                y[0] = y[0] + (ar[i] @ vr[j] - ai[i] @ vi[j]).astype(object) * 256 ** (7 - i - j)
                y[1] = y[1] + (ai[i] @ vr[j] + ar[i] @ vi[j]).astype(object) * 256 ** (7 - i - j)

        def value(t, e):   # (times 2^56) the 63 bits that are kept, to the nearest double
            s = 12 if abs(t) >> 62 else 0
            return float(Fraction(t >> s) * Fraction(2) ** (s + 56 - 124 + int(e)))

        total += [complex(value(int(a), e + ev), value(int(b), e + ev)) for a, b, e in zip(*y, ea)]
    return total


# source layer's k, target layer's (None: the same), the other layer's; k_max (cell width w); source and
# target heights over w; part of the cell that holds the sources
@pytest.mark.parametrize("ks,kt,k2,kw,hs,ht,part", [
    (1.97, None, 7.74, 5.2, 0.0, 0.0, 0.5), (1.97, None, 7.74, 7.8, 0.0, 0.0, 1.0), (1.2, None, 5.2, 9.0, 0.0, 0.0, 0.25),
    (1.13, None, 9.97, 10.3, 0.0, 0.0, 0.5), (2.0, None, 8.0, 14.0, 0.0, 0.0, 0.1), (2.55, None, 8.02, 29.8, 0.25, 0.25, 0.25),
    (2.0, None, 8.0, 32.0, 0.27, 0.27, 0.5), (4.0, None, 8.0, 24.0, 0.16, 0.16, 0.25), (4.0, None, 8.0, 48.0, 0.33, 0.33, 0.5),
    (4.0, None, 8.0, 24.0, 0.42, 0.42, 0.25), (7.5, None, 8.0, 44.0, 0.2, 0.2, 0.5), (8.0, None, 2.0, 48.0, 0.2, 0.2, 0.25),
    (2.0, 8.0, 8.0, 16.0, 0.0, 0.6, 0.25), (4.0, 8.0, 8.0, 24.0, 0.1, 0.5, 0.5), (8.0, 2.0, 8.0, 16.0, 0.6, 0.0, 0.25),
    (8.0, 4.0, 8.0, 24.0, 0.1, 0.5, 0.1), (5.4, 8.0, 8.0, 20.0, 0.0, 0.25, 0.5), (2.0, 8.0, 8.0, 12.0, 0.5, 0.5, 0.25)])
def test_products_keep_fp64_accuracy(segment_size, ks, kt, k2, kw, hs, ht, part):
    kmax = max(ks, k2)
    w, kr, T = kw / kmax, kw * np.sqrt(0.5), kmax + 0.75
    p = max(20, int(np.ceil(kr + 9 * kr ** (1 / 3))))
    # pairs two cells apart are admitted where this holds
    assert np.sqrt(T * T - min(ks, kt or ks) ** 2) * w * (1 - hs - ht) <= 16.0
    A = reaction_table(ks, kt, k2, hs * w, ht * w, 2 * w, p, T)
    rng = np.random.default_rng(int(1000 * kw))
    n = np.arange(-p, p + 1)

    def polar(part):
        z = (rng.uniform(-0.5, 0.5, 64) + 1j * rng.uniform(-0.5, 0.5, 64)) * w * part
        return np.abs(z)[:, None], np.angle(z)[:, None]

    rho, th = polar(part)
    q = rng.standard_normal(64) + 1j * rng.standard_normal(64)
    M = q @ (jv(n, ks * rho) * np.exp(-1j * n * th))
    rho, th = polar(1.0)
    J = jv(n, (kt or ks) * rho) * np.exp(1j * n * th)
    env = np.maximum.accumulate(np.abs(jv(np.arange(p + 1), ks * w * np.sqrt(0.5)))[::-1])[::-1]
    d = -np.floor(np.log2(env)).astype(int)

    F = lambda x: Fraction(float(x))   # noqa: E731
    Mr, Mi = [F(z.real) for z in M], [F(z.imag) for z in M]
    size = segment_size(p, ks, kt or ks, kmax, T, w, hs * w, ht * w, 0.0)
    L = split_product(A, M, d, size, p)
    off = np.empty(2 * p + 1, complex)
    for r in range(2 * p + 1):
        ar, ai = [F(z.real) for z in A[r]], [F(z.imag) for z in A[r]]
        re = sum(a * x - b * y for a, b, x, y in zip(ar, ai, Mr, Mi))
        im = sum(a * y + b * x for a, b, x, y in zip(ar, ai, Mr, Mi))
        off[r] = complex(F(L[r].real) - re, F(L[r].imag) - im)
    # an FP64 sum of 2 (2p + 1) products is off by up to (4p + 4) 2^-53 of its terms' magnitudes;
    # here 4 of them
    assert np.abs(J @ off).max() <= 4 * 2.0 ** -53 * (np.abs(J) @ (np.abs(A) @ np.abs(M))).max()
