"""The fundamental solution in 64-bit fixed point (csrc/phi_fx.h), compiled for
the host, against 40-digit mpmath.  The device's FP32 reciprocal roots are
accurate to 2^-22.9; the host's are given errors of up to 4 * 2^-24.

Bounds.  e^{2 pi i theta} at 2^62: the steps' tables end at 2^-62, the products
at 2^-57 (the 24-bit sine correction): 2e-17 with room.  phi: distances are
fractions of 2^e with an error of a few 2^-62, so phases carry kappa 2^e 2^-60
or so; amplitudes end near 2^-51 (w is kept at 2^-51): kappa 2^e 2^-58 + 2e-15."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HARNESS = os.path.join(ROOT, "tests", "phi_fx_harness.cpp")
mp = pytest.importorskip("mpmath")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    out = tmp_path_factory.mktemp("phifx") / "libphifx_test.so"
    subprocess.run([gxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-DFX_RSQRT_ULP=8", HARNESS, "-o", str(out)],
                   check=True, capture_output=True)
    return ctypes.CDLL(str(out))


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def test_cis_at_and_between_the_steps(lib):
    mp.mp.dps = 40
    rng = np.random.default_rng(0)
    th = []
    for k in list(range(0, 1024, 31)) + [255, 256, 511, 512, 1023]:
        at = k << 54
        for d in (0, 1, -1, 2, 1 << 27, -(1 << 27), 1 << 31, -(1 << 31), (1 << 32) + 7, 1 << 40,
                  (1 << 53) - 1, -(1 << 53), -(1 << 53) + 1):
            th.append((at + d) % (1 << 64))
    th += [int(x) for x in rng.integers(0, 1 << 63, 300)]
    t = np.array(th, dtype=np.uint64)
    c, s = np.zeros(len(t), np.int64), np.zeros(len(t), np.int64)
    lib.cis_fx_batch(len(t), _p(t), _p(c), _p(s))
    for i, x in enumerate(th):
        a = 2 * mp.pi * mp.mpf(x) / mp.mpf(2) ** 64
        assert abs(mp.mpf(int(c[i])) / mp.mpf(2) ** 62 - mp.cos(a)) < 1e-16, x
        assert abs(mp.mpf(int(s[i])) / mp.mpf(2) ** 62 - mp.sin(a)) < 1e-16, x


@pytest.mark.parametrize("dim,kappa,lo,hi", [(3, 3.0, 1.2, 8), (3, 8.0, 1.2, 60), (3, 40.0, 2, 200), (2, 10.0, 1.3, 14),
                                             (2, 40.0, 1.2, 4), (2, 40.0, 3, 150), (2, 200.0, 1.26, 2000),
                                             (2, 6.0, 1.3, 6), (3, 0.01, 1.3, 50)])
def test_phi_fixed_point(lib, dim, kappa, lo, hi):
    """Targets from just outside a body's radius to far away: every fit of H0,
    every left shift of the phase, every scaling of the amplitude."""
    mp.mp.dps = 40
    rng = np.random.default_rng(int(kappa * 7) + dim)
    n = 160
    rho = rng.uniform(0.55, 1.1, n)
    R = rho * np.exp(rng.uniform(np.log(lo), np.log(hi), n))
    u, w = rng.normal(size=(n, dim)), rng.normal(size=(n, dim))
    D = np.ascontiguousarray(R[:, None] * u / np.linalg.norm(u, axis=1)[:, None])
    delta = w / np.linalg.norm(w, axis=1)[:, None] * (rho * rng.uniform(0, 1, n))[:, None]
    es = np.array([int(np.frexp(r * (1 + 1e-6))[1]) for r in rho], np.int32)
    dj = np.array([[int(np.rint(d * 2.0 ** (63 - e))) for d in row] for row, e in zip(delta, es)], dtype=np.int64)
    out, ok, raw = np.zeros((n, 2)), np.zeros(n, np.int32), np.zeros((n, 2), np.int64)
    lib.phi_fx_batch(dim, ctypes.c_double(kappa), n, _p(D), _p(rho), _p(es), _p(dj), _p(out), _p(ok), _p(raw))
    assert (ok == 1).sum() > n // 3  # the formats hold most bodies
    for i in np.nonzero(ok == 1)[0]:
        d = [mp.mpf(float(D[i, a])) - mp.mpf(int(dj[i, a])) / mp.mpf(2) ** (63 - int(es[i])) for a in range(dim)]
        r = mp.sqrt(sum(x * x for x in d))
        ref = (mp.mpc(0, mp.mpf(1) / 4) * mp.hankel1(0, kappa * r) if dim == 2
               else mp.exp(mp.mpc(0, 1) * kappa * r) / (4 * mp.pi * r))
        err = float(abs(mp.mpc(float(out[i, 0]), float(out[i, 1])) - ref) / abs(ref))
        scale = 2.0 ** np.ceil(np.log2((R[i] + rho[i]) * 1.0001))
        assert err < 2e-15 + kappa * scale * 2.0 ** -58, (i, float(kappa * r))
        assert np.abs(raw[i]).max() <= 1.01 * 2 ** 59  # the sums' headroom
    if dim == 2:  # below kappa r = 4 the caller takes the series
        for i in np.nonzero(ok == 2)[0]:
            d = [float(D[i, a]) - float(dj[i, a]) / 2.0 ** (63 - int(es[i])) for a in range(dim)]
            assert kappa * np.linalg.norm(d) < 4.0 * (1 + 1e-9)


def test_bodies_outside_the_formats_are_refused(lib):
    """Targets at or inside the hull's fifteenth, extreme sizes and kappas."""
    cases = [(2, 10.0, [1.0, 0.0], 1.0), (2, 10.0, [1.05, 0.0], 1.0), (2, 10.0, [0.2, 0.0], 1.0), (2, 1e-6, [4.0, 0.0], 1.0),
             (2, 1e14, [4.0, 0.0], 1.0), (3, 1e14, [4.0, 0.0, 0.0], 1.0), (3, 3.0, [1e100, 0.0, 0.0], 1.0),
             (2, 3.0, [np.inf, 0.0], 1.0), (2, 3.0, [np.nan, 0.0], 1.0)]
    for dim, kappa, D, rho in cases:
        D, r = np.array([D]), np.array([rho])
        es, dj = np.array([1], np.int32), np.zeros((1, dim), np.int64)
        out, ok, raw = np.zeros((1, 2)), np.ones(1, np.int32), np.zeros((1, 2), np.int64)
        lib.phi_fx_batch(dim, ctypes.c_double(kappa), 1, _p(D), _p(r), _p(es), _p(dj), _p(out), _p(ok), _p(raw))
        assert ok[0] == 0, (dim, kappa, D)


@pytest.mark.parametrize("kappa,hi", [(0.01, 50), (1.0, 8)])
def test_phi_near_bodies_at_low_frequency(lib, kappa, hi):
    """3D, where the phase carries no error and the modulus all of it.  The result
    is rounded to FP64 twice (2.2e-16 together), its scale once (1.1e-16), and the
    integers end at 2^-56 of the nearest point's amplitude or 2^-54 of the farthest's
    (5.6e-17): 4e-16, which plain FP64 does not stay below."""
    mp.mp.dps = 40
    rng = np.random.default_rng(5)
    n = 1500
    rho = rng.uniform(0.55, 1.1, n)
    R = rho * np.exp(rng.uniform(np.log(1.3), np.log(hi), n))
    u, w = rng.normal(size=(n, 3)), rng.normal(size=(n, 3))
    D = np.ascontiguousarray(R[:, None] * u / np.linalg.norm(u, axis=1)[:, None])
    delta = w / np.linalg.norm(w, axis=1)[:, None] * (rho * rng.uniform(0, 1, n))[:, None]
    es = np.array([int(np.frexp(r * (1 + 1e-6))[1]) for r in rho], np.int32)
    dj = np.array([[int(np.rint(d * 2.0 ** (63 - e))) for d in row] for row, e in zip(delta, es)], dtype=np.int64)
    out, ok, raw = np.zeros((n, 2)), np.zeros(n, np.int32), np.zeros((n, 2), np.int64)
    lib.phi_fx_batch(3, ctypes.c_double(kappa), n, _p(D), _p(rho), _p(es), _p(dj), _p(out), _p(ok), _p(raw))
    assert (ok == 1).sum() > n // 2
    for i in np.nonzero(ok == 1)[0]:
        r = mp.sqrt(sum((mp.mpf(float(D[i, a])) - mp.mpf(int(dj[i, a])) / mp.mpf(2) ** (63 - int(es[i]))) ** 2 for a in range(3)))
        ref = mp.exp(mp.mpc(0, 1) * kappa * r) / (4 * mp.pi * r)
        err = float(abs(mp.mpc(float(out[i, 0]), float(out[i, 1])) - ref) / abs(ref))
        assert err < 4e-16 + kappa * 2.0 ** (np.ceil(np.log2((R[i] + rho[i]) * 1.0001)) - 58), i


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("size", [1e-25, 1e-20, 1e-16, 1e17, 1e20])
def test_bodies_whose_squared_distance_leaves_fp32_are_refused(lib, dim, size):
    """|D| is a root of FP32 squares: below 1e-19 they have lost their digits, above
    1e19 they overflow.  Bodies of any size between keep the formats."""
    kappa, D, r = 30.0 / size, np.zeros((1, dim)), np.array([size])
    D[0, 0] = 4.0 * size
    es, dj = np.array([int(np.frexp(size * (1 + 1e-6))[1])], np.int32), np.zeros((1, dim), np.int64)
    out, ok, raw = np.zeros((1, 2)), np.ones(1, np.int32), np.zeros((1, 2), np.int64)
    lib.phi_fx_batch(dim, ctypes.c_double(kappa), 1, _p(D), _p(r), _p(es), _p(dj), _p(out), _p(ok), _p(raw))
    assert ok[0] == (1 if 1e-17 < size < 1e18 else 0)


def test_fits_are_the_generators():
    """The coefficients for kappa r >= 64 are what their generator gives."""
    import re
    import sys
    csrc = os.path.join(ROOT, "paper_2603_19113_gb300", "csrc")
    sys.path.insert(0, csrc)
    try:
        import gen_bessel_coeffs as gen
    finally:
        sys.path.remove(csrc)
    text = open(os.path.join(csrc, "bessel_coeffs.h")).read()
    for lab, want in zip("FG", gen.fx_fit()):
        got = re.search(r"MBS_FX_X64_%s \{(.*)\}" % lab, text).group(1)
        assert [float(c) for c in got.split(",")] == want
