"""Line plans and register DFTs of the spectral solve (csrc/spectral.cuh) run on
the host, in both plan kinds: the wide plans (FP64 boxes and boxes of many
cells) and the narrow plans (the other FP32 boxes), and the passes of the
preconditioner on them.

Bounds: a DFT of R points as the library forms it takes at most R + 4
additions and products on the way to each output (two factors for a composite
R, whose sum is smaller), each rounded relative to a partial sum that the sum
of the magnitudes bounds: (R + 4) u sum |v|, doubled for the two parts.  A line
of stages R_1 .. R_m adds the bounds of its stages and one rounding per
twiddle product."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1712_08494_gb300", "csrc")
DFTS = (2, 3, 4, 5, 6, 7, 8, 9, 10, 12, 14, 15, 16)
LENGTHS = (2, 3, 5, 6, 7, 9, 10, 14, 15, 16, 21, 25, 28, 32, 35, 45, 49, 60, 63, 64, 72, 75, 84, 96, 100, 105, 120,
           128, 147, 180, 210, 225, 243, 245, 256, 320, 343, 384, 420, 448, 480, 486, 500, 512)


@pytest.fixture(scope="module")
def spec(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    out = str(tmp_path_factory.mktemp("plans") / "libspec_host.so")
    subprocess.run([gxx, "-O2", "-shared", "-fPIC", "-I", CSRC, "-o", out, os.path.join(HERE, "spectral_host.cpp")],
                   check=True, capture_output=True)
    lib = C.CDLL(out)
    for f in (lib.small_dft, lib.small_dft_f32):
        f.argtypes = [C.c_void_p, C.c_void_p, C.c_int]
    for f in (lib.plan_line, lib.plan_line_f32):
        f.argtypes = [C.c_void_p, C.c_void_p, C.c_int, C.c_int]
    lib.plan_stages.argtypes = [C.c_int, C.c_int, C.c_void_p]
    lib.box_form.argtypes = [C.c_int] * 3
    lib.precond_plan.argtypes = [C.c_void_p, C.c_int, C.c_int, C.c_int, C.c_int, C.c_double, C.c_int, C.c_int]
    return lib


def _complex(rng, n, prec):
    x = (rng.uniform(-1, 1, n) + 1j * rng.uniform(-1, 1, n)).astype(np.complex64 if prec == "fp32" else np.complex128)
    return x, np.zeros_like(x), 2.0 ** -24 if prec == "fp32" else 2.0 ** -53


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("R", DFTS)
def test_register_dft(spec, R, prec):
    x, y, u = _complex(np.random.default_rng(R), R, prec)
    assert (spec.small_dft_f32 if prec == "fp32" else spec.small_dft)(x.ctypes.data, y.ctypes.data, R) == 0
    ref = np.fft.fft(x.astype(np.complex128))
    assert np.abs(y - ref).max() <= 2 * (R + 4) * u * np.abs(x).sum()


def _radices(spec, n, wide):
    rad = (C.c_int * 12)()
    return list(rad[:spec.plan_stages(n, wide, rad)])


@pytest.mark.parametrize("wide", [0, 1])
def test_radices(spec, wide):
    allowed = set(DFTS) if wide else {2, 3, 4, 5, 7, 8}
    seen = set()
    for n in range(2, 513):
        rad = _radices(spec, n, wide)
        m = n
        for p in (2, 3, 5, 7):
            while m % p == 0:
                m //= p
        assert bool(rad) == (m == 1), n  # both kinds take the same lengths
        if rad:
            assert np.prod(rad) == n and set(rad) <= allowed, (n, rad)
            seen |= set(rad)
    assert seen == allowed


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("wide", [0, 1])
def test_lines(spec, wide, prec):
    rng = np.random.default_rng(wide)
    for n in LENGTHS:
        x, y, u = _complex(rng, n, prec)
        assert (spec.plan_line_f32 if prec == "fp32" else spec.plan_line)(x.ctypes.data, y.ctypes.data, n, wide) == 0
        ref = np.fft.fft(x.astype(np.complex128))
        roundings = sum(2 * (R + 4) + 4 for R in _radices(spec, n, wide))
        assert np.abs(y - ref).max() <= roundings * u * np.abs(x).sum(), n


def _lap(z):
    out = -6.0 * z
    for ax in range(3):
        out += np.roll(z, 1, ax) + np.roll(z, -1, ax)
    return out


@pytest.mark.parametrize("wide", [0, 1])
@pytest.mark.parametrize("W", [32, 16, 8])
def test_passes_invert_the_laplacian(spec, W, wide):
    """Bounds of the test of the wide plans' passes in test_spectral_host."""
    rng = np.random.default_rng(W + wide)
    for nz, ny, nx in ((16, 16, 16), (24, 40, 56), (32, 32, 48), (6, 10, 15), (7, 5, 9), (25, 21, 35), (9, 49, 30)):
        r = rng.normal(size=(nz, ny, nx)).astype(np.float32)
        z = r.copy()
        assert spec.precond_plan(z.ctypes.data, 0, nx, ny, nz, 0.3, W, wide) == 0
        res = 0.3 * _lap(z.astype(np.float64)) - (r - r.mean())
        assert np.abs(res).max() < 2e-5 * np.abs(r).max(), (nz, ny, nx)
        r64 = r.astype(np.float64)
        z64 = r64.copy()
        assert spec.precond_plan(z64.ctypes.data, 1, nx, ny, nz, 0.3, W, wide) == 0
        res = 0.3 * _lap(z64) - (r64 - r64.mean())
        assert np.abs(res).max() < 1e-12 * np.abs(r64).max(), (nz, ny, nx)


# steps of FP32 boxes of at least 2^20 cells, us: (small form, large form)
FORMS = {
    (128, 128, 128): (681, 657), (128, 128, 384): (1993, 1908), (192, 128, 128): (1065, 980),
    (96, 96, 128): (598, 523), (144, 144, 144): (1261, 1141), (120, 120, 120): (832, 764),
    (150, 150, 150): (1436, 1343), (105, 105, 105): (714, 701), (128, 432, 128): (2346, 2227),
    (128, 450, 128): (2406, 2283), (504, 128, 128): (2835, 2681), (128, 128, 512): (2510, 2783),
    (128, 512, 128): (2541, 2731), (125, 128, 128): (794, 885), (81, 128, 128): (634, 701),
    (175, 175, 175): (2620, 2732), (512, 512, 32): (2774, 3031), (512, 16, 512): (1666, 1929),
    (343, 64, 64): (649, 712), (375, 128, 128): (2142, 2307), (100, 128, 128): (690, 708),
    (128, 128, 175): (1027, 1079), (270, 128, 128): (1627, 1702), (128, 225, 128): (1166, 1147),
}


def test_form_of_a_box(spec):
    """Within 3% of the faster form; smaller boxes take the small form."""
    for b, t in FORMS.items():
        assert t[spec.box_form(*b)] <= 1.03 * min(t), b
    for b in ((96, 96, 96), (101, 101, 101), (64, 64, 64), (32, 32, 512), (125, 64, 64)):
        assert spec.box_form(*b) == 0, b
