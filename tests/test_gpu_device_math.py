"""Device functions that take the place of CUDA's division and tanh, against
64 bits."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2212_14153_gb300 import build
    so = str(tmp_path_factory.mktemp("math") / "device_math.so")
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I" + build.CSRC, "-shared", "-o", so,
                    os.path.join(HERE, "device_math.cu")], check=True)
    return ctypes.CDLL(so)


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def test_fp64_reciprocal_of_a_density(lib):
    # one rounding (half an ulp) and the third-order remainder of a seed of
    # relative error e < 2^-19: e^3 = 2^-57, a sixteenth of an ulp at most
    # (an ulp is 2^-53 of a value just below a power of two); e itself carries
    # roundings of 2^-53 of it, far below that
    rng = np.random.default_rng(1)
    x = np.concatenate([rng.uniform(0.5, 2.0, 1_000_000), 1.0 + rng.normal(0, 1e-3, 1_000_000),
                        1.0 + np.arange(-64, 65) * 2.0 ** -53, [0.5, 1.0, 2.0]])
    y = np.empty_like(x)
    assert lib.recip_f64(_p(x), _p(y), len(x)) == 0
    # the error in ulps of the quotient: x y - 1 in extended precision
    err = np.abs((x.astype(np.longdouble) * y - 1) / x) / np.spacing(1.0 / x)
    if np.finfo(np.longdouble).nmant < 60:
        pytest.skip("no extended precision")
    print(f"FP64 reciprocal: {float(err.max()):.4f} ulp at most, {100 * np.mean(y == 1.0 / x):.3f} % correctly rounded")
    assert err.max() <= 0.5 + 1.0 / 16


@pytest.mark.parametrize("a,xi", [(2.0, 0.5), (2.5, 0.625), (3.3, 0.1), (4.0, 1.0), (8.0, 0.25), (8.0, 0.5),
                                  (12.0, 0.36), (3.0, 0.0625), (1.0, 8.0), (4.0, 2.0)])
def test_fp32_profile(lib, a, xi):
    # phi = 1 / (1 + e^z), z = 2 (r - a) / xi.  Its roundings in units of 2^-24:
    # nine or so of z as a whole (approximate square root, reciprocal and power
    # of two within two each), which count z phi (1 - phi) <= 0.23; the power of
    # two's four, which count 1/4; one of the sum and two of the last reciprocal:
    # 6 2^-24 = 3.6e-7.  And r^2 - a^2, of terms up to about a^2 where phi is
    # steep, each rounded at 2^-24 of itself: two, over r + a = 2 a, at a slope of
    # 1 / (2 xi): 2^-24 a / (2 xi).  On profiles at most a quarter of the radius
    # wide, as runs have them, it is no further off than through tanhf.
    rng = np.random.default_rng(2)
    n = 1_000_000
    rc = a + 8.0 * xi
    # over the support, and as many where the profile is steep
    r = np.concatenate([rc * np.sqrt(rng.uniform(0, 1, n)), a + 2.0 * xi * rng.uniform(-1, 1, n)])
    t = rng.uniform(0, 2 * np.pi, 2 * n)
    dx, dy = (r * np.cos(t)).astype(np.float32), (r * np.sin(t)).astype(np.float32)
    fa, fi, f2 = np.float32(a), np.float32(1.0 / xi), np.float32(rc * rc)
    out, plain = np.empty_like(dx), np.empty_like(dx)
    assert lib.phi_f32(_p(dx), _p(dy), ctypes.c_float(fa), ctypes.c_float(fi), ctypes.c_float(f2), _p(out), _p(plain),
                       2 * n) == 0
    r64 = np.hypot(dx.astype(np.float64), dy.astype(np.float64))
    want = 0.5 * (np.tanh((float(fa) - r64) * float(fi)) + 1.0)
    inside = (out != 0) & (plain != 0)
    assert inside.mean() > 0.5
    rms, top = {}, {}
    for name, v in (("logistic", out), ("tanh", plain)):
        e = (v.astype(np.float64) - want)[inside]
        rms[name], top[name] = float(np.sqrt(np.mean(e * e))), float(np.abs(e).max())
    print(f"a = {a}, xi = {xi}: rms {rms['logistic']:.2e} (tanh {rms['tanh']:.2e}), largest {top['logistic']:.2e} "
          f"({top['tanh']:.2e})")
    assert top["logistic"] <= 2.0 ** -24 * (6.0 + a / (2.0 * xi))
    if xi <= a / 4.0:
        assert rms["logistic"] <= rms["tanh"] and top["logistic"] <= top["tanh"]
