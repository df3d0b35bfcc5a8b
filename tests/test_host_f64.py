"""Parts of the device arithmetic, compiled for the host: FP64 sums against
extended arithmetic, and step scalars in any unit of time."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "hostmath")
ROOT = os.path.dirname(os.path.dirname(HERE))
CSRC = os.path.join(ROOT, "paper_2601_02527_gb300", "csrc")
EPS = 2.0 ** -53
D = ctypes.c_double


@pytest.fixture(scope="module")
def lib():
    src = os.path.join(HERE, "gpss_f64_harness.cu")
    out = os.path.join(HERE, "_build", "libgpss_f64.so")
    os.makedirs(os.path.dirname(out), exist_ok=True)
    deps = [src] + [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cuh")]
    if not os.path.exists(out) or os.path.getmtime(out) < max(map(os.path.getmtime, deps)):
        tmp = out + f".tmp{os.getpid()}"
        subprocess.check_call(["/usr/local/cuda/bin/nvcc", "-O2", "-std=c++17", "-Xcompiler",
                               "-fPIC", "-shared", "-I", os.path.join(ROOT, "include"), "-I",
                               CSRC, src, "-o", tmp])
        os.replace(tmp, out)
    lib = ctypes.CDLL(out)
    lib.hf_prod_tally.argtypes = [D, D, D, D, ctypes.POINTER(D)]
    lib.hf_plain64_scalars.argtypes = [D, D, D, ctypes.POINTER(D)]
    f = ctypes.c_float
    lib.hf_prod_dual.argtypes = [f, f, f, ctypes.c_int, ctypes.POINTER(D)]
    return lib


def test_product_sums_keep_double_precision(lib):
    # at most eight roundings of half a unit each, of the terms' size
    assert np.finfo(np.longdouble).eps < 2.0 ** -60
    rng = np.random.default_rng(0)
    L = np.longdouble
    for _ in range(4000):
        S = float(np.float32(np.exp(rng.uniform(-60, 60))))
        e = float(np.float32(np.sqrt(S) * rng.standard_normal()))
        dS = float(np.float32(S * rng.standard_normal() * 10.0 ** rng.uniform(-3, 3)))
        de = float(np.float32(e * rng.standard_normal() * 10.0 ** rng.uniform(-3, 3)))
        out = (D * 2)()
        lib.hf_prod_tally(S, dS, e, de, out)
        ll = [np.log(L(S)), L(e) * e / S]
        d = [L(dS) / S, -L(e) * e * dS / (L(S) * S), 2 * L(e) * de / S]
        assert abs(L(out[0]) - sum(ll)) <= 8 * EPS * sum(map(abs, ll))
        assert abs(L(out[1]) - sum(d)) <= 8 * EPS * sum(map(abs, d))


@pytest.mark.parametrize("q", [0.2, 0.5, 0.7, 8.0])
@pytest.mark.parametrize("x", [1e-3, 0.3, 0.99, 1.7, 30.0])  # omega0 t: Taylor and closed branches
@pytest.mark.parametrize("k", [-120, -60, -7, 7, 60, 120])
def test_plain64_scalars_in_any_unit_of_time(lib, q, x, k):
    # times in units of 2^k: every scalar scales by a power of two, exactly
    def scalars(u):
        w0 = 0.7 / u
        a = w0 / (2 * q)
        beta = 0.0 if q == 0.5 else w0 * w0 * (1 - 1 / (4 * q * q))
        out = (D * 6)()
        lib.hf_plain64_scalars(x / w0, a, beta, out)
        return np.array(out)

    u = 2.0 ** k
    one = scalars(1.0)
    assert np.all(np.isfinite(one)) and np.all(one[3:] > 0)  # the integrals of squares
    assert np.array_equal(scalars(u), one * [u, 1.0, u ** 2, u ** 3, u, u ** 5])


@pytest.mark.parametrize("q", [0.2, 0.5, 0.7, 8.0])
@pytest.mark.parametrize("x", [0.1, 1.1, 1.7, 30.0])
@pytest.mark.parametrize("which", [0, 1])
@pytest.mark.parametrize("k", [-24, -10, 10, 24])
def test_product_tangents_in_any_unit_of_time(lib, q, x, which, k):
    # FP32 scalars and the tangent with respect to omega0 or Q scale by powers
    # of two, exactly (d I_ff / d omega0 is of the size 2^(4 k))
    def scalars(u):
        out = (D * 8)()
        w0 = float(np.float32(0.7)) / u
        lib.hf_prod_dual(float(np.float32(x / 0.7)) * u, w0, q, which, out)
        return np.array(out)

    u = 2.0 ** k
    one = scalars(1.0)
    assert np.all(np.isfinite(one)) and np.all(one[4:6] != 0)
    size = np.array([u, 1.0, u ** 3, u])
    assert np.array_equal(scalars(u), one * np.concatenate([size, size * (u if which == 0 else 1)]))
