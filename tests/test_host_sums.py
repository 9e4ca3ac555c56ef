"""The host/device arithmetic of the kernels' sums, compiled for the host."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2004_08146_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
FP = ctypes.POINTER(ctypes.c_float)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("host") / "host_sums.so")
    try:
        subprocess.run([build.nvcc(), "-shared", "-O2", "-std=c++17", "-Xcompiler", "-fPIC,-ffp-contract=off",
                        "--expt-relaxed-constexpr", "-I", build.CSRC, os.path.join(HERE, "host_sums.cu"), "-o", so]
                       + build.ARCH, check=True, capture_output=True, text=True)
    except FileNotFoundError:
        pytest.skip("no nvcc")
    return ctypes.CDLL(so)


def ptr(a):
    return a.ctypes.data_as(FP)


def test_inner_products_round_the_running_sum_once(lib):
    """Sums of 400 complex products of Gaussian numbers: as close to the exact ones
    as products added one by one, to 3 % (a hundred sums of many roundings each)."""
    rng = np.random.default_rng(3)
    a, b = (rng.standard_normal((400, 400, 2)).astype(np.float32) for _ in range(2))
    out = np.empty((400, 2), dtype=np.float32)
    lib.host_cdot(ptr(a), ptr(b), 400, 400, ptr(out))
    ca, cb = a[..., 0] + 1j * a[..., 1], b[..., 0] + 1j * b[..., 1]
    plain = np.zeros(400, dtype=np.complex64)
    for t in range(400):
        plain = plain + (ca[:, t].conj() * cb[:, t]).astype(np.complex64)
    exact = np.sum(ca.astype(np.complex128).conj() * cb.astype(np.complex128), axis=1)
    err = [np.linalg.norm(v - exact) / np.linalg.norm(exact) for v in (out[:, 0] + 1j * out[:, 1], plain)]
    assert err[0] <= 1.03 * err[1], err


def test_double_float_sums_keep_fp64(lib):
    """Partial sums of double-floats passed from stage to stage with all three parts
    stay within a rounding of FP64 (2^-53) of the sum of the absolute values; rounded
    to double-floats in between they do not (2^-49 of it and less, rms)."""
    lib.host_stage_sum.restype = ctypes.c_double
    rng = np.random.default_rng(5)
    worst = [0.0, 0.0]
    for _ in range(20):
        v = rng.standard_normal((12, 8, 32)) ** 2          # a squared norm: no cancellation
        h = v.astype(np.float32)
        hl = np.stack([h, (v - h).astype(np.float32)], axis=-1)
        exact = np.sum(hl.astype(np.longdouble))
        for keep in (0, 1):
            d = abs(np.longdouble(lib.host_stage_sum(ptr(np.ascontiguousarray(hl)), 12, keep)) - exact)
            worst[keep] = max(worst[keep], float(d / exact))
    assert worst[1] <= 2.0 ** -53 < worst[0], worst
