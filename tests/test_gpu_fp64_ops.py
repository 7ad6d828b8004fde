"""The FP64 exponential, reciprocal and argument of fp64_ops.cuh, one by one, against extended precision
and against CUDA's functions outside their ranges."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
L = np.longdouble


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_1312_4698_gb300 import build as B
    lib = str(tmp_path_factory.mktemp("fp64_ops") / "probe.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "fp64_ops_probe.cu")
    subprocess.run([B.nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-shared", "-o", lib, src, "-lcudart"], check=True)
    fn = ctypes.CDLL(lib).probe
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int]

    def run(x, y=None):
        x = np.ascontiguousarray(x, dtype=np.float64)
        y = np.ones_like(x) if y is None else np.ascontiguousarray(y, dtype=np.float64)
        out = np.empty((6, x.size))
        assert fn(x.ctypes.data, y.ctypes.data, out.ctypes.data, x.size) == 0
        return out
    return run


def _ulps(got, ref):
    """Error in units of the last place of the exact value."""
    r = np.abs(ref.astype(np.float64))
    return (np.abs(got.astype(L) - ref) / np.spacing(r).astype(L)).astype(np.float64)


def _report(name, own, cuda):
    print(f"{name}: max {own.max():.4g} rms {np.sqrt((own ** 2).mean()):.4g}, CUDA's {cuda.max():.4g} {np.sqrt((cuda ** 2).mean()):.4g}")


def test_exponential(probe):
    """0.5 ulp for the last addition; behind it |e^r - 1| <= 0.0055 carries its roundings (4 of half an ulp of
    itself) and the table's trailing word one of 2^-107: 0.52."""
    assert np.finfo(L).eps < 1e-18
    rng = np.random.default_rng(1)
    k = np.arange(-60000, 60000)
    edge = (k + 0.5) * np.log(2.0) / 64          # |r| at its largest
    x = np.concatenate([rng.uniform(-40, 40, 400000), rng.uniform(-703.9, 703.9, 400000), edge, np.nextafter(edge, 0),
                        k * np.log(2.0) / 64, [46.41374557698667, -49.93373218640315, 0.0, -0.0, 1e-300, 703.99, -703.99]])
    out = probe(x)
    own, cuda = _ulps(out[0], np.exp(x.astype(L))), _ulps(out[1], np.exp(x.astype(L)))
    _report("exp", own, cuda)
    assert own.max() <= 0.52
    # beyond: CUDA's function, the same bits
    x = np.array([704.0, -704.0, 709.7, 709.8, -708.5, -745.0, -746.0, 1e5, -1e5, np.inf, -np.inf, np.nan])
    out = probe(x)
    assert np.array_equal(out[0], out[1], equal_nan=True)


def test_reciprocal(probe):
    """e = 1 - x r to 2^-53 of itself (2^-73), its square's remainder e^3 below 2^-58: 0.5 ulp and 2^-5 of one
    at worst; the division's result wherever that rounds alike."""
    rng = np.random.default_rng(2)
    x = np.concatenate([rng.uniform(1, 2, 400000), rng.normal(size=400000) * 10.0 ** rng.uniform(-280, 280, 400000),
                        1.0 + np.arange(2000) * 2.0 ** -52, 2.0 - np.arange(1, 2000) * 2.0 ** -52])
    out = probe(x)
    own, cuda = _ulps(out[2], 1 / x.astype(L)), _ulps(out[3], 1 / x.astype(L))
    _report("reciprocal", own, cuda)
    print(f"other than the division's: {np.mean(out[2] != out[3]):.2e}")
    assert own.max() <= 0.5 + 2.0 ** -5
    x = np.array([0.0, -0.0, 5e-324, -1e-310, 2.3e-308, 1e-290, 1.7e308, -1e307, np.inf, -np.inf, np.nan])
    out = probe(x)
    assert np.array_equal(out[2], out[3], equal_nan=True)


def test_argument(probe):
    """t = v / u is off by the roundings of v's two products and its table words (3 * 2^-53) and of the
    quotient and series (2^-57), k pi / 64 by 2^-54 of at most pi / 2 and its sum by 2^-53, and the
    reflection at pi by 2^-53 (pi's own rounding) and 2^-52: 7.8 * 2^-53, 8.7e-16.  CUDA's atan2 is
    within 2 ulp, 8.9e-16 in the last octant."""
    rng = np.random.default_rng(3)
    th = np.concatenate([rng.uniform(-np.pi, np.pi, 400000), (np.arange(-128, 128) + 0.5) * np.pi / 64,
                         np.arange(-64, 65) * np.pi / 64, rng.normal(size=20000) * 10.0 ** rng.uniform(-30, 0, 20000)])
    m = 10.0 ** rng.uniform(-200, 200, th.size)
    x, y = m * np.cos(th), m * np.sin(th)
    ref = np.arctan2(y.astype(L), x.astype(L))
    out = probe(x, y)
    own, cuda = np.abs(out[4].astype(L) - ref).astype(float), np.abs(out[5].astype(L) - ref).astype(float)
    _report("argument (absolute)", own, cuda)
    assert own.max() <= 8.7e-16
    small = np.abs(ref) < 1e-3
    assert (own[small] <= 8 * 2.0 ** -53 * np.abs(ref[small].astype(float))).all()
    x = np.array([1.0, -1.0, 0.0, 0.0, 0.0, -0.0, 1.0, -1.0, 1e-320, np.nan, 1.0, np.inf, -np.inf])
    y = np.array([0.0, 0.0, 1.0, -1.0, 0.0, 0.0, -0.0, -0.0, 1e-320, 1.0, np.nan, 1.0, 1.0])
    out = probe(x, y)
    assert np.array_equal(np.isnan(out[4]), np.isnan(out[5]))
    ok = ~np.isnan(out[4])
    assert np.abs(out[4][ok] - out[5][ok]).max() <= 8.7e-16
    assert np.array_equal(np.signbit(out[4][ok]), np.signbit(out[5][ok]))
