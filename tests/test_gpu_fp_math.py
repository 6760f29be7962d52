"""Device functions of csrc/fp_math.cuh against FP64: the error that each states,
over every argument of its range, and the special values.  tests/gpu_fp_math.cu is
compiled here with nvcc."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2506_10526_gb300", "csrc")


@pytest.fixture(scope="module")
def fpm(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = tmp_path_factory.mktemp("fpm") / "libfpm.so"
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O3",
                        "-shared", "-Xcompiler", "-fPIC", "-I", CSRC, "-o", str(out),
                        os.path.join(HERE, "gpu_fp_math.cu")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(str(out))


def _tanh(fpm, x, kind):
    x = np.ascontiguousarray(x, np.float32)
    y = np.empty_like(x)
    p = ctypes.POINTER(ctypes.c_float)
    assert fpm.fpm_tanh(kind, x.ctypes.data_as(p), y.ctypes.data_as(p), x.size) == 0
    return y


# of tanh_pair and tanh_pair_grad: the stated relative error and bias
TANH = [(1.8e-7, 1e-8), (2.3e-7, 2e-8)]


@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("exponent", range(-13, 4))
def test_tanh_of_every_argument(fpm, exponent, kind):
    """Each binade from 2^-13 to 16, every FP32 value, both signs: within the stated
    relative error of tanh, and against the correctly rounded value no bias above the
    stated one (rounding alone is biased near 2^-13, where tanh(x) lies just below x)."""
    lo = (127 + exponent) << 23
    out = (ctypes.c_double * 2)()
    assert fpm.fpm_tanh_err(kind, ctypes.c_uint32(lo), ctypes.c_uint32(1 << 23), out) == 0
    assert out[0] <= TANH[kind][0]
    assert abs(out[1]) <= TANH[kind][1]


@pytest.mark.parametrize("kind", [0, 1])
def test_tanh_special_values(fpm, kind):
    """Zeros with their sign, the smallest and small values (tanh(x) = x to rounding
    below 2^-13), values beyond 16, infinities, NaN, and an odd function."""
    inf, nan = np.float32(np.inf), np.float32(np.nan)
    y = _tanh(fpm, [0.0, -0.0, inf, -inf, nan, 16.0, -1e30, 3e38], kind)
    assert y[0] == 0 and not np.signbit(y[0]) and y[1] == 0 and np.signbit(y[1])
    assert y[2] == 1 and y[3] == -1 and np.isnan(y[4])
    np.testing.assert_array_equal(y[5:], [1, -1, 1])
    r = np.random.default_rng(1)
    x = r.integers(1, 114 << 23, 100001).astype(np.uint32).view(np.float32)  # up to 2^-13
    np.testing.assert_allclose(_tanh(fpm, x, kind).astype(np.float64), np.tanh(x.astype(np.float64)),
                               rtol=TANH[kind][0], atol=0)
    x = np.concatenate([x, r.standard_normal(100001).astype(np.float32)])
    np.testing.assert_array_equal(_tanh(fpm, -x, kind), -_tanh(fpm, x, kind))


@pytest.mark.parametrize("spread", [1.0, 60.0, 126.0, 149.0])
def test_normalised_inputs_round_as_quotients(fpm, spread):
    """(x - mu) / sd for ordinary deviations and for deviations up to 2^121 and down
    to the smallest: never more than one unit in the last place from the division's
    result, and equal to it in all but one in a thousand (the residual step rounds
    as a division but where the remainder lies within the rounding of 1 / sd)."""
    n = 1 << 19
    r = np.random.default_rng(int(spread))
    sd = (r.uniform(0.5, 2, 2 * n) * 2.0 ** r.uniform(-spread, min(spread, 120), 2 * n)).astype(np.float32)
    sd[sd == 0] = np.float32(2.0 ** -149)
    mu = (sd * r.standard_normal(2 * n)).astype(np.float32)
    x = (mu + sd * r.standard_normal(2 * n)).astype(np.float32)
    a = np.ascontiguousarray(np.concatenate([x, mu, sd]), np.float32)
    got = np.empty(2 * n, np.float32)
    p = ctypes.POINTER(ctypes.c_float)
    assert fpm.fpm_normalise(a.ctypes.data_as(p), got.ctypes.data_as(p), n) == 0
    want = (x - mu) / sd
    assert np.all(np.abs(got.astype(np.float64) - want) <= np.spacing(np.abs(want)))
    assert np.mean(got != want) <= 1e-3


def test_reciprocal_square_root(fpm):
    """Squared lengths from the smallest to the largest that the binnings accept (k_perp
    in [1e-8, 1e8], |k_par| up to 1e8: 1e-16 to 5e16), over FP32's normal range, at
    powers of two and their neighbours: below 2^-52 relative, against extended
    precision."""
    r = np.random.default_rng(4)
    two = 2.0 ** np.arange(-126, 128)
    s = np.concatenate([10.0 ** r.uniform(-16, np.log10(5e16), 1 << 20), [1e-16, 5e16],
                        two * r.uniform(1, 2, two.size), two, np.nextafter(two[1:], 0),
                        np.nextafter(two, np.inf)])
    y = np.empty_like(s)
    p = ctypes.POINTER(ctypes.c_double)
    assert fpm.fpm_rsqrt(s.ctypes.data_as(p), y.ctypes.data_as(p), s.size) == 0
    want = 1 / np.sqrt(s.astype(np.longdouble))
    assert np.abs(y / want - 1).max() < 2.0 ** -52


def test_normalised_inputs_of_infinite_deviations(fpm):
    """Quotients by an infinite deviation are zero, as by a division; the neighbouring
    column is not touched."""
    a = np.array([3.0, 5.0, 1.0, 1.0, np.inf, 2.0], np.float32)
    got = np.empty(2, np.float32)
    p = ctypes.POINTER(ctypes.c_float)
    assert fpm.fpm_normalise(a.ctypes.data_as(p), got.ctypes.data_as(p), 1) == 0
    np.testing.assert_array_equal(got, [0.0, 2.0])
