"""The double logarithm of the FP64 forms: the integer path on the host against long double, and on the
GPU the whole function against CUDA's log, where it hands over to it and where it does not."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2212_10680_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    lib = str(tmp_path_factory.mktemp("log") / "liblogprobe.so")
    subprocess.run([nvcc, *build.ARCH, *build.FLAGS, "-shared", os.path.join(HERE, "log_probe.cu"), "-o", lib],
                   check=True, capture_output=True, timeout=300)
    p = ctypes.CDLL(lib)
    p.log_takes.argtypes = [ctypes.c_double]
    p.log_max_ulp.argtypes = [ctypes.c_longlong, ctypes.POINTER(ctypes.c_double)]
    p.log_max_ulp.restype = ctypes.c_double
    p.log_device.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int]
    return p


def test_integer_path_is_within_0_6_ulp(probe):
    # half an ulp of the final rounding, and the fixed-point sum's error (2^-58 for k != 0 against a result
    # of 0.3 and more, 2^-61 relative around 1) and the polynomial's 2^-61: below 0.1 ulp together
    at = ctypes.c_double()
    worst = probe.log_max_ulp(4_000_000, ctypes.byref(at))
    assert worst < 0.6, (worst, at.value.hex())


def test_the_integer_path_takes_normal_numbers_of_its_exponents_alone(probe):
    for x in (2.0 ** -43, 1.0, np.nextafter(2.0 ** 44, 0.0)):
        assert probe.log_takes(x)
    for x in (np.nextafter(2.0 ** -43, 0.0), 2.0 ** 44, 0.0, -0.0, -1.0, -2.0 ** -20, np.inf, -np.inf, np.nan, 5e-324,
              2.2250738585072014e-308, 1.7976931348623157e308):
        assert not probe.log_takes(x)


@pytest.mark.gpu
def test_device_logarithm_against_cudas(probe):
    import torch
    rng = np.random.default_rng(1)
    ends = np.array([0.0, -0.0, -1.0, -1e-300, np.nan, np.inf, -np.inf, 5e-324, 1e-310, 2.2250738585072014e-308,
                     1.7976931348623157e308, np.nextafter(2.0 ** -43, 0.0), 2.0 ** 44, 2.0 ** 60, 2.0 ** -60])
    inner = np.concatenate([
        [2.0 ** -43, np.nextafter(2.0 ** 44, 0.0), 1.0, np.nextafter(1.0, 0.0), np.nextafter(1.0, 2.0)],
        np.ldexp(1.0 + np.arange(128) / 128.0, rng.integers(-43, 44, 128)),
        np.ldexp(rng.uniform(1.0, 2.0, 200_000), rng.integers(-43, 44, 200_000)),
        rng.uniform(0.5, 2.0, 200_000), 1.0 + rng.uniform(-1, 1, 100_000) * 2.0 ** rng.integers(-40, -1, 100_000)])
    x = torch.tensor(np.concatenate([ends, inner]), device="cuda")
    ours, cuda = torch.empty_like(x), torch.empty_like(x)
    torch.cuda.synchronize()
    assert probe.log_device(x.data_ptr(), ours.data_ptr(), cuda.data_ptr(), x.numel()) == 0
    ours, cuda = ours.cpu().numpy(), cuda.cpu().numpy()
    k = len(ends)
    assert np.array_equal(ours[:k], cuda[:k], equal_nan=True)   # the same function
    # 0.6 ulp of ours and the 1 ulp that CUDA documents, of the larger of the two
    ulp = np.spacing(np.maximum(np.abs(ours[k:]), np.abs(cuda[k:])))
    assert np.all(np.abs(ours[k:] - cuda[k:]) <= 1.6 * ulp)
    assert ours[k + 2] == 0.0
