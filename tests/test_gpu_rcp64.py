"""The FP64 step's reciprocal against CUDA's correctly rounded division: random
mantissas at all exponents, the edges of its range, zero, subnormals, infinities
and NaN, both signs."""
import numpy as np
import pytest

from paper_1308_0653_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _both(x):
    import torch
    from paper_1308_0653_gb300 import dbm
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    x = torch.from_numpy(x).cuda()
    fast, ieee = torch.empty_like(x), torch.empty_like(x)
    assert dbm.lib().dbm_selftest_rcp64(x.data_ptr(), fast.data_ptr(), ieee.data_ptr(), x.numel(), None) == dbm.DBM_OK
    torch.cuda.synchronize()
    return fast.cpu().numpy(), ieee.cpu().numpy()


def _bits(sign, exponent, mantissa):
    return ((sign << np.uint64(63)) | (exponent << np.uint64(52)) | mantissa).view(np.float64)


def test_random_mantissas_at_all_exponents():
    n = 1 << 22
    r = W.splitmix64(1, 1, n)
    exponent = W.splitmix64(1, 2, n) % np.uint64(2048)
    exponent[: n // 2] = np.uint64(1013) + W.splitmix64(1, 3, n // 2) % np.uint64(20)  # densities, temperatures
    fast, ieee = _both(_bits(r >> np.uint64(63), exponent, r & np.uint64((1 << 52) - 1)))
    nan = np.isnan(ieee)
    assert np.array_equal(np.isnan(fast), nan)
    off = np.abs(fast.view(np.int64) - ieee.view(np.int64))[~nan]
    # 2^-19 squared twice is 2^-23 of an ulp: that share of the roundings may differ, by one ulp
    assert off.max() <= 1 and np.count_nonzero(off) <= 2 + n * 2.0 ** -22


def test_edges():
    exponents = np.array([0, 1, 2, 22, 23, 24, 1022, 1023, 1024, 2022, 2023, 2024, 2045, 2046, 2047], dtype=np.uint64)
    top = (1 << 52) - 1
    mantissas = np.array([0, 1, 2, top >> 1, (top >> 1) + 1, top - 1, top], dtype=np.uint64)
    s, e, m = np.meshgrid(np.array([0, 1], dtype=np.uint64), exponents, mantissas, indexing="ij")
    fast, ieee = _both(np.ascontiguousarray(_bits(s, e, m)).ravel())
    nan = np.isnan(ieee)
    assert np.array_equal(np.isnan(fast), nan) and np.array_equal(fast[~nan].view(np.int64), ieee[~nan].view(np.int64))
