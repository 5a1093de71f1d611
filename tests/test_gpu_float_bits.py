"""pe_sum (the pole segments' sum of the per-energy formation) and to_float (the wide assembly's rounding), which work on
integers (csrc/float_bits.cuh), against the plain FP64 sum in order and the conversion instruction on the device, bit
for bit: exponents up to, at and past the largest gap that is summed on integers, mixed signs, cancellation, zeros,
subnormals, infinities and NaNs; doubles around every rounding and at both ends of the float range."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    so = str(tmp_path_factory.mktemp("bits") / "float_bits_check.so")
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared", "-Xcompiler",
                    "-fPIC", "-o", so, os.path.join(HERE, "cuda", "float_bits_check.cu")], check=True)
    L = ctypes.CDLL(so)
    L.sums.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p]
    L.floats.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p]

    def sums(v):
        x = torch.tensor(v, device="cuda")
        out = torch.empty((2, len(v)), dtype=torch.float64, device="cuda")
        assert L.sums(x.data_ptr(), v.shape[1], len(v), out[0].data_ptr(), out[1].data_ptr()) == 0
        return out.cpu().numpy()

    def floats(v):
        x = torch.tensor(v, device="cuda")
        out = torch.empty((2, v.size), dtype=torch.float32, device="cuda")
        assert L.floats(x.data_ptr(), v.size, out[0].data_ptr(), out[1].data_ptr()) == 0
        return out.cpu().numpy()

    return sums, floats


def same(a, b, kind):
    nan = np.isnan(b)
    return np.array_equal(np.isnan(a), nan) and np.array_equal(a[~nan].view(kind), b[~nan].view(kind))


def rows(n, gap, base):
    """Rows of n floats whose exponents span `gap` from `base` on, special rows among them."""
    rng = np.random.default_rng(1000 * gap + 10 * base + n)
    m = 4000
    e = rng.integers(base, base + gap + 1, (m, n))
    e[: m // 2, 0], e[: m // 2, -1] = base, base + gap
    frac = np.where(rng.random((m, n)) < 0.3, 0x7fffff, rng.integers(0, 1 << 23, (m, n)))
    frac = np.where(rng.random((m, n)) < 0.1, 0, frac)
    sign = np.where(np.arange(m)[:, None] % 3 == 0, 0, rng.integers(0, 2, (m, n)))
    v = ((sign << 31) | (e << 23) | frac).astype(np.uint32).view(np.float32)
    v[m // 4: m // 2][rng.random((m // 2 - m // 4, n)) < 0.3] = 0.0
    v[m // 2: m // 2 + 40, 1:] = -0.0
    v[m // 2 + 40: m // 2 + 80, 0], v[m // 2 + 40: m // 2 + 80, 1:] = 0.0, -0.0
    k = m // 2 + 80   # sums that cancel
    v[k: k + 200, 1] = -v[k: k + 200, 0]
    v[k: k + 200, 2:] = 0.0
    v[k + 200: k + 260, 1] = rng.integers(1, 1 << 23, 60).astype(np.uint32).view(np.float32)   # subnormal
    v[k + 260: k + 270, 0], v[k + 270: k + 280, 1], v[k + 280: k + 290, 0] = np.inf, -np.inf, np.nan
    return v


@pytest.mark.parametrize("n", [2, 3, 5, 7, 8])
def test_sums(dev, n):
    for gap in (0, 1, 12, 25, 26, 27, 28, 40, 120):
        for base in (1, 2, 60, 127, 214):
            if base + gap <= 254:
                got, plain = dev[0](np.ascontiguousarray(rows(n, gap, base)))
                assert same(got, plain, np.uint64), (gap, base)


def test_floats(dev):
    rng = np.random.default_rng(3)
    m = 1 << 20
    exps = rng.integers(1023 - 152, 1023 + 130, m).astype(np.uint64)
    frac = rng.integers(0, 1 << 52, m).astype(np.uint64)
    tail = np.array([0, 1, (1 << 28) - 1, 1 << 28, (1 << 28) + 1, (1 << 29) - 1], dtype=np.uint64)   # around a half
    frac[::2] = (frac[::2] >> np.uint64(29) << np.uint64(29)) | tail[rng.integers(0, 6, m // 2)]
    frac[::16] |= np.uint64(((1 << 23) - 1) << 29)   # the rounding carries into the exponent
    v = ((rng.integers(0, 2, m).astype(np.uint64) << np.uint64(63)) | (exps << np.uint64(52)) | frac).view(np.float64)
    edge = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 2.0 ** -126, 2.0 ** -149, 2.0 ** -150, 2.0 ** 127,
                     np.float64(np.finfo(np.float32).max), 3.4028235677973366e38, 1e300])
    v = np.concatenate([v, edge, np.nextafter(edge, 0.0), np.nextafter(edge, np.inf), -edge])
    got, plain = dev[1](v)
    assert same(got, plain, np.uint32)
