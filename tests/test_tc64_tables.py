"""The digit tables of the FP64 tensor-core convolutions (host code of the library, called on
the CPU): the digits are the axis' kernel, keep its mean, fit FP16, and the accumulators' levels
stay where the kernel's header says they do.

Level l holds sum_{i + j = l} X_i K_j with |X_0| <= 2^9, |X_i| <= 2^8: whatever the X_i are it
is at most 2^9 sum |K_l| + 2^8 (sum |K_{l-1}| + ... + sum |K_0|), and an FP32 accumulator of
integers is exact up to 2^24."""
import ctypes

import numpy as np
import pytest

LENGTHS = (16, 32, 48, 64, 96, 128)
LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288")


@pytest.fixture(scope="module")
def table():
    from paper_1204_5434_gb300 import build
    lib = ctypes.CDLL(build.build())
    size = lib._ZN3pft21tc64_axis_table_bytesEi
    size.restype = ctypes.c_size_t

    def make(n, d):
        dst = np.zeros(size(n), np.uint8)
        d = np.ascontiguousarray(d, LD)
        lib._ZN3pft15tc64_axis_tableEiPKePh(ctypes.c_int(n), ctypes.c_void_p(d.ctypes.data),
                                            ctypes.c_void_p(dst.ctypes.data))
        p = int(dst[:4].view(np.int32)[0])
        blocks = dst[16:].view(np.float16).astype(float).reshape(7, 2 * (n // 8) - 1, 8, 8)
        K = np.zeros((7, n))
        for b in range(blocks.shape[1]):
            for r in range(8):
                for e in range(8):
                    K[:, (8 * (b - n // 8 + 1) + r - e) % n] = blocks[:, b, r, e]
        K[6] *= 512
        return p, K

    return make


def _factors(n, L, Ns):
    k = 2 * PI * np.arange(n // 2 + 1).astype(LD) / LD(L)
    return np.exp(-k * k / LD(Ns))


# kernel widths sqrt(2 ds) from a fiftieth of a grid cell to three times the longest line
WIDTHS = np.exp(np.linspace(np.log(0.02), np.log(400.0), 80))


@pytest.mark.parametrize("n", LENGTHS)
def test_digits(table, n):
    for width in WIDTHS:
        d = _factors(n, n / width * np.sqrt(2.0), 1)
        p, K = table(n, d)
        assert np.array_equal(K, np.rint(K)) and np.max(np.abs(K)) <= 2047
        assert K[0].sum() == 2.0 ** p and np.all(K[1:].sum(axis=1) == 0)
        # the kernel: the seven digits to their last unit, in extended precision (an 80-bit long
        # double carries 2^-64 of the largest value, so the comparison ends there)
        j, k = np.arange(n), np.arange(n // 2 + 1)
        mult = np.where((k == 0) | (2 * k == n), LD(1), LD(2))
        c = np.cos(2 * PI * np.arange(n).astype(LD) / LD(n))
        kern = (mult * d / LD(n) * c[(j[:, None] * k[None, :]) % n]).sum(axis=1)
        got = sum(K[s].astype(LD) * LD(2.0) ** (-9 * s - p) for s in range(7))
        assert float(np.max(np.abs(got - kern))) <= n * 2.0 ** -64
        size = np.abs(K).sum(axis=1)
        level = np.array([512 * size[lev] + 256 * size[:lev].sum() for lev in range(6)]) / 2.0 ** 24
        assert max(level[:5] if n <= 64 else level[:2] if n == 96 else level[:3]) <= 1, (width, level)
        if n == 96 and width < n / 2:
            assert max(level[:4]) <= 1, (width, level)
        assert level[3] <= 1.5 and level[5] <= 2.2, (width, level)
