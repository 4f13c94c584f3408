"""The host work of a new box.  An FP64 context also builds the tables of its tensor-core
convolutions, in extended precision, which is software on the GPU's aarch64 host: 65 exponentials
an axis of 128 points, and a sum of 65 x 65 double-double products (some 0.06 ms an axis).  Twice
that is allowed beyond an FP32 context's box; evaluating the factors and the cosines inside the
sum takes five times as much."""
import time

import pytest

from paper_1204_5434_gb300 import pft

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1204_5434_gb300 import build
    build.build()


def _box_ms(prec, scheme=pft.PFT_SCHEME_SPLIT2):
    best = float("inf")
    with pft.System((128, 128, 128), (8.0, 8.0, 8.0), 1, 0.5, 15.0, 1.0, pft.PFT_SCFT_REAL, prec, scheme=scheme) as s:
        for i in range(30):
            L = (8.0 + 0.01 * i, 7.0 + 0.02 * i, 9.0 + 0.03 * i)  # three tables of their own
            t = time.perf_counter()
            pft.pft_set_box(s.h, L)
            best = min(best, time.perf_counter() - t)
    return 1e3 * best


def test_box_of_an_fp64_context():
    f32, f64 = _box_ms(pft.PFT_FP32_MIXED), _box_ms(pft.PFT_FP64)
    print(f"\npft_set_box 128^3: FP32 {f32:.2f} ms, FP64 {f64:.2f} ms")
    assert f64 <= f32 + 0.4


def test_box_of_a_scheme_without_those_tables():
    f32 = _box_ms(pft.PFT_FP32_MIXED, pft.PFT_SCHEME_RQM4)
    f64 = _box_ms(pft.PFT_FP64, pft.PFT_SCHEME_RQM4)
    print(f"\npft_set_box 128^3, RQM4: FP32 {f32:.2f} ms, FP64 {f64:.2f} ms")
    assert f64 <= f32 + 0.1
