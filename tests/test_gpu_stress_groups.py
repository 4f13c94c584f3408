"""The box derivative with its contour steps taken in groups of up to 32 a launch: chains of
one step, of one short, whole and overlong group and of several, on the pencil passes (both
precisions) and on the FP32 plane kernel, against the oracle at the tolerances of
test_gpu_gradients; called twice, with another box in between."""
import numpy as np
import pytest

import oracle as o
from paper_1204_5434_gb300 import pft

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1204_5434_gb300 import build
    build.build()


CASES = [((8, 12, 16), pft.PFT_FP64, Ns, 1e-9) for Ns in (1, 31, 32, 33, 65)]
CASES += [((12, 8, 6), pft.PFT_FP32_MIXED, 34, 2e-4), ((16, 64, 64), pft.PFT_FP32_MIXED, 33, 2e-4)]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_box_derivative_in_groups(case):
    n, prec, Ns, tol = CASES[case]
    rng = np.random.default_rng(900 + case)
    wp = rng.normal(0, 0.2, n)
    wm = 3.0 * np.cos(2 * np.pi * np.arange(n[0]) / n[0])[:, None, None] + rng.normal(0, 0.2, n)
    with pft.System(n, (4.0, 3.0, 2.0), Ns, 0.4, 18.0, 2.0, pft.PFT_SCFT_REAL, prec) as s:
        for L in ((4.0, 3.0, 2.0), (4.5, 2.8, 2.2)):
            s.set_box(L)
            s.set_fields(wp, wm)
            s.solve()
            _, _, _, dq = s.gradients(want_fields=False)
            ref = o.solve(wp, wm, n, L, Ns, 0.4, o.SCFT_REAL)
            gq = o.dlnQ_dL(ref, n, L)
            err = max(abs(dq[a] - gq[a]) / abs(gq[a]) for a in range(3))
            print(f"\n{n} Ns={Ns} prec={prec} L={L}: dlnQ/dL rel {err:.2e}")
            assert err <= tol, (dq, gq)
