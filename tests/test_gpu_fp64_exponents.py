"""FP64 solves at the ends of the exponent range, on grids whose axes all run on the tensor cores:
a constant added to W+ multiplies every slice by a power of ten and leaves the densities and the
shape of the propagators alone.  Up to 1e-300 and 1e+300 the solve follows the unshifted one at
the FP64 tolerances of the parity tests."""
import numpy as np
import pytest

from paper_1204_5434_gb300 import pft

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1204_5434_gb300 import build
    build.build()


@pytest.mark.parametrize("shift", [640.0, 670.0, 690.0, -640.0, -690.0])
@pytest.mark.parametrize("n", [(32, 16, 48), (16, 96, 128)])
def test_shift_to_the_ends_of_the_range(n, shift):
    L, Ns, fA = (4.0, 2.0, 6.0), 100, 0.5
    rng = np.random.default_rng(830)
    wp, wm = rng.normal(0, 0.3, n), rng.normal(0, 1.0, n)
    with pft.System(n, L, Ns, fA, 17.0, 2.0, pft.PFT_SCFT_REAL, pft.PFT_FP64) as s:
        s.set_fields(wp, wm)
        s.solve()
        A0, B0 = s.densities()
        lnQ0 = s.observables()["lnQ"].real
        q0 = [s.propagator(w, Ns) for w in (0, 2)]
        s.set_fields(wp + shift, wm)
        s.solve()
        A1, B1 = s.densities()
        dQ = abs(s.observables()["lnQ"].real + shift - lnQ0)
        eq = 0.0
        for w in (0, 2):
            q = s.propagator(w, Ns)
            h = q0[w // 2] / np.max(q0[w // 2])
            eq = max(eq, np.max(np.abs(q / np.max(q) - h)))
    ephi = max(np.max(np.abs(A1 - A0)), np.max(np.abs(B1 - B0)))
    print(f"\n{n} shift {shift}: lnQ {dQ:.1e} phi {ephi:.1e} slices {eq:.1e}")
    assert dQ <= 1e-10 and ephi <= 1e-10 and eq <= 1e-11  # exp of a field near 700: 700 x 1e-16
