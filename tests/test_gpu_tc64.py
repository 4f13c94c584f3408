"""The FP64 separable march with its convolutions on the tensor cores (axes of 16, 32, 48, 64,
96 and 128 points) against the FP64 oracle, at the FP64 tolerances of test_gpu_parity: tiles
of 128 lines partly outside the grid, axes on the tensor cores beside axes on the FFT kernels,
one- and two-step chains, the block junction, real and complex fields, both stream layouts;
propagators over many decades; a non-finite field."""
import numpy as np
import pytest

import oracle as o
from paper_1204_5434_gb300 import pft

pytestmark = pytest.mark.gpu
FP64 = pft.PFT_FP64
SCFT, CL = pft.PFT_SCFT_REAL, pft.PFT_CL_COMPLEX


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1204_5434_gb300 import build
    build.build()


def _fields(n, kind, seed, amp):
    rng = np.random.default_rng(seed)
    wp = rng.normal(0, 0.3, n)
    wm = rng.normal(0, amp, n)
    if kind == CL:
        wp = wp + 1j * rng.normal(0, 0.3, n)
        wm = wm + 1j * rng.normal(0, 0.3, n)
    return wp, wm


def _errors(n, L, Ns, fA, kind, streams, wp, wm):
    ref = o.solve(wp, wm, n, L, Ns, fA, o.SCFT_REAL if kind == SCFT else o.CL_COMPLEX)
    with pft.System(n, L, Ns, fA, 17.0, 2.0, kind, FP64) as s:
        pft.pft_set_plan(s.h, 3, streams)
        s.set_fields(wp, wm)
        s.solve()
        s.solve()  # the replayed graph
        obs = s.observables()
        phiA, phiB = s.densities()
        eq = 0.0
        for which, k in ((0, 1), (0, Ns), (2, 1), (2, Ns)):
            h = (ref.q if which == 0 else ref.qd)[k]
            eq = max(eq, np.max(np.abs(s.propagator(which, k) - h)) / np.max(np.abs(h)))
    Q = obs["Q"] if kind == CL else obs["Q"].real
    ephi = max(np.max(np.abs(phiA - ref.phiA)), np.max(np.abs(phiB - ref.phiB)))
    return abs(Q - ref.Q) / abs(ref.Q), ephi, eq


# every length on every axis, with line counts that are no multiple of 128, and one or two axes
# left to the FFT kernels (4, 6, 24, 192, 256)
CASES = [
    ((16, 32, 48), (2.0, 4.0, 6.0), 5, 0.4, SCFT, 1),
    ((32, 48, 16), (4.0, 6.0, 2.0), 4, 0.3, CL, 0),
    ((48, 16, 32), (6.0, 2.0, 4.0), 1, 0.5, SCFT, 0),
    ((64, 6, 96), (8.0, 1.5, 12.0), 3, 0.4, SCFT, 1),
    ((96, 64, 4), (12.0, 8.0, 0.5), 2, 0.5, CL, 1),
    ((4, 96, 64), (1.0, 12.0, 8.0), 5, 0.4, CL, 0),
    ((128, 4, 24), (8.0, 1.0, 3.0), 4, 0.6, SCFT, 0),
    # both sides of the line below which x launches stay on the FFT kernels
    ((64, 24, 96), (8.0, 3.0, 12.0), 2, 0.5, CL, 1),
    ((64, 24, 64), (8.0, 3.0, 8.0), 2, 0.5, CL, 1),
    ((16, 24, 192), (2.0, 3.0, 24.0), 2, 0.5, SCFT, 1),
    ((16, 24, 128), (2.0, 3.0, 16.0), 2, 0.5, CL, 0),
    ((6, 128, 12), (1.5, 16.0, 3.0), 3, 0.4, CL, 1),
    ((6, 4, 128), (1.5, 1.0, 8.0), 6, 0.35, SCFT, 1),
    ((16, 192, 128), (2.0, 12.0, 8.0), 3, 0.5, SCFT, 1),
    ((128, 16, 256), (8.0, 2.0, 16.0), 3, 0.5, CL, 0),
    # kernels wider than the box and narrower than a grid cell
    ((32, 64, 128), (0.5, 0.5, 0.5), 2, 0.5, SCFT, 1),
    ((32, 64, 128), (40.0, 60.0, 90.0), 60, 0.5, SCFT, 1),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_matches_oracle(case):
    n, L, Ns, fA, kind, streams = CASES[case]
    wp, wm = _fields(n, kind, 700 + case, 1.0)
    eQ, ephi, eq = _errors(n, L, Ns, fA, kind, streams, wp, wm)
    print(f"\ntc64 {n} Ns={Ns} kind={kind}: Q rel {eQ:.2e} phi abs {ephi:.2e} slices {eq:.2e}")
    assert eQ <= 1e-12 and ephi <= 1e-10 and eq <= 1e-12


@pytest.mark.parametrize("n,kind", [((32, 16, 48), SCFT), ((48, 16, 32), CL), ((16, 24, 32), SCFT)])
def test_strong_fields(n, kind):
    """Boltzmann factors over ten decades (fixed-point and, with the 24-point axis, FP64 factors)."""
    wp, wm = _fields(n, kind, 730, 25.0)
    eQ, ephi, eq = _errors(n, (4.0, 3.0, 5.0), 6, 0.5, kind, 0, wp, wm)
    print(f"\n{n} kind={kind}: Q rel {eQ:.2e} phi abs {ephi:.2e} slices {eq:.2e}")
    assert eQ <= 1e-12 and ephi <= 1e-10 and eq <= 1e-12


def test_many_decades():
    """Fields that take the propagators through about twelve decades."""
    n, L, Ns, fA = (32, 48, 64), (8.0, 12.0, 16.0), 20, 0.4
    wp, wm = _fields(n, SCFT, 720, 0.5)
    wp = wp + 15.0 * np.cos(2 * np.pi * np.arange(64) / 64)[None, None, :]
    eQ, ephi, eq = _errors(n, L, Ns, fA, SCFT, 1, wp, wm)
    print(f"\nQ rel {eQ:.2e} phi abs {ephi:.2e} slices {eq:.2e}")
    assert eQ <= 1e-12 and ephi <= 1e-10 and eq <= 1e-12


def test_scaled_propagators_and_non_finite_fields():
    """A constant shift of W+ scales every slice: 1e130 and 1e-130 stay finite and follow the
    unshifted solve; a NaN in the field is reported, not hidden."""
    n, L, Ns, fA = (32, 32, 32), (4.0, 4.0, 4.0), 10, 0.5
    wp, wm = _fields(n, SCFT, 721, 1.0)
    with pft.System(n, L, Ns, fA, 17.0, 2.0, SCFT, FP64) as s:
        s.set_fields(wp, wm)
        s.solve()
        A0, _ = s.densities()
        lnQ0 = s.observables()["lnQ"].real
        for shift in (300.0, -300.0):
            s.set_fields(wp + shift, wm)
            s.solve()
            A1, _ = s.densities()
            assert np.max(np.abs(A1 - A0)) <= 1e-10
            assert abs(s.observables()["lnQ"].real + shift - lnQ0) <= 1e-10
        bad = wp.copy()
        bad[3, 5, 7] = np.nan
        s.set_fields(bad, wm)
        s.solve()
        with pytest.raises(pft.PftError) as e:
            s.observables()
        assert e.value.status == pft.PFT_ERR_NONFINITE
