"""FP64 solves whose Boltzmann factors or propagators span many orders of magnitude, on grids
whose axes all run on the tensor cores, so that a scale taken from anything but a line's own
values costs digits.

Gauge shifts: a constant added to W+ (i omega+) multiplies every slice and leaves the densities
alone, so strong fields whose factors are all far below one must be as accurate as any: the
FP64 tolerances of the parity tests (1e-12 of a slice's largest value, 1e-12 of Q, 1e-10 of
phi).

Impenetrable regions: whole lines of a propagator lie many decades below the slice's largest
value.  There the solve is held to the accuracy of an FP64 transform march point by point: its
largest relative error against an extended-precision march is at most twice that of the FP64
oracle (both accumulate the same number of roundings; two for their scatter)."""
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


@pytest.mark.parametrize("streams", [0, 1])
@pytest.mark.parametrize("shift", [1.0, 100.0, 200.0])
@pytest.mark.parametrize("n,kind", [((32, 16, 48), SCFT), ((48, 16, 32), CL), ((16, 96, 128), SCFT)])
def test_shifted_strong_fields(n, kind, shift, streams):
    """W- of ten decades of factors; the shift takes the largest factor from far above one to far
    below it (1: hardly, 100: near one, 200: 1e-4 and less)."""
    L, Ns, fA = (4.0, 3.0, 5.0), 6, 0.5
    rng = np.random.default_rng(810)
    wp, wm = rng.normal(0, 0.3, n), rng.normal(0, 25.0, n)
    if kind == CL:  # omega+ enters as i omega+
        wp = wp + 1j * rng.normal(0, 0.3, n) - 1j * shift
        wm = wm + 1j * rng.normal(0, 0.3, n)
    else:
        wp = wp + shift
    _check(n, L, Ns, fA, kind, streams, wp, wm)


@pytest.mark.parametrize("amp,shift,Ns", [(100.0, 100.0, 8), (60.0, 62.0, 12)])
def test_shifted_lamella(amp, shift, Ns):
    """A strongly segregated lamella on a coarse contour: the largest factors of the two blocks are
    apart, their products at the block junction everywhere far below the product of the largest."""
    n, L, fA = (64, 16, 32), (4.0, 1.0, 2.0), 0.5
    rng = np.random.default_rng(811)
    x = 2 * np.pi * np.arange(n[0]) / n[0]
    wm = amp * np.cos(x)[:, None, None] + rng.normal(0, 0.1, n)
    wp = shift + rng.normal(0, 0.1, n)
    _check(n, L, Ns, fA, SCFT, 0, wp, wm)


def _check(n, L, Ns, fA, kind, streams, wp, wm):
    ref = o.solve(wp, wm, n, L, Ns, fA, o.SCFT_REAL if kind == SCFT else o.CL_COMPLEX)
    with pft.System(n, L, Ns, fA, 17.0, 2.0, kind, FP64) as s:
        pft.pft_set_plan(s.h, 3, streams)
        s.set_fields(wp, wm)
        s.solve()
        obs = s.observables()
        phiA, phiB = s.densities()
        eq = 0.0
        for which in (0, 2):
            for k in (1, Ns // 2, Ns // 2 + 1, Ns):
                h = (ref.q if which == 0 else ref.qd)[k]
                eq = max(eq, np.max(np.abs(s.propagator(which, k) - h)) / np.max(np.abs(h)))
    Q = obs["Q"] if kind == CL else obs["Q"].real
    eQ = abs(Q - ref.Q) / abs(ref.Q)
    ephi = max(np.max(np.abs(phiA - ref.phiA)), np.max(np.abs(phiB - ref.phiB)))
    print(f"\n{n} kind={kind}: Q rel {eQ:.2e} phi abs {ephi:.2e} slices {eq:.2e}")
    assert eQ <= 1e-12 and ephi <= 1e-10 and eq <= 1e-12


@pytest.mark.parametrize("n,kind", [((96, 16, 48), SCFT), ((16, 64, 64), CL), ((32, 96, 128), CL), ((96, 128, 16), CL),
                                    ((128, 48, 96), SCFT), ((128, 32, 16), CL)])
def test_long_lines_on_every_axis(n, kind):
    """96 and 128 points on each axis, and complex lines of 16 on x, on grids without an axis on the
    FFT kernels (the last one's x launch is too short for the tensor cores)."""
    rng = np.random.default_rng(813)
    wp, wm = rng.normal(0, 0.3, n), rng.normal(0, 1.0, n)
    if kind == CL:
        wp, wm = wp + 1j * rng.normal(0, 0.3, n), wm + 1j * rng.normal(0, 0.3, n)
    _check(n, (5.0, 4.0, 6.0), 4, 0.4, kind, 1, wp, wm)


LD = np.longdouble


def _extended(w, n, L, Ns, steps):
    """q_s, s in `steps`, of one homopolymer march in extended precision: the three periodic
    convolutions as products with the axes' circulant matrices."""
    pi = LD("3.14159265358979323846264338327950288")
    mats = []
    for a in range(3):
        k = np.arange(n[a] // 2 + 1)
        f = np.where((k == 0) | (2 * k == n[a]), LD(1), LD(2)) / LD(n[a])
        d = np.exp(-((2 * pi * k.astype(LD) / LD(L[a])) ** 2) / LD(Ns))
        c = np.cos(2 * pi * np.arange(n[a]).astype(LD) / LD(n[a]))
        kern = np.array([np.sum(f * d * c[(j * k) % n[a]]) for j in range(n[a])])
        i = np.arange(n[a])
        mats.append(kern[(i[:, None] - i[None, :]) % n[a]])
    B = np.exp(-w.astype(LD) / LD(2 * Ns))
    q, out = np.ones(n, LD), {}
    for s in range(1, Ns + 1):
        q = B * q
        for a in range(3):
            q = np.moveaxis(np.tensordot(mats[a], q, axes=(1, a)), 0, a)
        q = B * q
        if s in steps:
            out[s] = q
    return out


@pytest.mark.parametrize("shape", ["pore", "slab"])
def test_lines_far_below_the_largest(shape):
    """q at W+ = 60 outside a pore (inside a slab: whole y-z planes), of both blocks alike."""
    n, L, Ns = (32, 16, 16), (4.0, 2.0, 2.0), 64
    X, Y, Z = np.meshgrid(*[(np.arange(m) + 0.5) * (l / m) - l / 2 for m, l in zip(n, L)], indexing="ij")
    if shape == "pore":
        wall = (X ** 2 + Y ** 2 + Z ** 2) > 0.64
    else:
        wall = np.abs(X) > 0.7
    w = 60.0 * wall + np.random.default_rng(812).normal(0, 0.1, n)
    wm = np.zeros(n)
    steps = (Ns // 2, Ns)
    ref = o.solve(w, wm, n, L, Ns, 0.5, o.SCFT_REAL)
    ex = _extended(w, n, L, Ns, steps)
    with pft.System(n, L, Ns, 0.5, 17.0, 2.0, SCFT, FP64) as s:
        s.set_fields(w, wm)
        s.solve()
        for k in steps:
            rel = lambda q: float(np.max(np.abs((q.astype(LD) - ex[k]) / ex[k])))  # noqa: E731
            eg, eo = rel(s.propagator(0, k)), rel(ref.q[k])
            span = float(np.max(ex[k]) / np.min(ex[k]))
            print(f"\n{shape} q_{k}: decades {np.log10(span):.1f}, relative error {eg:.2e}, FP64 oracle {eo:.2e}")
            assert eg <= 2 * eo
