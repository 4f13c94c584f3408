"""What the library's speed is judged on: one field update (or one gradient) per pass.

A case is a system of this library's own workload shapes (lamellar and gyroid SCFT, complex
Langevin, the uneven batch) and one pass is what a user's loop does with new fields: copy
them in from device memory, solve, read the densities, take the field step (or the adjoint
or the box gradient), read the result and the observables Q and h = H/(C V), which ends the
pass with the host holding them.  Fields are drawn on the GPU from the seed with the distributions of
paper_1204_5434_gb300/workloads.py.
"""
import math

import numpy as np
import torch

from paper_1204_5434_gb300 import pft

AXES = (8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256)  # grid extents drawn
RQ_WORK = 3  # split steps per contour step of the 4th-order scheme


def _case(name, what, n, L, Ns, fA, chiN, C, prec, **kw):
    c = {"what": what, "nx": n[0], "ny": n[1], "nz": n[2], "Lx": float(L[0]), "Ly": float(L[1]), "Lz": float(L[2]),
         "Ns": Ns, "fA": fA, "chiN": chiN, "C": C, "prec": prec, "seeding": "gyroid", "amp": 4.0, "noise": 0.1,
         "ck": 0, "count": 1}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    c8 = (8.0, 8.0, 8.0)
    hom = {"seeding": "homogeneous", "amp": 0.0, "noise": 0.05}
    return [
        # the lamellar relaxation of the paper, in the default precision: a small grid whose
        # update is a chain of short dependent launches
        _case("lam32_fp64", "scft", (32,) * 3, (4.0,) * 3, 64, 0.5, 15.0, 1.0, "fp64", seeding="lam", amp=5.0),
        # a gyroid relaxation at a working resolution
        _case("gyr64_fp32", "scft", (64,) * 3, c8, 100, 0.35, 18.0, 1.0, "fp32"),
        # the headline workload
        _case("gyr128_fp32", "scft", (128,) * 3, c8, 100, 0.35, 18.0, 1.0, "fp32"),
        # the same in the default precision (converged free energies)
        _case("gyr128_fp64", "scft", (128,) * 3, c8, 100, 0.35, 18.0, 1.0, "fp64"),
        # a cell that is not cubic, with extents that are not powers of two and an odd number of steps
        _case("cell96x48x64_fp32", "scft", (96, 48, 64), (12.0, 6.0, 8.0), 77, 0.4, 20.0, 1.0, "fp32"),
        # one step of a complex Langevin run with the library's own noise, both precisions
        _case("cl64_fp32", "cl", (64,) * 3, c8, 100, 0.3, 20.0, 50.0, "fp32", **hom),
        _case("cl64_fp64", "cl", (64,) * 3, c8, 100, 0.3, 20.0, 50.0, "fp64", **hom),
        # the largest grid, with the history checkpointed as a run does that shares the card
        _case("cl256_ck14_fp32", "cl", (256,) * 3, (16.0,) * 3, 200, 0.5, 14.0, 100.0, "fp32", ck=14, **hom),
        # the paper's 4th-order scheme
        _case("gyr128_rqm4_fp32", "rqm4", (128,) * 3, c8, 100, 0.35, 18.0, 1.0, "fp32"),
        # inverse design: gradient of a loss on the densities through a solve
        _case("adjoint128_fp32", "adjoint", (128,) * 3, c8, 100, 0.35, 18.0, 1.0, "fp32"),
        # variable-cell relaxation: new box, solve, field and box gradients
        _case("varcell64_fp32", "cell", (64,) * 3, c8, 100, 0.35, 18.0, 1.0, "fp32"),
        # a parameter sweep: uneven independent systems, half SCFT and half complex Langevin
        _case("batch64_fp32", "batch", (64,) * 3, c8, 200, 0.35, 18.0, 1.0, "fp32", seeding="sinusoids", count=64),
    ]


def _units(c):
    """Grid-point contour steps of one pass (both propagators), the cost measure of `draw`."""
    if c["what"] == "batch":
        return sum(2 * m["n"] ** 3 * m["Ns"] * (2 if m["cl"] else 1) for m in _members(c, 0))
    u = 2.0 * c["nx"] * c["ny"] * c["nz"] * c["Ns"]
    u *= {"scft": 1, "cl": 2, "rqm4": RQ_WORK, "adjoint": 2, "cell": 2}[c["what"]]
    return u * (1.5 if c["ck"] else 1.0)


def draw(rng):
    """A system of one of the listed kinds: extents from 8 to 256, Ns from 10 to 200, grid
    spacings of 1/16 to 1/8 Rg, compositions and segregations of the workloads."""
    while True:
        what = rng.choice(["scft", "scft", "scft", "cl", "cl", "rqm4", "adjoint", "cell", "batch"])
        prec = "fp32" if what == "batch" else rng.choice(["fp32", "fp32", "fp64"])
        Ns = int(round(math.exp(rng.uniform(math.log(10), math.log(200)))))
        if rng.random() < 0.5:
            n = (rng.choice(AXES[2:]),) * 3
        else:
            n = tuple(rng.choice(AXES) for _ in range(3))
        L = tuple(v * rng.uniform(1 / 16, 1 / 8) for v in n)
        M = n[0] * n[1] * n[2]
        cl = what == "cl"
        c = _case(None, what, n, L, Ns, rng.uniform(0.2, 0.8), rng.uniform(12, 25),
                  rng.uniform(20, 100) if cl else 1.0, prec)
        if cl:
            c.update(seeding="homogeneous", amp=0.0, noise=0.05)
        elif what == "batch":
            n, Ns = (64,) * 3, 200  # the largest member's
            c = _case(None, what, n, (8.0,) * 3, Ns, 0.35, 18.0, 1.0, prec, seeding="sinusoids", amp=0.0,
                      count=rng.randrange(3, 65))
            return c
        else:
            c.update(seeding=rng.choice(["gyroid", "lam"]), amp=rng.uniform(2, 5))
            if what in ("scft", "cell") and rng.random() < 0.2:
                c["ck"] = max(2, int(round(math.sqrt(Ns)))) if what == "scft" else 0
        # histories within 12 GB, cost within the largest listed case's (an FP64 unit costs
        # about twenty FP32 ones)
        keep = {"scft": 2, "cl": 4, "rqm4": 2, "adjoint": 4, "cell": 2}[what]
        if keep * M * Ns * (8 if prec == "fp64" else 4) > 12e9 or M < 512:
            continue
        if _units(c) * (20 if prec == "fp64" else 1) > 9e9:
            continue
        return c


# ---------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)


def _normal(g, n, s):
    return torch.randn(n, generator=g, device="cuda", dtype=torch.float64) * s


def _grid(n, L):
    x = [torch.arange(n[a], device="cuda", dtype=torch.float64) * (2 * math.pi / n[a]) for a in range(3)]
    return x[0][:, None, None], x[1][None, :, None], x[2][None, None, :]


def _fields(c, seed):
    """(W+, W-) of a single system (real), or (omega+, omega-) as complex tensors."""
    n, L = (c["nx"], c["ny"], c["nz"]), (c["Lx"], c["Ly"], c["Lz"])
    g = _gen(seed)
    X, Y, Z = _grid(n, L)
    if c["seeding"] == "lam":
        wm = c["amp"] * torch.cos(X) + _normal(g, n, c["noise"])
        wp = _normal(g, n, c["noise"])
    elif c["seeding"] == "gyroid":
        G = torch.sin(X) * torch.cos(Y) + torch.sin(Y) * torch.cos(Z) + torch.sin(Z) * torch.cos(X)
        wm = c["amp"] * G + _normal(g, n, c["noise"])
        wp = _normal(g, n, c["noise"])
    else:
        wp = _normal(g, n, c["noise"])
        wm = c["chiN"] * (2 * c["fA"] - 1) / 2 + _normal(g, n, c["noise"])
    if c["what"] == "cl":
        return wp.to(torch.complex128), wm.to(torch.complex128)
    return wp, wm


def _members(c, seed):
    """The members of a batch: sizes and parameters from the count alone (so that every seed
    costs the same), fields from the seed."""
    r = np.random.default_rng(1000 + c["count"])
    out = []
    for i in range(c["count"]):
        nn = int(r.choice([32, 48, 64]))
        Ns = int(r.choice([50, 100, 200]))
        cl = i >= c["count"] // 2
        out.append({"n": nn, "Ns": Ns, "cl": cl, "fA": float(r.uniform(0.25, 0.5)), "chiN": float(r.uniform(12, 25)),
                    "C": 50.0 if cl else 1.0, "seed": 100000 * (int(seed) % 10000) + i})
    return out


def _member_fields(m):
    n = (m["n"],) * 3
    g = _gen(m["seed"])
    r = np.random.default_rng(m["seed"])
    X, Y, Z = _grid(n, None)
    wm = _normal(g, n, 0.1)
    for _ in range(4):
        k = r.integers(-2, 3, size=3)
        wm = wm + r.uniform(0, 2) * torch.cos(float(k[0]) * X + float(k[1]) * Y + float(k[2]) * Z + r.uniform(0, 2 * math.pi))
    wp = _normal(g, n, 0.1)
    return (wp.to(torch.complex128), wm.to(torch.complex128)) if m["cl"] else (wp, wm)


LAM, DT = 0.1, 0.01


def prepare(case, seed):
    c = dict(case)
    if c["what"] == "batch":
        ms = _members(c, seed)
        desc = [{"n": (m["n"],) * 3, "L": (m["n"] / 8.0,) * 3, "Ns": m["Ns"], "fA": m["fA"], "chiN": m["chiN"],
                 "C": m["C"], "kind": pft.PFT_CL_COMPLEX if m["cl"] else pft.PFT_SCFT_REAL, "seed": m["seed"]}
                for m in ms]
        b = _Batch(pft.pft_batch_create(desc, pft.PFT_FP32_MIXED))
        fields = [_member_fields(m) for m in ms]
        # one buffer per quantity and kind of field, a view of it for each member
        total = [sum(m["n"] ** 3 for m in ms if m["cl"] == k) for k in (False, True)]
        bufs = {q: [torch.empty(max(1, total[0]), dtype=torch.float64, device="cuda"),
                    torch.empty(max(1, total[1]), dtype=torch.complex128, device="cuda")]
                for q in ("phiA", "phiB", "wp", "wm")}
        at, views = [0, 0], []
        for m in ms:
            k, M = int(m["cl"]), m["n"] ** 3
            views.append({q: bufs[q][k][at[k]:at[k] + M] for q in bufs})
            at[k] += M
        torch.cuda.synchronize()
        return {"c": c, "b": b, "fields": fields, "views": views, "bufs": bufs}
    n = (c["nx"], c["ny"], c["nz"])
    L = (c["Lx"], c["Ly"], c["Lz"])
    cl = c["what"] == "cl"
    wp, wm = _fields(c, seed)
    s = pft.System(n, L, c["Ns"], c["fA"], c["chiN"], c["C"], pft.PFT_CL_COMPLEX if cl else pft.PFT_SCFT_REAL,
                   pft.PFT_FP64 if c["prec"] == "fp64" else pft.PFT_FP32_MIXED, seed=int(seed) & 0xFFFFFFFF,
                   scheme=pft.PFT_SCHEME_RQM4 if c["what"] == "rqm4" else pft.PFT_SCHEME_SPLIT2, checkpoint=c["ck"])
    new = lambda: torch.empty_like(wp)  # noqa: E731
    st = {"c": c, "s": s, "wp": wp, "wm": wm, "phiA": new(), "phiB": new(), "op": new(), "om": new(), "L": L}
    if c["what"] == "adjoint":
        st["GA"], st["GB"] = _loss(c, seed)
    torch.cuda.synchronize()
    return st


class _Batch:
    """Owner of a batch handle."""

    def __init__(self, h):
        self.h = h

    def __del__(self):
        try:
            pft.pft_batch_destroy(self.h)
        except Exception:
            pass


def _loss(c, seed):
    """dL/dphiA, dL/dphiB of a loss on the densities, as its user would have them."""
    g = _gen(int(seed) + 77)
    n = (c["nx"], c["ny"], c["nz"])
    return _normal(g, n, 1.0), _normal(g, n, 1.0)


def _real(t):
    return torch.view_as_real(t) if t.is_complex() else t


def run(state):
    c = state["c"]
    if c["what"] == "batch":
        h = state["b"].h
        for i, (wp, wm) in enumerate(state["fields"]):
            pft.pft_batch_set_fields(h, i, wp, wm)
        pft.pft_batch_run(h, 1, LAM, DT)
        for i, v in enumerate(state["views"]):
            pft.pft_batch_get_densities(h, i, v["phiA"], v["phiB"])
            pft.pft_batch_get_fields(h, i, v["wp"], v["wm"])
        pft.pft_batch_synchronize(h)
        return {q: [_real(t) for t in state["bufs"][q]] for q in state["bufs"]}
    s = state["s"]
    h = s.h
    if c["what"] == "cell":
        pft.pft_set_box(h, state["L"])
    pft.pft_set_fields(h, state["wp"], state["wm"])
    pft.pft_solve(h)
    pft.pft_get_densities(h, state["phiA"], state["phiB"])
    out = {}
    if c["what"] == "adjoint":
        pft.pft_adjoint(h, state["GA"], state["GB"], state["op"], state["om"])
    elif c["what"] == "cell":
        dL, _ = pft.pft_gradients(h, state["op"], state["om"])
        out["dL"] = list(dL)
    else:
        if c["what"] == "cl":
            pft.pft_field_step(h, pft.PFT_STEP_CL_EULER_MARUYAMA, DT)
        else:
            pft.pft_field_step(h, pft.PFT_STEP_SCFT_EULER, LAM)
        pft.pft_get_fields(h, state["op"], state["om"])
    obs = pft.pft_get_observables(h)
    out.update(phiA=_real(state["phiA"]), phiB=_real(state["phiB"]), op=_real(state["op"]), om=_real(state["om"]),
               obs=np.array([obs["Q"].real, obs["Q"].imag, obs["h"].real, obs["h"].imag]))
    return out


def work(case):
    """Bytes: the fields in, the densities and the new fields (or gradients) out, FP64.  Flops:
    per grid point, contour step and propagator a transform there and back (2.5 log2 M real
    flops a point each way for real fields, 5 log2 M for complex ones), the two Boltzmann
    products and the diffusion factor; the contour quadrature."""
    c = dict(case)
    items = [((m["n"],) * 3, m["Ns"], m["cl"]) for m in _members(c, 0)] if c["what"] == "batch" else \
        [((c["nx"], c["ny"], c["nz"]), c["Ns"], c["what"] == "cl")]
    by = fl = 0.0
    for n, Ns, cl in items:
        M = float(n[0] * n[1] * n[2])
        by += M * (16 if cl else 8) * 6
        if c["what"] == "adjoint":
            by += M * 16
        # an adjoint or a box gradient is at least one more march of each propagator's spectra
        marches = {"scft": 2, "cl": 2, "rqm4": 2 * RQ_WORK, "adjoint": 4, "cell": 3, "batch": 2}[c["what"]]
        per = (2 * 5.0 * math.log2(M) + 14 if cl else 2 * 2.5 * math.log2(M) + 3)
        fl += marches * M * Ns * per + M * Ns * (8 if cl else 2)
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------- 64-bit reference
def _ksq(n, L):
    k = [2 * math.pi * torch.fft.fftfreq(n[a], 1.0 / n[a], device="cuda", dtype=torch.float64) / L[a] for a in range(3)]
    return [(k[0] ** 2)[:, None, None], (k[1] ** 2)[None, :, None], (k[2] ** 2)[None, None, :]]


def _diffuse(D, cl):
    if cl:
        return lambda q: torch.fft.ifftn(D * torch.fft.fftn(q))
    n = D.shape
    Dh = D[:, :, : n[2] // 2 + 1]
    return lambda q: torch.fft.irfftn(Dh * torch.fft.rfftn(q), s=n)


def _weights(Ns, a, b, simpson):
    w = np.zeros(Ns + 1)
    m = b - a
    if m <= 0:
        return w
    if not simpson or m == 1:
        w[a:b + 1] = 1.0
        w[a] = w[b] = 0.5
        return w
    e = b if m % 2 == 0 else b - 3
    for i in range(a, e, 2):
        w[i:i + 3] += np.array([1.0, 4.0, 1.0]) / 3
    if m % 2:
        w[e:e + 4] += np.array([3.0, 9.0, 9.0, 3.0]) / 8
    return w


def _chain(wp, wm, n, L, Ns, fA, rq):
    """(step function of split step s, number of A steps) of the discrete march."""
    cl = wp.is_complex()
    NsA = int(math.floor(fA * Ns + 0.5))
    ds = 1.0 / Ns
    wA, wB = (1j * wp - wm, 1j * wp + wm) if cl else (wp - wm, wp + wm)
    kk = _ksq(n, L)
    k2 = kk[0] + kk[1] + kk[2]

    def block(h):
        K = _diffuse(torch.exp(-k2 * h), cl)
        BA, BB = torch.exp(-wA * (h / 2)), torch.exp(-wB * (h / 2))

        def step(q, s):
            B = BA if s <= NsA else BB
            return B * K(B * q)
        return step

    full = block(ds)
    if not rq:
        return full, NsA
    half = block(ds / 2)
    return lambda q, s: (4 * half(half(q, s), s) - full(q, s)) / 3, NsA


def _solve(wp, wm, n, L, Ns, fA, rq=False):
    """(Q, phiA, phiB) of the discrete solve; q is kept in part and recomputed where the
    whole history would be large."""
    step, NsA = _chain(wp, wm, n, L, Ns, fA, rq)
    K = 1 if wp.numel() * wp.element_size() * (Ns + 1) < 6e9 else max(2, int(math.sqrt(Ns)))
    q = torch.ones_like(wp)
    kept = {0: q}
    for s in range(1, Ns + 1):
        q = step(q, s)
        if s % K == 0:
            kept[s] = q
    Q = q.mean()
    cA, cB = _weights(Ns, 0, NsA, rq), _weights(Ns, NsA, Ns, rq)
    accA, accB = torch.zeros_like(wp), torch.zeros_like(wp)
    qd, seg = torch.ones_like(wp), {Ns: q}
    for m in range(Ns + 1):
        if m:
            qd = step(qd, Ns + 1 - m)
        k = Ns - m
        if k not in seg:
            base = k - k % K
            seg = {base: kept[base]}
            for j in range(base + 1, k + 1):
                seg[j] = step(seg[j - 1], j)
        p = seg[k] * qd
        accA += cA[k] * p
        accB += cB[k] * p
    return Q, accA / (Ns * Q), accB / (Ns * Q)


def _hamiltonian(wp, wm, Q, chiN, C, n, L):
    V = L[0] * L[1] * L[2]
    w = 1j * wp if wp.is_complex() else wp
    return C * (V / wp.numel()) * (wm ** 2 / chiN - w).sum() - C * V * torch.log(Q)


def _philox(seed, field, instance, M):
    """Standard normals of the library's documented noise stream at step 0."""
    m32 = np.uint64(0xFFFFFFFF)
    nb = (M + 3) // 4
    x = [np.arange(nb, dtype=np.uint64), np.full(nb, field, np.uint64), np.zeros(nb, np.uint64),
         np.full(nb, instance, np.uint64)]
    k = [seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF]
    for _ in range(10):
        a, b = x[0] * np.uint64(0xD2511F53), x[2] * np.uint64(0xCD9E8D57)
        x = [(b >> np.uint64(32)) ^ x[1] ^ np.uint64(k[0]), b & m32,
             (a >> np.uint64(32)) ^ x[3] ^ np.uint64(k[1]), a & m32]
        k = [(k[0] + 0x9E3779B9) & 0xFFFFFFFF, (k[1] + 0xBB67AE85) & 0xFFFFFFFF]
    u = [(v.astype(np.float64) + 0.5) / 4294967296.0 for v in x]
    z = []
    for r, t in ((u[0], u[1]), (u[2], u[3])):
        r = np.sqrt(-2 * np.log(r))
        z += [r * np.cos(2 * np.pi * t), r * np.sin(2 * np.pi * t)]
    return torch.from_numpy(np.stack(z, axis=-1).reshape(-1)[:M]).cuda()


def _update(wp, wm, A, B, chiN, C, n, L, seed, instance):
    """The explicit field step (Euler, or Euler-Maruyama with the library's noise)."""
    fp, fm = A + B - 1, 2 * wm / chiN + B - A
    if not wp.is_complex():
        return wp + LAM * fp, wm - LAM * fm
    std = math.sqrt(2 * DT / (C * L[0] * L[1] * L[2] / wp.numel()))
    e = [std * _philox(seed, f, instance, wp.numel()).reshape(wp.shape) for f in (0, 1)]
    return wp - DT * 1j * fp + e[0], wm - DT * fm + e[1]


def _autograd(c, wp, wm, n, L, seed):
    """Gradients of the loss <GA, phiA> + <GB, phiB> (adjoint) or of H (cell) by reverse mode."""
    wp, wm = wp.clone().requires_grad_(True), wm.clone().requires_grad_(True)
    Lt = [torch.tensor(v, dtype=torch.float64, device="cuda", requires_grad=c["what"] == "cell") for v in L]
    if c["what"] == "adjoint":
        Q, A, B = _solve_plain(wp, wm, n, Lt, c["Ns"], c["fA"])
        GA, GB = _loss(c, seed)
        gp, gm = torch.autograd.grad((GA * A + GB * B).sum(), [wp, wm])
        dL = None
    else:
        # lnQ needs the forward march only
        step, _ = _chain(wp, wm, n, Lt, c["Ns"], c["fA"], False)
        q = torch.ones_like(wp)
        for s in range(1, c["Ns"] + 1):
            q = step(q, s)
        Q = q.mean()
        H = _hamiltonian(wp, wm, Q, c["chiN"], c["C"], n, Lt)
        gp, gm, *dL = torch.autograd.grad(H, [wp, wm] + Lt)
        dL = [float(v) for v in dL]
    return gp, gm, dL


def _solve_plain(wp, wm, n, L, Ns, fA):
    step, NsA = _chain(wp, wm, n, L, Ns, fA, False)
    qs = [torch.ones_like(wp)]
    for s in range(1, Ns + 1):
        qs.append(step(qs[-1], s))
    Q = qs[-1].mean()
    cA, cB = _weights(Ns, 0, NsA, False), _weights(Ns, NsA, Ns, False)
    qd = torch.ones_like(wp)
    A = B = 0.0
    for m in range(Ns + 1):
        if m:
            qd = step(qd, Ns + 1 - m)
        p = qs[Ns - m] * qd
        A, B = A + cA[Ns - m] * p, B + cB[Ns - m] * p
    return Q, A / (Ns * Q), B / (Ns * Q)


def exact(case, seed):
    c = dict(case)
    if c["what"] == "batch":
        out = {q: [[], []] for q in ("phiA", "phiB", "wp", "wm")}
        for i, m in enumerate(_members(c, seed)):
            n, L = (m["n"],) * 3, (m["n"] / 8.0,) * 3
            wp, wm = _member_fields(m)
            Q, A, B = _solve(wp, wm, n, L, m["Ns"], m["fA"])
            p, q = _update(wp, wm, A, B, m["chiN"], m["C"], n, L, m["seed"], i)
            for name, v in (("phiA", A), ("phiB", B), ("wp", p), ("wm", q)):
                out[name][int(m["cl"])].append(_real(v).reshape(-1, 2) if m["cl"] else v.reshape(-1))
        return {k: [torch.cat(x) if x else None for x in v] for k, v in out.items()}
    n, L = (c["nx"], c["ny"], c["nz"]), (c["Lx"], c["Ly"], c["Lz"])
    M = n[0] * n[1] * n[2]
    if c["what"] == "adjoint" and M * c["Ns"] * 8 * 12 > 60e9:
        return None  # reverse mode over the whole history would not fit beside the rest
    wp, wm = _fields(c, seed)
    Q, A, B = _solve(wp, wm, n, L, c["Ns"], c["fA"], c["what"] == "rqm4")
    H = _hamiltonian(wp, wm, Q, c["chiN"], c["C"], n, L)
    out = {}
    if c["what"] in ("adjoint", "cell"):
        op, om, dL = _autograd(c, wp, wm, n, L, seed)
        if dL is not None:
            out["dL"] = dL
    else:
        op, om = _update(wp, wm, A, B, c["chiN"], c["C"], n, L, int(seed) & 0xFFFFFFFF, 0)
    h = H / (c["C"] * L[0] * L[1] * L[2])
    obs = [float(v) for z in (Q, h) for v in (z.real, z.imag if z.is_complex() else 0.0)]
    out.update(phiA=_real(A), phiB=_real(B), op=_real(op), om=_real(om), obs=np.array(obs))
    return out
