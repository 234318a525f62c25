"""The work that a user of this framework has it do, as cases that can be timed and compared.

A case is one call, or the calls of one step, of the public API in
paper_1909_01467_gb300.lsweep on seeded synthetic inputs:

  solve   one lsweep_solve on a factored handle (one source)
  step    a new medium: lsweep_update_m, lsweep_factor and one lsweep_solve
  multi   lsweep_solve_multi: k sources of one medium together
  batch   lsweep_solve_batch: several problems of different sizes, a stream each
  grad    lsweep_grad: misfit and gradient of a waveform inversion
  apply   one lsweep_apply, kept as one vector of a preconditioned basis.  A program with a
          Krylov method of its own keeps many of these; where the sweeps run in complex64 it
          keeps them in complex64, their precision, at half the memory

Solves run to the default relative residual of 1e-8.  The media, PML widths and subdomain
widths are those of the repository's workloads: constant, Gaussian-bump and random smooth
media in 2D, layers in 3D, 10 points per wavelength of the slowest speed in 2D and 8 in 3D.
"""
import math

import numpy as np
import torch

from paper_1909_01467_gb300 import lsweep as L

PRECISION = {"c64": L.LSWEEP_C64, "c128": L.LSWEEP_C128, "tf32": L.LSWEEP_C64_TF32,
             "bf16x3": L.LSWEEP_C64_BF16X3}
DEVICE = "cuda"


def case2d(kind, q, r, width, npml, medium, **more):
    """n = q * width nodes per axis in q rows and r columns of subdomains."""
    return dict({"kind": kind, "dim": 2, "n": q * width, "npml": npml, "p": 1, "q": q, "r": r,
                 "medium": medium, "precision": "c64", "side": "right", "krylov": "gmres",
                 "windows": 0, "nrhs": 1, "tol": 1e-8}, **more)


def case3d(kind, q, width, npml, **more):
    return dict({"kind": kind, "dim": 3, "n": q * width, "npml": npml, "p": 1, "q": q, "r": q,
                 "medium": "layers", "precision": "c64", "side": "right", "krylov": "gmres",
                 "windows": 0, "nrhs": 1, "tol": 1e-8}, **more)


def listed():
    return [
        # the smallest problem: 128^2, 4 x 4 subdomains, a few iterations of short levels
        dict(case2d("solve", 4, 4, 32, 10, "constant"), name="solve_128"),
        # one forward model of the 1024^2 workload: coefficients, factors and a solve
        dict(case2d("step", 16, 16, 64, 12, "bump"), name="step_1024"),
        # the paper's own 2D geometry: 101-point subdomains, PML of two wavelengths
        dict(case2d("solve", 4, 4, 101, 20, "constant"), name="solve_404_wide"),
        # complex128 sweeps on an odd grid with unequal block counts
        dict(case2d("solve", 6, 5, 55, 11, "random", precision="c128"), name="solve_330_c128"),
        # odd subdomain width, other Krylov methods: fixed memory, left preconditioning
        dict(case2d("solve", 7, 7, 51, 13, "random", krylov="bicgstab"), name="solve_357_bicgstab"),
        # a survey: eight sources of one medium solved as a block
        dict(case2d("multi", 16, 16, 32, 12, "bump", nrhs=8), name="multi_512_k8"),
        # inversion: forward and adjoint solves of six sources, misfit and gradient
        dict(case2d("grad", 8, 8, 32, 12, "bump", nrhs=6), name="grad_256"),
        # many media at once: problems of 256^2 to 512^2 nodes, each on its own stream
        dict(case2d("batch", 16, 16, 32, 16, "random", nrhs=5), name="batch_512"),
        # 3D beams spanning z: a new medium (tensor-core factor) and a solve, ragged planes
        dict(case3d("step", 4, 15, 6), name="step3d_60"),
        # one application of the 96^3 workload's sweeps (30 GB of factors)
        dict(case3d("apply", 6, 16, 6, precision="bf16x3"), name="apply3d_96"),
        # the cube decomposition: boxes cut along z too, 26 sweeps
        dict(case3d("apply", 3, 16, 6, p=3), name="apply_cube_48"),
        # one application in 2D, as a solver of the user's own calls it
        dict(case2d("apply", 12, 12, 48, 12, "bump"), name="apply_576"),
    ]


def cost(case):
    """Block products of one pass, roughly: what decides how long it takes."""
    a = apply_work(case)["flops"] * (16 if case["precision"] == "c128" else 1)
    if case["kind"] == "apply":
        return a
    per = 12 + 2 * max(case["q"], case["r"])
    return a * per * case["nrhs"] * (2 if case["kind"] == "grad" else 1)


def spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    most = max(cost(c) for c in listed())
    while True:
        if rng.random() < 0.75:
            kind = rng.choice(["solve", "solve", "step", "multi", "grad", "batch", "apply"])
            npml = rng.randint(10, 20)
            width = spread(rng, max(16, npml + 2), 101)
            q = spread(rng, 2, 16)
            r = rng.choice([q, q] + [k for k in range(2, 17) if (q * width) % k == 0 and
                                     npml + 2 <= q * width // k <= 101])
            c = case2d(kind, q, r, width, npml, rng.choice(["constant", "bump", "random"]))
            if kind in ("solve", "apply") and rng.random() < 0.25:
                c["precision"] = "c128"
            if kind == "solve":
                c["krylov"] = rng.choice(["gmres", "gmres", "gmres", "bicgstab"])
                if c["krylov"] == "gmres" and c["precision"] == "c128" and rng.random() < 0.5:
                    c["side"] = "left"
            if kind == "apply" and r == q and width % 2 == 0 and width // 2 >= npml + 2:
                c["windows"] = rng.choice([0, 1])
            if kind in ("multi", "grad", "batch"):
                c["nrhs"] = rng.randint(2, 8)
        else:
            kind = rng.choice(["step", "apply", "apply"])
            npml = rng.randint(4, 6)
            q = rng.randint(2, 6)
            c = case3d(kind, q, rng.randint(npml + 4, 18), npml,
                       precision=rng.choice(["c64", "c64", "bf16x3", "tf32"]))
            if kind == "apply" and q < 4:
                c["p"] = rng.choice([1, q])
        if c["n"] >= 48 and c["n"] ** c["dim"] <= 1100 ** 2 and cost(c) <= most:
            return c


# ------------------------------------------------------------------------------- inputs
def omega_of(case):
    """Angular frequency: 10 (3D: 8) points per wavelength of the slowest speed."""
    cmin = {"constant": 1.0, "bump": 0.6, "random": 1.0, "layers": 1.5}[case["medium"]]
    return 2 * math.pi * cmin * case["n"] / (10 if case["dim"] == 2 else 8)


def axis_points(n):
    return (torch.arange(n, dtype=torch.float64, device=DEVICE) + 0.5) / n


def medium(case, rng, n):
    """Squared slowness 1 / c^2 on the bulk grid."""
    x = axis_points(n)
    if case["medium"] == "constant":
        c = torch.ones((n,) * case["dim"], dtype=torch.float64, device=DEVICE)
    elif case["medium"] == "bump":
        x0, y0 = rng.uniform(0.25, 0.75, size=2)
        c = 1 - 0.4 * torch.exp(-((x[None, :] - x0) ** 2 + (x[:, None] - y0) ** 2) / 0.02)
    elif case["medium"] == "random":
        # white noise under a Gaussian filter of correlation length 0.1, c in [1, 3]
        w = torch.tensor(rng.standard_normal((n, n)), device=DEVICE)
        k = 2 * math.pi * torch.fft.fftfreq(n, d=1.0 / n, dtype=torch.float64, device=DEVICE)
        g = torch.fft.ifft2(torch.fft.fft2(w) *
                            torch.exp(-0.005 * (k[None, :] ** 2 + k[:, None] ** 2))).real
        c = 1 + 2 * (g - g.min()) / (g.max() - g.min())
    else:
        # eight layers in z with sinusoidal interfaces, c from 1.5 to 4.5
        t, phi = rng.uniform(0, 2 * math.pi, size=(2, 7))
        cl = rng.uniform(1.5, 4.5, size=8)
        cl = torch.tensor(1.5 + 3 * (cl - cl.min()) / (cl.max() - cl.min()), device=DEVICE)
        layer = torch.zeros((n, n, n), dtype=torch.int64, device=DEVICE)
        for k in range(7):
            zk = (k + 1) / 8 + 0.05 * torch.sin(2 * math.pi * (
                x[None, :] * math.cos(t[k]) + x[:, None] * math.sin(t[k])) + phi[k])
            layer += (x[:, None, None] > zk[None]).to(torch.int64)
        c = cl[layer]
    return (1 / c ** 2).contiguous()


def source(case, rng, n):
    """A Gaussian of standard deviation two nodes at a random position of the bulk."""
    x, dim = axis_points(n), case["dim"]
    f = torch.ones((1,) * dim, dtype=torch.float64, device=DEVICE)
    for a in range(dim):
        at = rng.uniform(0.1, 0.9)
        g = torch.exp(-((x - at) * n) ** 2 / 8) * n / math.sqrt(8 * math.pi)
        f = f * g.reshape([-1 if b == a else 1 for b in range(dim)])
    return f.contiguous()


def sizes(case):
    """Bulk sizes of the problems of a pass: a batch mixes half, three quarters and all."""
    if case["kind"] != "batch":
        return [case["n"]]
    q = case["q"]
    rows = [max(2, q // 2), max(2, 3 * q // 4), q]
    return [rows[k % 3] * (case["n"] // q) for k in range(case["nrhs"])]


def inputs(case, seed):
    """The media, bulk sources and (grad) receivers and data of a pass, from the seed alone."""
    rng = np.random.default_rng(seed)
    media = [medium(case, rng, n) for n in sizes(case)]
    if case["kind"] == "batch":
        src = [source(case, rng, n) for n in sizes(case)]
    else:
        src = [source(case, rng, case["n"]) for _ in range(case["nrhs"])]
    out = {"m": media, "f": src}
    if case["kind"] == "grad":
        # receivers on a row below the surface; observed data: the far field of point sources
        # in a medium of speed 1, as recorded from a model that is not the current one
        n, om = case["n"], omega_of(case)
        cols = torch.arange(1, n, 4, device=DEVICE)
        out["rec"] = ((n - 5) * n + cols).to(torch.int64)
        pos = torch.tensor(rng.uniform(0.1, 0.9, size=(case["nrhs"], 2)), device=DEVICE)
        xr, yr = (cols + 0.5) / n, (n - 4.5) / n
        dist = torch.sqrt((xr[None] - pos[:, :1]) ** 2 + (yr - pos[:, 1:]) ** 2) + 1.0 / n
        out["d"] = (torch.polar(0.25 * torch.sqrt(2 / (math.pi * om * dist)),
                                om * dist + math.pi / 4)).contiguous()
    return out


def blocks_of(case, n):
    """Rows and columns of the decomposition of a problem of n nodes per axis."""
    if case["kind"] != "batch":
        return case["q"], case["r"]
    rows = n // (case["n"] // case["q"])
    return rows, rows


def handle(case, n, m, stream=None):
    q, r = blocks_of(case, n)
    cdd = (case["p"], q, r) if case["p"] > 1 else (q, r)
    return L.Handle(case["dim"], n, case["npml"], cdd, omega_of(dict(case, n=n)), m,
                    precision=PRECISION[case["precision"]], tol=case["tol"], maxit=2000,
                    side=L.LSWEEP_LEFT if case["side"] == "left" else L.LSWEEP_RIGHT,
                    krylov=L.LSWEEP_BICGSTAB if case["krylov"] == "bicgstab" else L.LSWEEP_GMRES,
                    windows=case["windows"], stream=stream)


def prepare(case, seed):
    x = inputs(case, seed)
    streams = [torch.cuda.Stream() for _ in x["m"]] if case["kind"] == "batch" else [None]
    torch.cuda.synchronize()
    hs = [handle(case, n, m, s.cuda_stream if s else None)
          for n, m, s in zip(sizes(case), x["m"], streams)]
    state = {"case": case, "hs": hs, "streams": streams, "m": x["m"]}
    for h in hs:
        if case["kind"] != "step":
            L.lsweep_factor(h.h)
    if case["kind"] == "grad":
        state.update(f=torch.stack(x["f"]), rec=x["rec"], d=x["d"], g=torch.empty_like(x["m"][0]))
        return state
    f = []
    for k, s in enumerate(x["f"]):
        h = hs[k if len(hs) > 1 else 0]
        f.append(h.ext_zeros())
        torch.cuda.synchronize()
        L.lsweep_extend_source(h.h, s, f[-1])
    torch.cuda.synchronize()
    if case["kind"] == "multi":
        state.update(f=torch.stack(f), u=torch.zeros_like(torch.stack(f)))
    else:
        state.update(f=f, u=[torch.zeros_like(v) for v in f])
    if case["kind"] == "apply":
        # what a Krylov method hands to the preconditioner: a vector spread over the whole grid
        v = f[0]
        g = torch.Generator(device=DEVICE).manual_seed(seed)
        v += torch.view_as_complex(torch.randn(v.shape + (2,), dtype=torch.float64, device=DEVICE,
                                               generator=g)) * v.abs().max() * 0.1
        if case["precision"] != "c128":
            state["basis"] = torch.zeros(v.shape, dtype=torch.complex64, device=DEVICE)
    return state


def run(state):
    kind, hs, f = state["case"]["kind"], state["hs"], state["f"]
    h = hs[0].h
    if kind == "grad":
        J = L.lsweep_grad(h, f, state["rec"], state["d"], state["g"])
        return {"J": J, "grad": state["g"]}
    u = state["u"]
    if kind == "multi":
        L.lsweep_solve_multi(h, f, u)
        return u
    if kind == "batch":
        L.lsweep_solve_batch([x.h for x in hs], f, u)
        return u
    if kind == "apply":
        L.lsweep_apply(h, f[0], u[0])
        if "basis" not in state:
            return u[0]
        state["basis"].copy_(u[0])
        return state["basis"]
    if kind == "step":
        L.lsweep_update_m(h, state["m"][0])
        L.lsweep_factor(h)
    L.lsweep_solve(h, f[0], u[0])
    return u[0]


# --------------------------------------------------------------------------------- work
def axis_blocks(nb, n, npml):
    """(own0, own1, loc0, loc1, lo, hi) of the blocks of one axis: owned and local ranges on
    the extended grid, and the interval without local PML."""
    s, Ne, out = n // nb, n + 2 * npml, []
    for b in range(nb):
        o0 = 0 if b == 0 else npml + b * s
        o1 = Ne if b == nb - 1 else npml + (b + 1) * s
        out.append((o0, o1, 0 if b == 0 else o0 - 2 - npml, Ne if b == nb - 1 else o1 + 2 + npml,
                    0.0 if b == 0 else (b * s - 2) / n, 1.0 if b == nb - 1 else ((b + 1) * s + 2) / n))
    return out


def boxes(case, n=None):
    """The blocks of the z, y and x axes (2D: one block of one node along z)."""
    n = n or case["n"]
    q, r = blocks_of(case, n)
    z = axis_blocks(case["p"], n, case["npml"]) if case["dim"] == 3 else [(0, 1, 0, 1, 0.0, 1.0)]
    return [z, axis_blocks(q, n, case["npml"]), axis_blocks(r, n, case["npml"])]


def apply_work(case, n=None):
    """Bytes and flops of one application: every local solve reads the triangle of its
    symmetric inverse blocks once and multiplies each block with two vectors (2D: lines of x
    nodes, 3D: planes), in the precision of the sweeps; the input and output once."""
    ax = boxes(case, n)
    ne = (n or case["n"]) + 2 * case["npml"]
    e = 16 if case["precision"] == "c128" else 8
    by, fl = 2.0 * 16 * ne ** case["dim"], 0.0
    for z in range(len(ax[0])):
        for y in range(len(ax[1])):
            for x in range(len(ax[2])):
                size = [a[i][3] - a[i][2] for a, i in zip(ax, (z, y, x))]
                lines, b = (size[1], size[2]) if case["dim"] == 2 else (size[0], size[1] * size[2])
                visits = 1
                for a, i in zip(ax, (z, y, x)):
                    visits *= 1 + (i > 0) + (i < len(a) - 1)
                by += visits * lines * e * b * (b + 1) / 2
                fl += visits * lines * 2 * 8.0 * b * b
    k = 4 if case["windows"] else 1
    return {"bytes": k * by, "flops": k * fl}


def work(case):
    """One pass; a Krylov method makes at least one application per subdomain that a wave
    crosses on its way through the medium and back."""
    if case["kind"] == "apply":
        return apply_work(case)
    total = {"bytes": 0.0, "flops": 0.0}
    for n in sizes(case):
        w = apply_work(case, n)
        its = max(len(a) for a in boxes(case, n)) * (2 if case["kind"] == "grad" else 1)
        share = case["nrhs"] if case["kind"] in ("multi", "grad") else 1
        total["bytes"] += its * w["bytes"]              # a block solve shares the factors
        total["flops"] += its * w["flops"] * share
        if case["kind"] == "step":
            for z in boxes(case, n)[0]:
                for y in boxes(case, n)[1]:
                    for x in boxes(case, n)[2]:
                        s = [v[3] - v[2] for v in (z, y, x)]
                        lines, b = (s[1], s[2]) if case["dim"] == 2 else (s[0], s[1] * s[2])
                        total["flops"] += lines * 4.0 * b ** 3   # symmetric complex inverse
    return total


# -------------------------------------------------------------------- 64-bit reference
class Box:
    """The PML-extended symmetric operator -div(Lambda grad) - omega^2 m / prod(alpha) on a box
    of the extended grid: diagonal and the couplings to the next node along z, y, x."""

    def __init__(self, case, n, m_ext, ax):
        om, npml = omega_of(dict(case, n=n)), case["npml"]
        C, d, h = math.log(om), npml / n, 1.0 / n

        def alpha(p, lo, hi):
            out = torch.clamp(lo - p, min=0) + torch.clamp(p - hi, min=0)
            s = C / d * (out / d) ** 3
            return 1 / torch.complex(torch.ones_like(s), s)

        nodes, faces = [], []
        for k, (o0, o1, l0, l1, lo, hi) in enumerate(ax):
            shape = [1, 1, 1]
            shape[k] = -1
            if case["dim"] == 2 and k == 0:
                one = torch.ones((1, 1, 1), dtype=torch.complex128, device=DEVICE)
                nodes.append(one)
                faces.append(None)
                continue
            i = torch.arange(l0, l1 + 1, dtype=torch.float64, device=DEVICE) - npml
            nodes.append(alpha((i[:-1] + 0.5) * h, lo, hi).reshape(shape))
            faces.append(alpha(i * h, lo, hi).reshape(shape))
        self.shape = tuple(a[3] - a[2] for a in ax)
        m = m_ext[tuple(slice(a[2], a[3]) for a in ax)]
        self.prod = nodes[0] * nodes[1] * nodes[2]
        self.diag = -(om ** 2) * m / self.prod
        self.c = [None] * 3
        for k in range(3):
            if faces[k] is None:
                continue
            S = (faces[k] / (nodes[k - 1] * nodes[k - 2]) / h ** 2).expand(
                [s + (a == k) for a, s in enumerate(self.shape)])
            self.diag = self.diag + S.narrow(k, 0, self.shape[k]) + S.narrow(k, 1, self.shape[k])
            self.c[k] = -S.narrow(k, 1, self.shape[k] - 1)

    def matvec(self, u):
        y = self.diag * u
        for k in range(3):
            if self.c[k] is None:
                continue
            s = self.shape[k]
            y.narrow(k, 0, s - 1).add_(self.c[k] * u.narrow(k, 1, s - 1))
            y.narrow(k, 1, s - 1).add_(self.c[k] * u.narrow(k, 0, s - 1))
        return y

    def lines(self):
        """Blocks of the operator over its lines (2D: rows, 3D: planes): (L, b, b) and the
        couplings of consecutive lines (L - 1, b)."""
        Z, Y, X = self.shape
        n = (Y, X) if Z == 1 else (Z, Y * X)
        A = torch.diag_embed(self.diag.reshape(n))
        cx = torch.zeros(self.shape, dtype=torch.complex128, device=DEVICE)
        cx[:, :, :-1] = self.c[2]
        v = cx.reshape(n)[:, :-1]
        A.diagonal(1, 1, 2).add_(v)
        A.diagonal(-1, 1, 2).add_(v)
        if Z == 1:
            return A, self.c[1].reshape(n[0] - 1, n[1])
        cy = torch.zeros(self.shape, dtype=torch.complex128, device=DEVICE)
        cy[:, :-1] = self.c[1]
        v = cy.reshape(n)[:, :n[1] - X]
        A.diagonal(X, 1, 2).add_(v)
        A.diagonal(-X, 1, 2).add_(v)
        return A, self.c[0].reshape(n[0] - 1, n[1])


class Direct:
    """Block-tridiagonal elimination of boxes of one shape, side by side."""

    def __init__(self, group):
        parts = [b.lines() for b in group]
        self.c = torch.stack([c for _, c in parts], 1)                # (L - 1, boxes, b)
        A = torch.stack([a for a, _ in parts], 1)
        del parts
        self.D = A
        for k in range(A.shape[0]):
            if k:
                c = self.c[k - 1]
                A[k] -= c[:, :, None] * A[k - 1] * c[:, None, :]
            A[k] = torch.linalg.inv(A[k])

    def solve(self, which, g):
        """g: (lines, boxes of `which`, b, right-hand sides)"""
        D, c = self.D, self.c[:, which, :, None]
        y = []
        for k in range(g.shape[0]):
            v = g[k] - c[k - 1] * y[-1] if k else g[0]
            y.append(D[k][which] @ v)
        for k in range(g.shape[0] - 2, -1, -1):
            y[k] = y[k] - D[k][which] @ (c[k] * y[k + 1])
        return torch.stack(y)


def extend(case, n, m):
    """m copied outwards along the normals onto the extended grid, as (z, y, x)."""
    i = torch.clamp(torch.arange(n + 2 * case["npml"], device=DEVICE) - case["npml"], 0, n - 1)
    if case["dim"] == 2:
        return m[i][:, i][None]
    return m[i][:, i][:, :, i]


def embed(case, n, f):
    """f, zero-extended onto the extended grid and complex, as (z, y, x)."""
    p, ne = case["npml"], n + 2 * case["npml"]
    out = torch.zeros((ne,) * case["dim"], dtype=torch.complex128, device=DEVICE)
    out[(slice(p, p + n),) * case["dim"]] = f
    return out[None] if case["dim"] == 2 else out


def whole(case, n):
    ne = n + 2 * case["npml"]
    a = (0, ne, 0, ne, 0.0, 1.0)
    return [a if case["dim"] == 3 else (0, 1, 0, 1, 0.0, 1.0), a, a]


def direct(case, n, m, fs):
    """Solutions of the whole problem and its operator."""
    A = Box(case, n, extend(case, n, m), whole(case, n))
    lines = A.shape[0] if case["dim"] == 3 else A.shape[1]
    g = torch.stack([f.reshape(lines, -1) for f in fs], -1)[:, None]
    lu = Direct([A])
    u = lu.solve([0], g)[:, 0]
    return [u[..., k].reshape((A.shape if case["dim"] == 3 else A.shape[1:]))
            for k in range(len(fs))], A, lu


def sweeps(case, m, r):
    """The L-sweeps approximate inverse applied to r: local solves, then for every direction d
    of {-1, 0, 1}^3 the boxes front by front, their sources made from the traces of the boxes
    upstream (the two planes either side of the shared face)."""
    n, ax = case["n"], boxes(case)
    nb = [len(a) for a in ax]
    m_ext = extend(case, n, m)
    every = [(z, y, x) for z in range(nb[0]) for y in range(nb[1]) for x in range(nb[2])]
    loc = {t: Box(case, n, m_ext, [ax[k][t[k]] for k in range(3)]) for t in every}
    groups = {}
    for t in every:
        groups.setdefault(loc[t].shape, []).append(t)
    lus = {s: Direct([loc[t] for t in g]) for s, g in groups.items()}
    out = torch.zeros(m_ext.shape, dtype=torch.complex128, device=DEVICE)
    own = {t: tuple(slice(ax[k][t[k]][0] - ax[k][t[k]][2], ax[k][t[k]][1] - ax[k][t[k]][2])
                    for k in range(3)) for t in every}
    glob = {t: tuple(slice(*ax[k][t[k]][:2]) for k in range(3)) for t in every}
    traces = {}

    def plane(t, k, s):                    # lower plane across face (k, s), local index
        return own[t][k].stop - 1 if s > 0 else own[t][k].start - 1

    def solve(tasks):                      # [(box, source)] -> fields added and traced
        for s, g in groups.items():
            mine = [(t, v) for t, v in tasks if loc[t].shape == s]
            if not mine:
                continue
            lines = s[0] if case["dim"] == 3 else s[1]
            v = torch.stack([v.reshape(lines, -1, 1) for _, v in mine], 1)
            which = [g.index(t) for t, _ in mine]
            u = lus[s].solve(which, v)
            for k, (t, _) in enumerate(mine):
                yield t, u[:, k].reshape(s)

    def keep(d, t, u):
        out[glob[t]] += u[own[t]]
        for k in range(3):
            for s in ((d[k],) if d[k] else (-1, 1)):
                if not 0 <= t[k] + s < nb[k]:
                    continue
                fam = (k, s, tuple(0 if a == k else d[a] for a in range(3)), t)
                w = u.narrow(k, plane(t, k, s), 2)
                traces[fam] = traces[fam] + w if d[k] else w.clone()

    first = []
    for t in every:
        g = torch.zeros(loc[t].shape, dtype=torch.complex128, device=DEVICE)
        g[own[t]] = r[glob[t]]
        first.append((t, g))
    for t, u in solve(first):
        keep((0, 0, 0), t, u)
    ways = [(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)]
    for d in sorted(ways, key=lambda d: sum(map(abs, d))):
        if d == (0, 0, 0):
            continue
        fronts = {}
        for t in every:
            if all(d[k] == 0 or (t[k] > 0 if d[k] > 0 else t[k] < nb[k] - 1) for k in range(3)):
                fronts.setdefault(sum(t[k] * d[k] for k in range(3)), []).append(t)
        for at in sorted(fronts):
            tasks = []
            for t in fronts[at]:
                box = loc[t]
                Q = [slice(own[t][k].start, None) if d[k] > 0 else
                     slice(0, own[t][k].stop) if d[k] < 0 else slice(None) for k in range(3)]
                w = torch.zeros(box.shape, dtype=torch.complex128, device=DEVICE)
                for k in (2, 1, 0):        # x, then y, then z: the later one is kept
                    if not d[k]:
                        continue
                    up = tuple(t[a] - d[a] * (a == k) for a in range(3))
                    fam = (k, d[k], tuple(0 if a == k else d[a] for a in range(3)), up)
                    to, fr = list(Q), list(Q)
                    p = plane(t, k, -d[k])
                    to[k], fr[k] = slice(p, p + 2), slice(None)
                    w[tuple(to)] = traces[fam][tuple(fr)]
                chi = torch.zeros(box.shape, dtype=torch.float64, device=DEVICE)
                chi[tuple(Q)] = 1
                tasks.append((t, box.matvec(chi * w) - chi * box.matvec(w)))
            for t, u in list(solve(tasks)):
                keep(d, t, u)
    return out


def exact(case, seed):
    """What run() returns in 64 bits, from plain torch; None where that takes too long."""
    dim, ne = case["dim"], case["n"] + 2 * case["npml"]
    if case["kind"] == "apply":
        ax = boxes(case)
        vol = 1.0
        for k, a in enumerate(ax):
            vol *= sum((b[3] - b[2]) ** (1 if k == (0 if dim == 3 else 1) else 3) for b in a)
        if case["windows"] or vol > 1.2e12:
            return None
        x, s = inputs(case, seed), prepare(case, seed)
        r = s["f"][0].clone()
        for h in s["hs"]:
            h.close()
        z = sweeps(case, x["m"][0], r if dim == 3 else r[None])
        return z if dim == 3 else z[0]
    if ne ** 4 > 1e11 if dim == 2 else ne ** 7 > 6e11:
        return None
    x = inputs(case, seed)
    if case["kind"] == "batch":
        return [direct(case, n, m, [embed(case, n, f)])[0][0]
                for n, m, f in zip(sizes(case), x["m"], x["f"])]
    n, m = case["n"], x["m"][0]
    us, A, lu = direct(case, n, m, [embed(case, n, f) for f in x["f"]])
    if case["kind"] == "grad":
        i = x["rec"]
        at = (i // n + case["npml"]) * ne + i % n + case["npml"]
        res = torch.stack([u.reshape(-1)[at] for u in us]) - x["d"]
        back = []
        for k in range(len(us)):
            v = torch.zeros(ne * ne, dtype=torch.complex128, device=DEVICE)
            v.index_add_(0, at, res[k].conj())
            back.append(v)
        v = lu.solve([0], torch.stack([b.reshape(ne, ne) for b in back], -1)[:, None])[:, 0]
        g = sum((v[..., k] * us[k] / A.prod[0]).real for k in range(len(us))) * omega_of(case) ** 2
        i = torch.clamp(torch.arange(ne, device=DEVICE) - case["npml"], 0, n - 1)
        to = (i[:, None] * n + i[None]).reshape(-1)
        grad = torch.zeros(n * n, dtype=torch.float64, device=DEVICE).index_add_(0, to, g.reshape(-1))
        return {"J": 0.5 * float((res.abs() ** 2).sum()), "grad": grad.reshape(n, n)}
    if case["kind"] == "multi":
        return torch.stack(us)
    return us[0]
