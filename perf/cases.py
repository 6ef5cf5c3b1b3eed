"""What is timed: the calls a user of this library makes, from the smallest to the largest.

Every case names a kind of call (`"call"`), the cell (FFT box, grid spacing, atoms, k-point) and the
block of bands.  Cells follow the repository's workloads: about one atom per 16000 grid points, two
projector channels (8 projectors) per atom, a cut-off sphere that fills about half of each box length.
The problem (atoms, V_loc, D, Q), the starting block and the Lanczos vector are all drawn from the seed.

Calls:
  apply    pw_hamiltonian_apply, complex128: H psi (and S psi with Q)
  bounds   pw_spectrum_bounds: Rayleigh quotients of a block and the 10-step Lanczos upper bound
  filter   pw_chebyshev_filter, complex64 ("mixed") or complex128 ("f64")
  batch    pw_batch_filter over a 2 x 2 x 2 k-point grid with ragged spheres
  rr       pw_rayleigh_ritz and the density of its lowest half (what the SCF loop takes from it: the
           Ritz vectors themselves are fixed only up to a phase each)
  solve    pw_chebfi_solve, complex128: Lanczos bound, filters and Rayleigh-Ritz steps
  density  pw_density_grad of a block
  diff     ChebFiRR + Density through torch.autograd: forward, loss and the gradients in V_loc and D
"""
import math

import numpy as np
import torch

from paper_2604_11139_gb300 import autograd as ag
from paper_2604_11139_gb300 import pwlib

DEV = "cuda"
C128, C64 = torch.complex128, torch.complex64


def _case(name, call, box, bands, *, spacing=0.25, fill=0.95, channels=2, kpt=0.0, q=False, precision="f64",
          degree=10, cycles=1, pieces=3, tuned=False):
    c = {"call": call, "n1": box[0], "n2": box[1], "n3": box[2], "bands": bands, "spacing": spacing, "fill": fill,
         "channels": channels, "kpt": kpt, "q": q, "precision": precision, "degree": degree, "cycles": cycles,
         "pieces": pieces, "tuned": tuned}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one H-apply of a toy molecule: launches and latency
        _case("apply_24_f64", "apply", (24, 24, 24), 16, spacing=10.0 / 24, fill=1.0, channels=1),
        # what every solve starts with: a serial chain of single-vector applies
        _case("bounds_64_f64", "bounds", (64, 64, 64), 32, spacing=0.22),
        # a small, ragged PAW cell off Gamma, called once and untuned
        _case("filter_48_mixed", "filter", (45, 50, 54), 37, kpt=0.21, q=True, precision="mixed", degree=8),
        # one k-point of a metal's grid, untuned
        _case("filter_72_mixed", "filter", (72, 72, 90), 128, spacing=0.222, kpt=0.125, precision="mixed"),
        # the norm-conserving cell at scale, tuned
        _case("filter_96_mixed", "filter", (96, 96, 96), 256, precision="mixed", tuned=True),
        # the headline: PAW overlap, 512 bands, two bf16 pieces as the benchmark runs it, tuned
        _case("filter_120_paw_mixed", "filter", (120, 120, 120), 512, q=True, precision="mixed", degree=12, pieces=2,
              tuned=True),
        # 8 k-points in one graph
        _case("batch_72_mixed", "batch", (72, 72, 90), 128, spacing=0.222, precision="mixed", pieces=2, tuned=True),
        # the plain FP64 filter at scale
        _case("filter_96_f64", "filter", (96, 96, 96), 256),
        # the FP64 Rayleigh-Ritz step that follows the headline filter
        _case("rr_120_paw_f64", "rr", (120, 120, 120), 512, q=True),
        # a whole small FP64 solve
        _case("solve_64_f64", "solve", (64, 64, 64), 96, spacing=0.22, cycles=2),
        # the density of an SCF step
        _case("density_96_f64", "density", (96, 96, 96), 256),
        # a gradient step of an inverse problem
        _case("diff_64_f64", "diff", (64, 64, 64), 128, spacing=0.22, cycles=2),
    ]


#: box lengths users pick: products of 2, 3 and 5
LENGTHS = (24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 80, 90, 96, 100, 108, 120)


def draw(rng):
    call = rng.choice(["apply", "bounds", "filter", "filter", "filter", "filter", "batch", "rr", "solve", "density",
                       "diff"])
    mixed = call == "batch" or (call == "filter" and rng.random() < 0.7)
    top = {"apply": 120, "bounds": 120, "filter": 120 if mixed else 96, "batch": 72, "rr": 100, "solve": 64,
           "density": 100, "diff": 64}[call]
    n = math.exp(rng.uniform(math.log(24), math.log(top)))
    box = []
    for _ in range(3):
        want = min(top, n * math.exp(rng.uniform(-0.15, 0.15)))
        box.append(min(LENGTHS, key=lambda m: abs(m - want)))
    most = {"apply": 256, "bounds": 128, "filter": 384 if mixed else 192, "batch": 128, "rr": 320, "solve": 120,
            "density": 320, "diff": 96}[call]
    least = 1 if call in ("apply", "bounds", "density") else 8
    bands = int(round(math.exp(rng.uniform(math.log(least), math.log(most)))))
    if call in ("rr", "solve", "diff"):
        # the block must stay well inside the sphere, or its Gram matrices lose rank
        npw = _npw_estimate(box, 0.9)
        bands = max(4, min(bands, int(npw / 12)))
    return _case(None, call, tuple(box), bands, spacing=round(rng.uniform(0.2, 0.3), 3),
                 fill=round(rng.uniform(0.85, 0.98), 3), channels=rng.choice([1, 2, 2]),
                 kpt=rng.choice([0.0, 0.125, 0.21]) if call not in ("diff",) else 0.0,
                 q=call not in ("diff", "bounds") and rng.random() < 0.4, precision="mixed" if mixed else "f64",
                 degree=rng.randint(4, 12) if call != "diff" else rng.randint(4, 10),
                 cycles=rng.randint(1, 2), pieces=rng.choice([2, 3]), tuned=mixed and rng.random() < 0.5)


# ---------------------------------------------------------------------------------- inputs
def _npw_estimate(box, fill):
    return 4.0 / 3.0 * math.pi * np.prod([0.25 * fill * n for n in box])


def _ecut(case):
    """|G|_max L / 2 pi = fill n / 4 along each box length."""
    return 0.5 * (math.pi * case["fill"] / (2.0 * case["spacing"])) ** 2


def _interval(case):
    """Filter interval: the lower part of the kinetic range is kept; b bounds the spectrum of these cells from above
    (the nonlocal term lifts its top to about 1.25 times the cut-off)."""
    return 0.45 * _ecut(case), 1.28 * _ecut(case)


def _problem(case, seed):
    """Cell, atoms, V_loc on the grid, D and Q, as arrays a program would have read from its input."""
    rng = np.random.default_rng(int(seed))
    box = (case["n1"], case["n2"], case["n3"])
    L = np.array([case["spacing"] * n for n in box])
    natom = max(2, int(round(np.prod(box) / 16000.0)))
    # atoms on a jittered grid: no pair is close
    g = int(math.ceil(natom ** (1.0 / 3.0) - 1e-9))
    cells = np.stack(np.meshgrid(*[np.arange(g)] * 3, indexing="ij"), -1).reshape(-1, 3)
    cells = cells[np.sort(rng.permutation(len(cells))[:natom])]
    tau = (cells + 0.5 + rng.uniform(-0.2, 0.2, cells.shape)) / g * L
    t = torch.as_tensor(tau, device=DEV)
    f = []
    for i in range(3):   # a Gaussian well of 2 Ha, width 1 bohr, with its periodic images
        x = torch.arange(box[i], device=DEV, dtype=torch.float64) * (L[i] / box[i])
        d = x[None, :, None] - t[:, i, None, None] - L[i] * torch.tensor([-1.0, 0.0, 1.0], device=DEV,
                                                                         dtype=torch.float64)
        f.append(torch.exp(-0.5 * d * d).sum(-1))
    V = -2.0 * (f[0].T @ (f[1][:, :, None] * f[2][:, None, :]).reshape(natom, -1)).reshape(box)
    sig = np.array([0.7, 1.1])[-case["channels"]:]
    nb = 4 * len(sig)
    nproj = natom * nb
    D, Q = np.zeros((nproj, nproj)), np.zeros((nproj, nproj)) if case["q"] else None
    for s in range(0, nproj, nb):
        B = rng.uniform(-0.5, 0.5, (nb, nb))
        D[s:s + nb, s:s + nb] = 0.5 * (B + B.T)
        if Q is not None:
            U, _ = np.linalg.qr(rng.standard_normal((nb, nb)))
            q = (U * rng.uniform(0.05, 0.3, nb)) @ U.T
            Q[s:s + nb, s:s + nb] = 0.5 * (q + q.T)
    kpt = case["kpt"] * np.array([1.0, -0.5, 0.25])
    return {"lattice": np.diag(L), "box": box, "ecut": _ecut(case), "vloc": V, "tau": tau, "sig": sig, "D": D, "Q": Q,
            "kpt": kpt}


def _kpoints(case, prob):
    """The k-points and cut-offs of a call: one, or a 2 x 2 x 2 grid with cut-offs that make the spheres ragged."""
    if case["call"] != "batch":
        return [(prob["kpt"], prob["ecut"])]
    rng = np.random.default_rng(31337)
    ks = [((2 * i - 1) / 4, (2 * j - 1) / 4, (2 * k - 1) / 4) for i in range(2) for j in range(2) for k in range(2)]
    return [(np.array(k), prob["ecut"] * f) for k, f in zip(ks, rng.uniform(0.86, 1.02, len(ks)))]


def _normal(seed, rows, npw):
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    return torch.randn((rows, npw), dtype=C128, device=DEV, generator=g)


def _block(case, seed, npw, kin, i=0):
    """Starting block of a filter or solve: complex normal.  What Rayleigh-Ritz and the density get has been
    through a filter: its high components have died away."""
    y = _normal(1000 * int(seed) + i, case["bands"], npw)
    if case["call"] in ("rr", "density", "diff"):
        y /= (1.0 + kin)[None, :]
    return y


def _diff_inputs(case, seed, prob):
    """Occupied bands, their weight and the target density of the inverse problem."""
    nocc = max(1, case["bands"] // 2)
    omega = float(np.prod(np.diag(prob["lattice"])))
    x = [torch.arange(n, device=DEV, dtype=torch.float64) * (2 * math.pi / n) for n in prob["box"]]
    ph = np.random.default_rng(int(seed) + 99).uniform(0, 2 * math.pi, 3)
    s = (torch.cos(x[0] + ph[0])[:, None, None] + torch.cos(x[1] + ph[1])[None, :, None]
         + torch.cos(x[2] + ph[2])[None, None, :])
    return nocc, omega, nocc / omega * (1.0 + 0.2 * s)


_TUNED = {}   # kernel forms the tuner picked, by shape: a program tunes once and keeps them


def _tune(ctx, case, prec):
    if not case["tuned"]:
        return
    key = tuple(case[k] for k in ("n1", "n2", "n3", "fill", "spacing", "kpt", "q", "channels", "bands", "pieces"))
    if key not in _TUNED:
        ctx.autotune(case["bands"], prec)
        _TUNED[key] = ctx.fft_config(prec)
    ctx.fft_config(prec, *_TUNED[key])


# ---------------------------------------------------------------------------------- calls
def prepare(case, seed):
    prob = _problem(case, seed)
    prec = pwlib.PW_MIXED if case["precision"] == "mixed" else pwlib.PW_FP64
    vloc = prob["vloc"].cpu().numpy()
    s = {"case": case, "prec": prec, "ctx": [], "psi": [], "work": []}
    for i, (k, ecut) in enumerate(_kpoints(case, prob)):
        ctx = pwlib.Context(prob["lattice"], k, ecut, prob["box"], vloc, prob["tau"], prob["sig"], prob["D"],
                            prob["Q"])
        if prec == pwlib.PW_MIXED:
            ctx.tc_config(case["pieces"])
            _tune(ctx, case, prec)
        kin = torch.as_tensor(ctx.gvectors()[1], device=DEV)
        y = _block(case, seed, ctx.npw, kin, i)
        s["ctx"].append(ctx)
        s["psi"].append(y.to(C64) if prec == pwlib.PW_MIXED else y)
        s["work"].append(torch.empty_like(s["psi"][-1]))
    npw = s["ctx"][0].npw
    if case["call"] in ("bounds", "solve", "diff"):
        s["v0"] = _normal(1000 * int(seed) + 500, 1, npw)
    if case["call"] == "apply":
        s["s_out"] = torch.empty_like(s["work"][0]) if case["q"] else None
    if case["call"] == "batch":
        s["batch"] = pwlib.Batch(s["ctx"])
    if case["call"] == "diff":
        s["nocc"], s["omega"], s["rho_t"] = _diff_inputs(case, seed, prob)
        s["V"] = prob["vloc"].clone().requires_grad_(True)
        s["D"] = torch.as_tensor(prob["D"], device=DEV).requires_grad_(True)
        s["handle"] = pwlib.Diff(s["ctx"][0], case["bands"], case["degree"], case["cycles"])
    if case["call"] == "density":
        s["w"] = np.random.default_rng(int(seed)).uniform(0.5, 2.0, case["bands"])
    return s


def run(s):
    case, ctx, prec = s["case"], s["ctx"][0], s["prec"]
    call, psi, work = case["call"], s["psi"][0], s["work"][0]
    a, b = _interval(case)
    if call == "apply":
        ctx.hamiltonian_apply(psi, work, s["s_out"], precision=prec)
        return [work] + ([s["s_out"]] if case["q"] else [])
    if call == "bounds":
        return ctx.spectrum_bounds(psi, 10, s["v0"])
    if call == "filter":
        work.copy_(psi)
        ctx.chebyshev_filter(work, case["degree"], a, b, precision=prec)
        return work
    if call == "batch":
        for w, p in zip(s["work"], s["psi"]):
            w.copy_(p)
        nk = len(s["ctx"])
        s["batch"].filter(s["work"], case["degree"], [a] * nk, [b] * nk, prec)
        return list(s["work"])
    if call == "rr":
        work.copy_(psi)
        eig, res = ctx.rayleigh_ritz(work)
        nocc = max(1, case["bands"] // 2)
        return {"eig": eig, "resid": res, "rho": ctx.density_grad(work[:nocc], [2.0] * nocc)}
    if call == "solve":
        work.copy_(psi)
        eig, res, bounds = ctx.chebfi_solve(work, case["degree"], case["cycles"], s["v0"], precision=prec)
        return {"eig": eig, "resid": res, "bounds": bounds, "psi": work}
    if call == "density":
        return ctx.density_grad(psi, s["w"])
    eig, vec = ag.chebfi_rr(s["V"], s["D"], s["handle"], psi, s["v0"], None, s["nocc"])
    rho = ag.density(vec[:s["nocc"]], 1.0 / s["omega"], ctx)
    cell = s["omega"] / rho.numel()
    loss = eig[:s["nocc"]].sum() + cell * (rho - s["rho_t"]).square().sum()
    dV, dD = torch.autograd.grad(loss, [s["V"], s["D"]])
    return {"eig": eig, "rho": rho, "loss": loss, "dV": dV, "dD": dD}


def work(case):
    """Bytes: blocks in and out, V_loc and P once.  Flops: 5 n log2 n per pruned FFT line both ways, the
    projector products, and the subspace products of Rayleigh-Ritz."""
    n = [case["n1"], case["n2"], case["n3"]]
    r = [0.25 * case["fill"] * m for m in n]
    npw, M = _npw_estimate(n, case["fill"]), case["bands"]
    nproj = 4 * case["channels"] * max(2, int(round(np.prod(n) / 16000.0)))
    nx = 2 * r[0] + 1
    lines = (math.pi * r[0] * r[1], n[2]), (nx * n[2], n[1]), (n[1] * n[2], n[0])
    fft = sum(k * 5 * m * math.log2(m) for k, m in lines)
    elem = 8 if case["precision"] == "mixed" else 16
    gemm = 8.0 * npw * nproj * M
    apply_ = 2 * M * fft + 2 * gemm
    nk = 8 if case["call"] == "batch" else 1
    base = npw * nproj * elem + np.prod(n) * elem / 2
    rr = 8.0 * npw * M * M * 4 + 40.0 * M ** 3
    call = case["call"]
    filt = case["degree"] * (apply_ + (gemm if case["q"] else 0))
    if call == "apply":
        by, fl = (2 + case["q"]) * npw * M * elem, apply_ + gemm * case["q"]
    elif call == "bounds":
        by, fl = (M + 1) * npw * elem, apply_ * (M + 10) / M
    elif call in ("filter", "batch"):
        by, fl = 2 * npw * M * elem, filt
    elif call == "rr":
        by, fl = 2 * npw * M * elem + np.prod(n) * 8, apply_ + rr + M / 2 * fft
    elif call == "solve":
        by, fl = 2 * npw * M * elem, apply_ * (M + 10) / M + case["cycles"] * (filt + apply_ + rr)
    elif call == "density":
        by, fl = npw * M * elem + np.prod(n) * 8, M * fft
        base = 0
    else:
        by, fl = 2 * npw * M * elem + 2 * np.prod(n) * 8, 3 * case["cycles"] * (filt + apply_ + rr)
    return {"bytes": float(nk * (by + base)), "flops": float(nk * fl)}


# ---------------------------------------------------------------------------------- 64-bit values
class _Plain:
    """The same problem in plain 64-bit torch: sphere, projectors, FFTs over the whole box, matrix products."""

    def __init__(self, prob, kpt, ecut):
        B = 2 * math.pi * np.linalg.inv(prob["lattice"]).T
        lim = [int(math.ceil((math.sqrt(2 * ecut) + np.linalg.norm(kpt @ B)) / B[i, i])) + 1 for i in range(3)]
        m = np.stack(np.meshgrid(*[np.arange(-v, v + 1) for v in lim], indexing="ij"), -1).reshape(-1, 3)
        q = m @ B + kpt @ B
        kin = 0.5 * (q * q).sum(1)
        keep = kin <= ecut
        m, q = m[keep], q[keep]
        self.box = prob["box"]
        n = self.box
        self.at = torch.as_tensor(((m[:, 0] % n[0]) * n[1] + m[:, 1] % n[1]) * n[2] + m[:, 2] % n[2], device=DEV)
        self.kin = torch.as_tensor(kin[keep], device=DEV)
        self.V, self.npw = prob["vloc"], len(m)
        q = torch.as_tensor(q, device=DEV)
        q2 = (q * q).sum(1)
        cols = []
        for R in torch.as_tensor(prob["tau"], device=DEV):
            ph = torch.exp(-1j * (q @ R))
            for sg in prob["sig"]:
                g = torch.exp(-0.5 * q2 * sg * sg)
                cols += [g * ph] + [-1j * q[:, c] * sg * g * ph for c in range(3)]
        P = torch.stack(cols)                       # one projector a row
        self.P = P / torch.linalg.vector_norm(P, dim=1, keepdim=True)
        self.D = torch.as_tensor(prob["D"], device=DEV).to(C128)
        self.Q = None if prob["Q"] is None else torch.as_tensor(prob["Q"], device=DEV).to(C128)
        if self.Q is not None:
            self.B = self.P.conj() @ self.P.T
            self.K = torch.linalg.inv(torch.linalg.inv(self.Q) + self.B)

    def grid(self, y):
        f = torch.zeros((y.shape[0], self.box[0] * self.box[1] * self.box[2]), dtype=C128, device=DEV)
        f = f.index_copy(1, self.at, y)
        return torch.fft.ifftn(f.reshape((-1,) + tuple(self.box)), dim=(1, 2, 3), norm="forward")

    def local(self, y, V):
        out = [torch.fft.fftn(self.grid(c) * V, dim=(1, 2, 3), norm="forward").reshape(c.shape[0], -1)[:, self.at]
               for c in y.split(64)]
        return torch.cat(out)

    def project(self, y):
        return y @ self.P.conj().T

    def h(self, y, V=None, D=None):
        V, D = self.V if V is None else V, self.D if D is None else D
        return self.kin * y + self.local(y, V) + (self.project(y) @ D.T) @ self.P

    def s(self, y):
        return y if self.Q is None else y + (self.project(y) @ self.Q.T) @ self.P

    def a(self, y, V=None, D=None):
        if self.Q is None:
            return self.h(y, V, D)
        w = self.kin * y + self.local(y, self.V)    # S^-1 (w + P z) in projector space
        z = self.project(y) @ self.D.T
        return w + (z - (self.project(w) + z @ self.B.T) @ self.K.T) @ self.P

    def filter(self, y, degree, a, b, V=None, D=None):
        c, e = 0.5 * (b + a), 0.5 * (b - a)
        prev, y = y, (self.a(y, V, D) - c * y) / e
        for _ in range(1, degree):
            prev, y = y, (2 / e) * (self.a(y, V, D) - c * y) - prev
        return y

    def quotients(self, y):
        num = (y.conj() * self.h(y)).sum(1).real
        return num / (y.conj() * self.s(y)).sum(1).real

    def upper(self, v, steps=10):
        v = v / torch.linalg.vector_norm(v)
        prev, beta, al, be = torch.zeros_like(v), 0.0, [], []
        for _ in range(steps):
            w = self.h(v)
            al.append(float((v.conj() * w).sum().real))
            w = w - al[-1] * v - beta * prev
            beta = float(torch.linalg.vector_norm(w))
            be.append(beta)
            prev, v = v, w / beta
        return float(np.linalg.eigvalsh(np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1))[-1]) + be[-1]

    def rr(self, y, V=None, D=None):
        for _ in range(2):
            L = torch.linalg.cholesky(y.conj() @ self.s(y).T)   # rows are bands: G[i, j] = <y_i | S y_j>
            y = torch.linalg.solve_triangular(L.conj(), y, upper=False)
        h = y.conj() @ self.h(y, V, D).T
        lam, U = torch.linalg.eigh(0.5 * (h + h.conj().T))
        return lam, U.T @ y

    def density(self, y, w):
        rho = 0
        for c, wc in zip(y.split(64), torch.as_tensor(w, dtype=torch.float64, device=DEV).split(64)):
            g = self.grid(c)
            rho = rho + (wc[:, None, None, None] * (g.real.square() + g.imag.square())).sum(0)
        return rho


def exact(case, seed):
    prob, call = _problem(case, seed), case["call"]
    if call == "diff" and case["bands"] * case["n1"] * case["n2"] * case["n3"] * case["degree"] > 1 << 29:
        return None                                  # the tape of plain 64-bit autograd would not fit the time
    a, b = _interval(case)
    ps = [_Plain(prob, k, e) for k, e in _kpoints(case, prob)]
    ys = [_block(case, seed, p.npw, p.kin, i) for i, p in enumerate(ps)]
    if case["precision"] == "mixed":
        ys = [y.to(C64).to(C128) for y in ys]
    p, y, M = ps[0], ys[0], case["bands"]
    v0 = _normal(1000 * int(seed) + 500, 1, p.npw) if call in ("bounds", "solve", "diff") else None
    if call == "apply":
        return [p.h(y)] + ([p.s(y)] if case["q"] else [])
    if call == "bounds":
        rq = p.quotients(y)
        return float(rq.min()), float(rq.max()), p.upper(v0)
    if call == "filter":
        return p.filter(y, case["degree"], a, b)
    if call == "batch":
        return [pk.filter(yk, case["degree"], a, b) for pk, yk in zip(ps, ys)]
    if call == "density":
        return p.density(y, np.random.default_rng(int(seed)).uniform(0.5, 2.0, M))
    if call == "rr":
        lam, x = p.rr(y)
        nocc = max(1, M // 2)
        res = torch.linalg.vector_norm(p.h(x) - lam[:, None] * p.s(x), dim=1)
        return {"eig": lam.cpu().numpy(), "resid": res.cpu().numpy(), "rho": p.density(x[:nocc], [2.0] * nocc)}
    up, cut = p.upper(v0), float(p.quotients(y).max())
    if call == "solve":
        first = cut
        for _ in range(case["cycles"]):
            lam, y = p.rr(p.filter(y, case["degree"], cut, up))
            cut = float(lam[-1])
        res = torch.linalg.vector_norm(p.h(y) - lam[:, None] * p.s(y), dim=1)
        return {"eig": lam.cpu().numpy(), "resid": res.cpu().numpy(), "bounds": np.array([up, first]), "psi": None}
    nocc, omega, rho_t = _diff_inputs(case, seed, prob)
    V = prob["vloc"].clone().requires_grad_(True)
    D = torch.as_tensor(prob["D"], device=DEV).requires_grad_(True)
    for _ in range(case["cycles"]):
        lam, y = p.rr(p.filter(y, case["degree"], cut, up, V, D.to(C128)), V, D.to(C128))
        cut = float(lam[-1].detach())
    rho = p.density(y[:nocc], [1.0 / omega] * nocc)
    loss = lam[:nocc].sum() + omega / rho.numel() * (rho - rho_t).square().sum()
    dV, dD = torch.autograd.grad(loss, [V, D])
    return {"eig": lam.detach(), "rho": rho.detach(), "loss": loss.detach(), "dV": dV, "dD": dD}
