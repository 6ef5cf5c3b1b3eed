"""complex128 local H-apply and density on the fixed-point FFT passes against extended precision.

The relative tolerance is 8 * 2^-53: one FP64 rounding each of 1/n1n2n3 and of V / n1n2n3, of the
values stored between the five passes and of the result, the fixed-point transforms between them
being closer than that."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2604_11139_gb300 import pwlib  # noqa: E402

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]
TOL = 8 * 2.0 ** -53

# every radix (16 to 2), one chunk of 32 lines and several with a remainder, lengths at the top of the range
BOXES = [(18, 24, 25), (27, 32, 36), (40, 45, 48), (50, 54, 60), (64, 72, 75), (80, 90, 20), (96, 30, 100),
         (24, 108, 120), (240, 18, 20), (18, 240, 24), (20, 24, 256), (256, 20, 18)]


def make(box, V, fill=0.9):
    L = np.array([0.25 * n for n in box])
    ecut = 0.5 * (np.pi * fill / 0.5) ** 2
    z = np.zeros((0, 0))
    ctx = pwlib.Context(np.diag(L), (0.1, 0.0, -0.2), ecut, box, V, np.zeros((0, 3)), np.zeros(0), z, None)
    m, kin = ctx.gvectors()
    m = np.asarray(m).reshape(-1, 3)
    return ctx, tuple(m[:, i] % box[i] for i in range(3)), np.asarray(kin)


def grid(box, at, y):
    f = np.zeros(box, np.clongdouble)
    f[at] = y
    return np.fft.ifftn(f, norm="forward")


def local(box, at, y, V):
    return np.fft.fftn(grid(box, at, y) * V.astype(np.longdouble), norm="forward")[at]


def block(rng, kind, kin):
    y = rng.standard_normal((3, kin.size)) + 1j * rng.standard_normal((3, kin.size))
    if kind == "decay":      # a filtered band: the low components carry it
        y *= np.exp(-20.0 * kin / kin.max())
    elif kind == "single":   # one component, the others 1e-6 of it
        y *= 1e-6
        y[:, kin.size // 2] = 1.0
    elif kind == "peak":     # all in phase: a delta function on the grid
        y = np.ones_like(y)
    elif kind == "tiny":
        y *= 1e-200
    elif kind == "large":
        y *= 1e200
    return y


def far(x, ref):
    s = np.longdouble(1) / abs(ref).max()
    return float(np.sqrt((abs((x - ref) * s) ** 2).sum() / (abs(ref * s) ** 2).sum()))


@pytest.mark.parametrize("box", BOXES, ids=str)
@pytest.mark.parametrize("kind", ["normal", "decay", "single", "peak", "tiny", "large"])
def test_local_apply(box, kind):
    rng = np.random.default_rng(7)
    V = 1e6 * rng.standard_normal(box)  # far above the kinetic term, which is not part of the comparison
    ctx, at, kin = make(box, V)
    y = block(rng, kind, kin)
    t = torch.from_numpy(y).cuda()
    h = torch.empty_like(t)
    ctx.hamiltonian_apply(t, h, None)
    h = h.cpu().numpy().astype(np.clongdouble) - kin.astype(np.longdouble) * y
    for b in range(3):
        assert far(h[b], local(box, at, y[b], V)) < TOL


def test_potential_of_wide_range():
    box = (24, 25, 27)
    rng = np.random.default_rng(8)
    V = 1e6 * rng.standard_normal(box) * np.exp(rng.uniform(-10, 2, box))
    ctx, at, kin = make(box, V)
    y = block(rng, "normal", kin)
    t = torch.from_numpy(y).cuda()
    h = torch.empty_like(t)
    ctx.hamiltonian_apply(t, h, None)
    h = h.cpu().numpy().astype(np.clongdouble) - kin.astype(np.longdouble) * y
    for b in range(3):
        assert far(h[b], local(box, at, y[b], V)) < TOL


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_not_finite_stays_in_its_band(bad):
    box = (24, 25, 27)
    rng = np.random.default_rng(9)
    V = rng.standard_normal(box)
    ctx, at, kin = make(box, V)
    y = block(rng, "normal", kin)
    t = torch.from_numpy(y).cuda()
    h0, h = torch.empty_like(t), torch.empty_like(t)
    ctx.hamiltonian_apply(t, h0, None)
    t[1, 5] = bad
    ctx.hamiltonian_apply(t, h, None)
    assert not torch.isfinite(torch.view_as_real(h[1])).all(-1).any()
    assert torch.equal(h[0], h0[0]) and torch.equal(h[2], h0[2])
    z = torch.zeros_like(t)
    ctx.hamiltonian_apply(z, h, None)
    assert not h.abs().any()


@pytest.mark.parametrize("box,two", [((18, 24, 25), False), ((18, 24, 25), True), ((96, 30, 100), False),
                                     ((96, 30, 100), True), ((240, 18, 20), False)], ids=str)
def test_density(box, two):
    rng = np.random.default_rng(10)
    ctx, at, kin = make(box, rng.standard_normal(box))
    a, b = block(rng, "decay", kin), block(rng, "decay", kin)
    w = rng.uniform(0.5, 2.0, 3)
    rho = ctx.density_grad(torch.from_numpy(a).cuda(), w, torch.from_numpy(b).cuda() if two else None)
    rho = np.asarray(rho.cpu().numpy() if hasattr(rho, "cpu") else rho).reshape(box)
    ref, size = np.zeros(box, np.longdouble), np.zeros(box, np.longdouble)
    for i in range(3):
        ga, gb = grid(box, at, a[i]), grid(box, at, b[i] if two else a[i])
        ref += w[i] * (ga.conj() * gb).real
        size += w[i] * abs(ga) * abs(gb)
    assert float(np.sqrt((abs(rho - ref) ** 2).sum() / (size ** 2).sum())) < TOL


@pytest.mark.parametrize("kind", ["normal", "single", "peak"])
def test_density_of_uneven_lines(kind):
    box = (45, 50, 54)
    rng = np.random.default_rng(11)
    ctx, at, kin = make(box, rng.standard_normal(box))
    a = block(rng, kind, kin)
    rho = ctx.density_grad(torch.from_numpy(a).cuda(), [1.0, -0.5, 2.0]).cpu().numpy().reshape(box)
    ref, size = np.zeros(box, np.longdouble), np.zeros(box, np.longdouble)
    for i, w in enumerate((1.0, -0.5, 2.0)):
        g = abs(grid(box, at, a[i])) ** 2
        ref += w * g
        size += abs(w) * g
    assert float(np.sqrt((abs(rho - ref) ** 2).sum() / (size ** 2).sum())) < TOL
