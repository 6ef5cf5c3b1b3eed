"""Digit-sliced FP64 products above the size where they start (2^22 complex products), with remainders in
M, N and K, against numpy's complex128 products (their error is a hundredth of the tolerance).

V = 0, so H psi = kin psi + P (D (P^dagger psi)): the projection sums over plane waves in K splits, the
back-projection adds to H psi, the filter's first step takes it through the recurrence epilogue and
Rayleigh-Ritz computes Grams of the lower tiles only.

Tolerance of a product with seven digits: its entries, relative to the maxima of their row and column,
lack the digit products of weight 2^-63 on entries scaled to 2^-2 .. 2^-1: 6 products of two digits of
r.m.s. 37 each per element of K, 2^-51.3 in all, at most 2^-47.3 of the maxima, and the square root of the
2 K real elements in the sum.  Twice that is allowed.  For normal entries (maxima of about 4 times the
r.m.s.) a product is then within 2^-46.3 * 16 = 2^-42.3 of its r.m.s. size; two products in a row, and
Grams of rotated blocks, are held to twice that, 3.7e-13.  The eigensolver stops at off-diagonals of 1e-13
of the matrix norm."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2604_11139_gb300 import pwlib  # noqa: E402

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]
TOL = 2 * 2.0 ** -42.3


def problem(nproj, seed):
    box = (27, 30, 32)
    L = np.array([0.25 * n for n in box])
    ecut = 0.5 * (np.pi * 0.9 / 0.5) ** 2
    rng = np.random.default_rng(seed)
    args = (np.diag(L), (0.1, 0.0, -0.2), ecut, box, np.zeros(box), np.zeros((0, 3)), np.zeros(0))
    npw = pwlib.Context(*args, np.zeros((0, 0)), None).npw
    P = rng.standard_normal((npw, nproj)) + 1j * rng.standard_normal((npw, nproj))
    P /= np.linalg.norm(P, axis=0)
    B = rng.standard_normal((nproj, nproj))
    ctx = pwlib.Context(*args, 0.5 * (B + B.T), None, P=P)
    return ctx, ecut, npw, P, 0.5 * (B + B.T), np.asarray(ctx.gvectors()[1])


def err(x, ref):
    return np.linalg.norm(x - ref) / np.linalg.norm(ref)


@pytest.mark.parametrize("nproj,bands", [(61, 67), (65, 129), (130, 33)])
def test_apply_and_filter(nproj, bands):
    ctx, ecut, npw, P, D, kin = problem(nproj, nproj)
    assert nproj * bands * npw > 1 << 22
    rng = np.random.default_rng(bands)
    y = rng.standard_normal((bands, npw)) + 1j * rng.standard_normal((bands, npw))
    nl = (y @ P.conj()) @ D.T @ P.T
    t = torch.from_numpy(y).cuda()
    h = torch.empty_like(t)
    ctx.hamiltonian_apply(t, h, None)
    got = h.cpu().numpy() - kin * y
    # kin psi is rounded to 2^-53 of itself, up to 16 times the size of the nonlocal term's components
    assert err(got, nl) < TOL
    a, b = 1.0, 1.0 + 2e-3 * ecut  # a narrow interval: 1 / e lifts the nonlocal term with the rest
    ctx.chebyshev_filter(t, 1, a, b)
    c, e = 0.5 * (b + a), 0.5 * (b - a)
    assert err(t.cpu().numpy(), (kin * y + nl - c * y) / e) < TOL


@pytest.mark.parametrize("bands", [67, 129, 163])
def test_rayleigh_ritz(bands):
    ctx, ecut, npw, P, D, kin = problem(61, 3)
    assert bands * bands * npw > 1 << 22
    rng = np.random.default_rng(bands)
    y = rng.standard_normal((bands, npw)) + 1j * rng.standard_normal((bands, npw))
    t = torch.from_numpy(y).cuda()
    eig, _ = ctx.rayleigh_ritz(t)
    z = t.cpu().numpy()
    hz = kin * z + (z @ P.conj()) @ D.T @ P.T
    size = np.abs(eig).max()
    assert np.abs(z.conj() @ hz.T - np.diag(eig)).max() < (TOL + 1e-13 * np.sqrt(bands)) * size
    assert np.abs(z.conj() @ z.T - np.eye(bands)).max() < TOL
