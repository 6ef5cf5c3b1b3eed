"""Rayleigh-Ritz where the reduced matrix lies outside FP32's range, around the sizes from which FP32
rotations start the eigensolver.

The Ritz vectors diagonalise H and are orthonormal to 1e-11 of the largest Ritz value: a hundred times
the eigensolver's stopping tolerance, for the two Cholesky-QR passes before it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2604_11139_gb300 import pwlib  # noqa: E402

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


@pytest.mark.parametrize("scale", [1e-60, 1.0, 1e37, 1e40, 1e120])
@pytest.mark.parametrize("n", [15, 16, 17, 64, 127])
def test_rayleigh_ritz(n, scale):
    box = (24, 25, 27)
    x = [np.cos(2 * np.pi * np.arange(m) / m) for m in box]
    V = scale * (x[0][:, None, None] + 1.3 * x[1][None, :, None] + 1.7 * x[2][None, None, :])
    L = np.array([0.25 * m for m in box])
    if scale < 1:  # a cell so large that the kinetic energies are as small as V
        L = L / np.sqrt(scale)
    ecut = 0.5 * (np.pi * 0.9 * box[0] / (2 * L[0])) ** 2
    ctx = pwlib.Context(np.diag(L), (0.0, 0.0, 0.0), ecut, box, V, np.zeros((0, 3)), np.zeros(0), np.zeros((0, 0)),
                        None)
    g = torch.Generator(device="cuda").manual_seed(1)
    t = torch.randn((n, ctx.npw), dtype=torch.complex128, device="cuda", generator=g)
    eig, res = ctx.rayleigh_ritz(t)
    h = torch.empty_like(t)
    ctx.hamiltonian_apply(t, h, None)
    A = (t.conj() @ (h / scale).T).cpu().numpy()
    e = eig / scale
    assert np.all(np.diff(e) >= 0) and np.isfinite(res).all()
    assert np.abs(A - np.diag(e)).max() < 1e-11 * np.abs(e).max()
    assert np.abs((t.conj() @ t.T).cpu().numpy() - np.eye(n)).max() < 1e-11
