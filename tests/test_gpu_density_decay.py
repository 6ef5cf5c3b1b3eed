"""complex128 density, point by point, of bands that decay by ten orders of magnitude within the cell.

Tolerance: an amplitude is off by at most TOL = 8 * 2^-53 of the band's largest one (the bound of the
transforms' own tests), the product and the sum over bands by TOL of themselves:
|d rho| <= sum_b |w_b| (|a| db + |b| da + da db + TOL |a| |b|), da = TOL max|a|, db = TOL max|b|."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2604_11139_gb300 import pwlib  # noqa: E402

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]
TOL = 8 * 2.0 ** -53


def decaying(box, axis):
    """Two Gaussian bands, 1.5 and 1.7 bohr wide along `axis`, smooth along the others."""
    L = np.array([0.25 * n for n in box])
    ecut = 0.5 * (np.pi * 0.9 / 0.5) ** 2
    ctx = pwlib.Context(np.diag(L), (0.0, 0.0, 0.0), ecut, box, np.zeros(box), np.zeros((0, 3)), np.zeros(0),
                        np.zeros((0, 0)), None)
    m, kin = ctx.gvectors()
    m, kin = np.asarray(m).reshape(-1, 3), np.asarray(kin)
    g = 2 * np.pi * m[:, axis] / L[axis]
    low = (abs(np.delete(m, axis, 1)) <= 2).all(1)
    y = [low * np.exp(-0.5 * (g * s) ** 2 - 0.3 * kin - 1j * g * c) for s, c in ((1.5, 3.0), (1.7, 7.5))]
    return ctx, tuple(m[:, i] % box[i] for i in range(3)), np.array(y)


@pytest.mark.parametrize("two", [False, True])
@pytest.mark.parametrize("box,axis", [((96, 24, 25), 0), ((25, 96, 24), 1), ((24, 25, 96), 2), ((120, 18, 20), 0)],
                         ids=str)
def test_density_where_the_bands_have_died_away(box, axis, two):
    ctx, at, a = decaying(box, axis)
    b = a[::-1].copy() if two else a
    w = [1.5, -0.5]
    rho = ctx.density_grad(torch.from_numpy(a).cuda(), w, torch.from_numpy(b).cuda() if two else None)
    rho = rho.cpu().numpy().reshape(box)

    def grid(y):
        f = np.zeros(box, np.clongdouble)
        f[at] = y
        return np.fft.ifftn(f, norm="forward")

    ref, tol = np.zeros(box, np.longdouble), np.zeros(box, np.longdouble)
    for i in range(2):
        ga, gb = grid(a[i]), grid(b[i])
        ma, mb = abs(ga), abs(gb)
        da, db = TOL * ma.max(), TOL * mb.max()
        assert ma.min() < 1e-10 * ma.max()
        ref += w[i] * (ga.conj() * gb).real
        tol += abs(w[i]) * (ma * db + mb * da + da * db + TOL * ma * mb)
    assert (abs(rho - ref) <= tol).all()
