"""complex128 passes on bands and potentials near the ends of FP64's range, against extended precision.

The line scales are powers of two, so values of any normal size are transformed alike: the tolerance is
that of ordinary values, 8 * 2^-53."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from test_gpu_fixed_fft import TOL, block, far, grid, local, make  # noqa: E402

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]
BOX = (24, 25, 27)


@pytest.mark.parametrize("psi,pot", [(1e-275, 1e6), (1e-290, 1e6), (1e-300, 1e6), (1e-300, 1e300), (1e-20, 1e-280),
                                     (1e290, 1e-290), (1e-150, 1e-150), (1e300, 1.0)])
def test_local_apply(psi, pot):
    rng = np.random.default_rng(12)
    V = pot * rng.standard_normal(BOX)
    ctx, at, kin = make(BOX, V)
    y = psi * block(rng, "normal", kin)
    v, t = torch.from_numpy(V).cuda(), torch.from_numpy(y).cuda()
    h = ctx.local_apply(v, t).cpu().numpy().astype(np.clongdouble)
    for b in range(3):
        assert far(h[b], local(BOX, at, y[b], V)) < TOL


@pytest.mark.parametrize("sa,sb", [(1e-290, 1e280), (1e-300, 1e300), (1e-150, 1e-140)])
def test_density(sa, sb):
    rng = np.random.default_rng(13)
    ctx, at, kin = make(BOX, rng.standard_normal(BOX))
    a, b = sa * block(rng, "normal", kin), sb * block(rng, "normal", kin)
    rho = ctx.density_grad(torch.from_numpy(a).cuda(), [1.0, 2.0, -0.5], torch.from_numpy(b).cuda())
    rho = rho.cpu().numpy().astype(np.longdouble).reshape(BOX) / sa / sb
    ref, size = np.zeros(BOX, np.longdouble), np.zeros(BOX, np.longdouble)
    for i, w in enumerate((1.0, 2.0, -0.5)):
        ga, gb = grid(BOX, at, a[i]) / sa, grid(BOX, at, b[i]) / sb
        ref += w * (ga.conj() * gb).real
        size += abs(w) * abs(ga) * abs(gb)
    assert float(np.sqrt((abs(rho - ref) ** 2).sum() / (size ** 2).sum())) < TOL
