"""complex64 calls with few planes on boxes without kernels of their own: one launch per FFT pass, as
long as the planes have a place on the chip at once (two planes per SM, four of up to 900 points), and
results as accurate on either side of that line.  Tolerances of the other tests of these passes: 3e-6
for H psi and 1e-4 for the filter, against FP64."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2604_11139_gb300 import pwlib  # noqa: E402
from test_gpu_lines_fft import far, make  # noqa: E402

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


def planes(ctx):
    return len(np.unique(np.asarray(ctx.gvectors()[0]).reshape(-1, 3)[:, 0]))


@pytest.mark.parametrize("box,limit", [((18, 18, 18), 608), ((25, 30, 30), 608), ((25, 30, 32), 304),
                                       ((45, 54, 60), 304), ((30, 72, 75), 304)], ids=str)
def test_either_side_of_the_line(box, limit):
    ctx, ecut = make(box, 2)
    bare, _ = make(box, 0)
    most = limit // planes(ctx)
    for nb in (1, most, most + 1):
        g = torch.Generator(device="cuda").manual_seed(nb)
        y = torch.randn((nb, ctx.npw), dtype=torch.complex64, device="cuda", generator=g)
        h, ref = torch.empty_like(y), torch.empty_like(y, dtype=torch.complex128)
        bare.hamiltonian_apply(y, h, None, precision=pwlib.PW_MIXED)
        n0 = pwlib.kernel_launches()
        bare.hamiltonian_apply(y, h, None, precision=pwlib.PW_MIXED)
        assert pwlib.kernel_launches() - n0 == (3 if nb <= most else 5)
        bare.hamiltonian_apply(y.to(torch.complex128), ref, None)
        assert far(h, ref) < 3e-6
        z = y.to(torch.complex128)
        ctx.chebyshev_filter(y, 4, 0.45 * ecut, 1.3 * ecut, precision=pwlib.PW_MIXED)
        ctx.chebyshev_filter(z, 4, 0.45 * ecut, 1.3 * ecut)
        assert far(y, z) < 1e-4
