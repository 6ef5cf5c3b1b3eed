"""PAW filters in complex64 on boxes without kernels of their own, where pass 3 also writes the bf16
pieces of (T + V) Y: the default and another kernel form, two and three pieces, FFT batches smaller than
the block.  Against FP64 on the same problem: 1e-4 with three pieces, as in the other filter tests; two
pieces (2^-16 of each projector product) 1e-3."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2604_11139_gb300 import pwlib  # noqa: E402
from test_gpu_lines_fft import far  # noqa: E402

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


def make(box, natom):
    rng = np.random.default_rng(5)
    L = np.array([0.25 * n for n in box])
    ecut = 0.5 * (np.pi * 0.9 / 0.5) ** 2
    x = [np.cos(2 * np.pi * np.arange(n) / n) for n in box]
    V = -(x[0][:, None, None] + x[1][None, :, None] + x[2][None, None, :])
    D, Q = np.zeros((4 * natom, 4 * natom)), np.zeros((4 * natom, 4 * natom))
    for s in range(0, 4 * natom, 4):
        B = rng.uniform(-0.5, 0.5, (4, 4))
        U, _ = np.linalg.qr(rng.standard_normal((4, 4)))
        D[s:s + 4, s:s + 4] = 0.5 * (B + B.T)
        Q[s:s + 4, s:s + 4] = (U * rng.uniform(0.05, 0.3, 4)) @ U.T
    Q = 0.5 * (Q + Q.T)
    return pwlib.Context(np.diag(L), (0.1, 0.0, -0.2), ecut, box, V, rng.uniform(0, 1, (natom, 3)) * L,
                         np.array([0.8]), D, Q), ecut


@pytest.mark.parametrize("pieces", [2, 3])
@pytest.mark.parametrize("form", [None, 0, 4 + 3 * 16])
@pytest.mark.parametrize("box,bands,batch", [((45, 50, 54), 37, None), ((45, 50, 54), 40, 7), ((27, 32, 36), 64, 30),
                                             ((80, 75, 64), 9, 2), ((20, 24, 256), 19, 19)], ids=str)
def test_filter(box, bands, batch, form, pieces):
    ctx, ecut = make(box, 6)
    ctx.tc_config(pieces)
    if form is not None:
        ctx.fft_config(pwlib.PW_MIXED, variant=form)
    if batch:
        planes = len(np.unique(np.asarray(ctx.gvectors()[0]).reshape(-1, 3)[:, 0]))
        ctx.fft_config(pwlib.PW_MIXED, batch_bytes=8 * planes * box[1] * box[2] * batch)
    g = torch.Generator(device="cuda").manual_seed(2)
    y = torch.randn((bands, ctx.npw), dtype=torch.complex64, device="cuda", generator=g)
    ref = y.to(torch.complex128)
    ctx.chebyshev_filter(y, 4, 0.45 * ecut, 1.3 * ecut, precision=pwlib.PW_MIXED)
    ctx.chebyshev_filter(ref, 4, 0.45 * ecut, 1.3 * ecut)
    assert far(y, ref) < (1e-4 if pieces == 3 else 1e-3)
