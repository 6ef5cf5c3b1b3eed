"""complex64 FFT passes for any two-stage box: H-apply and filter against FP64 on the same problem.

The FP64 path is accurate to 1e-15 here, so the differences are the complex64 path's own rounding: a
transform there and back is about 60 roundings of 2^-24 in sequence, within 3e-6 of the block's
norm; the filter is held to the 1e-4 of the other filter tests."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2604_11139_gb300 import pwlib  # noqa: E402

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]

# every radix (16 to 2), one chunk of 32 lines and several with a remainder, lengths at the top of
# the range, and boxes where only some passes have a kernel for the length
BOXES = [(18, 24, 25), (27, 32, 36), (40, 45, 48), (45, 50, 54), (64, 72, 75), (80, 90, 20), (96, 30, 100),
         (24, 108, 120), (240, 18, 20), (18, 240, 24), (20, 24, 256), (256, 20, 18), (25, 72, 90), (72, 20, 27),
         (16, 64, 64), (16, 20, 24)]


def make(box, atoms):
    rng = np.random.default_rng(3)
    L = np.array([0.25 * n for n in box])
    ecut = 0.5 * (np.pi * 0.9 / 0.5) ** 2
    x = [np.cos(2 * np.pi * np.arange(n) / n) for n in box]
    V = -(x[0][:, None, None] + x[1][None, :, None] + x[2][None, None, :])
    D = np.zeros((4 * atoms, 4 * atoms))
    for s in range(0, 4 * atoms, 4):
        B = rng.uniform(-0.5, 0.5, (4, 4))
        D[s:s + 4, s:s + 4] = 0.5 * (B + B.T)
    tau = rng.uniform(0, 1, (atoms, 3)) * L
    return pwlib.Context(np.diag(L), (0.1, 0.0, -0.2), ecut, box, V, tau, np.array([0.8] if atoms else []), D, None), ecut


def far(x, ref):
    return (torch.linalg.vector_norm(x.to(ref.dtype) - ref, dim=1) / torch.linalg.vector_norm(ref, dim=1)).max().item()


@pytest.mark.parametrize("box", BOXES, ids=str)
@pytest.mark.parametrize("form", [0, 4 + 3 * 16])
def test_apply(box, form):
    ctx, _ = make(box, 0)
    ctx.fft_config(pwlib.PW_MIXED, variant=form)
    g = torch.Generator(device="cuda").manual_seed(1)
    y = torch.randn((5, ctx.npw), dtype=torch.complex64, device="cuda", generator=g)
    h, ref = torch.empty_like(y), torch.empty_like(y, dtype=torch.complex128)
    ctx.hamiltonian_apply(y, h, None, precision=pwlib.PW_MIXED)
    ctx.hamiltonian_apply(y.to(torch.complex128), ref, None)
    assert far(h, ref) < 3e-6


@pytest.mark.parametrize("box", BOXES, ids=str)
@pytest.mark.parametrize("form", [0, 4 + 3 * 16])
def test_filter(box, form):
    ctx, ecut = make(box, 2)
    ctx.fft_config(pwlib.PW_MIXED, variant=form)
    g = torch.Generator(device="cuda").manual_seed(2)
    y = torch.randn((5, ctx.npw), dtype=torch.complex64, device="cuda", generator=g)
    ref = y.to(torch.complex128)
    ctx.chebyshev_filter(y, 4, 0.45 * ecut, 1.3 * ecut, precision=pwlib.PW_MIXED)
    ctx.chebyshev_filter(ref, 4, 0.45 * ecut, 1.3 * ecut, precision=pwlib.PW_FP64)
    assert far(y, ref) < 1e-4
