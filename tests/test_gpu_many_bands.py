"""More bands than one launch has in blockIdx.y (65535), with FFT batches that hold them all: H psi for a
constant potential c is (kin + c) psi.  Tolerances: those of the transforms' own tests, 3e-6 of a
component's size for complex64 and 1e-13 for complex128."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2604_11139_gb300 import pwlib  # noqa: E402

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


@pytest.mark.parametrize("bands", [65535, 65536, 70000])
@pytest.mark.parametrize("precision", [pwlib.PW_FP64, pwlib.PW_MIXED], ids=["f64", "mixed"])
@pytest.mark.parametrize("box,batch_bytes", [((10, 10, 10), None), ((9, 8, 10), None), ((18, 10, 18), 1 << 40),
                                             ((18, 18, 18), 1 << 60)], ids=str)
def test_apply(box, batch_bytes, precision, bands):
    L = np.array([0.25 * n for n in box])
    ctx = pwlib.Context(np.diag(L), (0.1, 0.0, -0.2), 0.5 * (np.pi * 0.9 / 0.5) ** 2, box, np.full(box, 1.5),
                        np.zeros((0, 3)), np.zeros(0), np.zeros((0, 0)), None)
    if batch_bytes:
        ctx.fft_config(precision, batch_bytes=batch_bytes)
    dt = torch.complex128 if precision == pwlib.PW_FP64 else torch.complex64
    g = torch.Generator(device="cuda").manual_seed(1)
    y = torch.randn((bands, ctx.npw), dtype=dt, device="cuda", generator=g)
    h = torch.full_like(y, float("nan"))
    ctx.hamiltonian_apply(y, h, None, precision=precision)
    ctx.sync()
    kin = torch.as_tensor(np.asarray(ctx.gvectors()[1]), device="cuda")
    tol = 1e-13 if precision == pwlib.PW_FP64 else 3e-6
    size = float(kin.max() + 1.5) * y.abs().max().item()
    assert (h - (kin + 1.5) * y).abs().max().item() < tol * size
