"""Gradients at a size where the adjoint's products run on the tensor cores with eight digits, against
the same gradients with every FP64 product on the FP64 pipe.

Tolerance: the 1e-8 (max-norm, relative) that the FP64 gradients are held to against the oracle.  A NaN
in the adjoint of the Ritz vectors reaches both gradients in either mode."""
import numpy as np
import pytest

from paper_2604_11139_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]

from paper_2604_11139_gb300 import autograd as AG  # noqa: E402
from paper_2604_11139_gb300 import pwlib  # noqa: E402


def gradients(mode, bands, nan=False):
    prob = W.make_problem("differentiation", nband=bands)
    ctx = pwlib.Context.from_problem(prob)
    ctx.fp64_config(mode)
    handle = pwlib.Diff(ctx, bands, 4, 1)
    V = torch.from_numpy(prob.vloc.copy()).cuda().requires_grad_(True)
    D = torch.from_numpy(prob.D.copy()).cuda().requires_grad_(True)
    psi0 = torch.from_numpy(W.psi0(prob.seed, ctx.npw, bands)).cuda()
    v0 = torch.from_numpy(W.lanczos_v0(prob.seed, ctx.npw)[None]).cuda()
    nocc = bands // 2
    eig, psi = AG.chebfi_rr(V, D, handle, psi0, v0, None, nocc)
    rho = AG.density(psi[:nocc], 1.0, ctx)
    loss = eig[:nocc].sum() + rho.square().mean()
    if nan:
        loss = loss + psi.real.sum() * float("nan")
    dV, dD = torch.autograd.grad(loss, [V, D])
    return dV.cpu().numpy(), dD.cpu().numpy()


@pytest.mark.parametrize("bands", [64, 75])
def test_gradients(bands):
    for a, b in zip(gradients(1, bands), gradients(0, bands)):
        assert np.abs(a - b).max() < 1e-8 * np.abs(b).max()


def test_nan_is_not_lost():
    for g in gradients(1, 64, nan=True):
        assert np.isnan(g).any()
