"""The FP64 plane and x-line kernels of the boxes with kernels of their own, through the call that runs
them: an FP64 ChebFi cycle, with either plane form, against the oracle (Ritz values 1e-10 Ha, the bar of
the other ChebFi tests)."""
import numpy as np
import pytest

from oracle import pw_oracle as O
from paper_2604_11139_gb300 import workloads as W

torch = pytest.importorskip("torch")
from paper_2604_11139_gb300 import pwlib  # noqa: E402

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]
CASES = {"64": dict(name="differentiation"), "72x72x90": dict(name="batched_kpoints", kpt=(0.125, 0.375, -0.25))}


@pytest.mark.parametrize("key", list(CASES))
def test_chebfi_cycle(key):
    kw = dict(CASES[key])
    kpt = kw.pop("kpt", None)
    prob = W.make_problem(kw.pop("name"))
    ham = O.Hamiltonian.from_problem(prob, kpt=None if kpt is None else np.array(kpt))
    with pwlib.Context.from_problem(prob, kpt=None if kpt is None else np.array(kpt)) as ctx:
        assert ctx.npw == ham.npw
        y0, v0 = W.psi0(prob.seed, ctx.npw, 4), W.lanczos_v0(prob.seed, ctx.npw)
        lam, *_ = O.chebfi(ham, y0, v0, 2, 1)
        for variant in (0, 48):
            ctx.fft_config(pwlib.PW_FP64, variant=variant)
            t = torch.from_numpy(y0).cuda()
            eig, res, _ = ctx.chebfi_solve(t, 2, 1, torch.from_numpy(v0[None]).cuda())
            np.testing.assert_allclose(eig, lam, atol=1e-10, rtol=0)
            h = ham.apply_h(t.cpu().numpy())
            s = ham.apply_s(t.cpu().numpy())
            np.testing.assert_allclose(res, np.linalg.norm(h - eig[:, None] * s, axis=1), atol=1e-9)
