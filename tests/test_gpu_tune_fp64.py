"""pw_autotune in FP64 on boxes of the fixed-point passes: the plane form, which only FP64 solves use
there, stays what it was, so that tuning does not change a solve's vectors."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2604_11139_gb300 import pwlib  # noqa: E402
from paper_2604_11139_gb300 import workloads as W  # noqa: E402

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


@pytest.mark.parametrize("variant", [0, 48])
@pytest.mark.parametrize("box", [(24, 24, 24), (64, 64, 64), (25, 27, 30)], ids=str)
def test_tuning_keeps_the_plane_form(box, variant):
    prob = W.make_problem("batched_kpoints", box=box, ecut=4.0, natom=2, nband=8)
    with pwlib.Context.from_problem(prob) as ctx:
        ctx.fft_config(pwlib.PW_FP64, variant=variant)
        y = torch.from_numpy(W.random_block(1, ctx.npw, 8)).cuda()
        v0 = torch.from_numpy(W.lanczos_v0(1, ctx.npw)[None]).cuda()
        a, b = y.clone(), y.clone()
        ctx.chebfi_solve(a, 4, 1, v0)
        for _ in range(4):
            ctx.autotune(8, pwlib.PW_FP64)
            assert ctx.fft_config(pwlib.PW_FP64)[1] == variant
        ctx.chebfi_solve(b, 4, 1, v0)
        assert torch.equal(a, b)
