"""An FP64 solve gives the same Ritz vectors, phases included, for a k-point alone and in a batch, and
the filters of a batch are not disturbed by its solves.  Tolerance 1e-9: levels here are far apart."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2604_11139_gb300 import pwlib  # noqa: E402
from paper_2604_11139_gb300 import workloads as W  # noqa: E402

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


@pytest.mark.parametrize("nband", [8, 20])
def test_vectors_of_a_batch(nband):
    prob = W.make_problem("batched_kpoints", box=(24, 25, 30), ecut=5.0, natom=3, nband=nband)
    kpts = [(0.125, 0.125, 0.25), (0.375, -0.125, 0.2), (-0.3, 0.375, -0.25)]
    ctxs = [pwlib.Context.from_problem(prob, kpt=np.array(k)) for k in kpts]
    ys = [torch.from_numpy(W.random_block(500 + i, c.npw, nband)).cuda() for i, c in enumerate(ctxs)]
    v0 = [torch.from_numpy(W.lanczos_v0(i, c.npw)[None]).cuda() for i, c in enumerate(ctxs)]
    alone, ref = [], []
    for c, y, v in zip(ctxs, ys, v0):
        x, f = y.clone(), y.clone()
        alone.append((x, c.chebfi_solve(x, 6, 2, v)[0]))
        c.chebyshev_filter(f, 6, 1.0, 20.0)
        ref.append(f)
    with pwlib.Batch(ctxs) as bt:
        xs = [torch.empty_like(y) for y in ys]
        for _ in range(2):  # the second call of each kind replays its graph
            for x, y in zip(xs, ys):
                x.copy_(y)
            eig, _ = bt.chebfi_solve(xs, 6, 2, v0)
            for i in range(3):
                assert np.abs(eig[i] - alone[i][1]).max() < 1e-11
                assert (xs[i] - alone[i][0]).abs().max().item() < 1e-9
            for x, y in zip(xs, ys):
                x.copy_(y)
            bt.filter(xs, 6, [1.0] * 3, [20.0] * 3)
            for x, f in zip(xs, ref):
                assert (torch.linalg.vector_norm(x - f) / torch.linalg.vector_norm(f)).item() < 1e-12
