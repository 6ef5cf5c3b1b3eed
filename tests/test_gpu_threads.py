"""Contexts of different boxes used at the same time by different host threads, each on its own stream:
every call succeeds and gives what it gives alone (the transforms add in a fixed order: equal bits)."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2604_11139_gb300 import pwlib  # noqa: E402

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]

# boxes that share kernels, of different line lengths: with kernels of their own, and without
SETS = {"special": [(64, 64, 64), (96, 96, 96), (72, 72, 90)], "any": [(20, 24, 256), (48, 45, 50), (200, 20, 24)],
        "one_stage": [(16, 12, 40), (16, 12, 10), (9, 10, 300)]}


@pytest.mark.parametrize("precision", [pwlib.PW_FP64, pwlib.PW_MIXED], ids=["f64", "mixed"])
@pytest.mark.parametrize("key", list(SETS))
def test_contexts_of_several_threads(key, precision):
    dt = torch.complex128 if precision == pwlib.PW_FP64 else torch.complex64
    errors = []

    def work(box):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                L = np.array([0.25 * n for n in box])
                V = np.random.default_rng(1).standard_normal(box)
                ctx = pwlib.Context(np.diag(L), (0.0, 0.0, 0.0), 0.5 * (np.pi * 0.9 / 0.5) ** 2, box, V,
                                    np.zeros((0, 3)), np.zeros(0), np.zeros((0, 0)), None)
                g = torch.Generator(device="cuda").manual_seed(1)
                y = torch.randn((2, ctx.npw), dtype=torch.complex128, device="cuda", generator=g).to(dt)
                first, h = torch.empty_like(y), torch.empty_like(y)
                start.wait(timeout=60)
                ctx.hamiltonian_apply(y, first, None, precision=precision)
                for _ in range(300):
                    ctx.hamiltonian_apply(y, h, None, precision=precision)
                torch.cuda.current_stream().synchronize()
                if not torch.equal(first, h):
                    errors.append(f"{box}: another result")
        except Exception as e:
            errors.append(f"{box}: {e}")

    start = threading.Barrier(len(SETS[key]))
    threads = [threading.Thread(target=work, args=(box,)) for box in SETS[key]]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
