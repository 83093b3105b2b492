"""Every call allocates from the pool of the context that it works on: a batch
solved after calls on another context leaves that context's memory alone, and
one closed by another thread is not asked for any."""
import threading

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1911_10814_gb300 import BatchSolver, Solver  # noqa: E402


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda:0")


def _other():
    s = Solver(synth.generate(synth.tiny()))
    s.setup()
    return s


@pytest.mark.parametrize("loop", [0, 1])
def test_batch_takes_its_memory_from_its_own_contexts(loop):
    systems = [synth.generate(sp) for sp in synth.batch(count=3, seed=4, smin=5, smax=8)]
    bs = [_t(d["b"]) for d in systems]
    B = BatchSolver(systems, precision=1)
    B.setup()
    other = _other()             # this thread's last call is on another context
    used = other.memory()["used"]
    assert used > 0
    xs, _ = B.solve(bs, device_loop=loop)
    assert other.memory()["used"] == used
    closing = threading.Thread(target=other.close)
    closing.start()
    closing.join()
    B2 = BatchSolver(systems, precision=1)
    B2.setup()
    other = _other()
    closing = threading.Thread(target=other.close)   # the last context is gone
    closing.start()
    closing.join()
    xs2, _ = B2.solve(bs, device_loop=loop)
    for x, x2 in zip(xs, xs2):
        assert torch.equal(x, x2)
    B.close()
    B2.close()

