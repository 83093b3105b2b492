"""An instance's result does not depend on its neighbours: batches whose total
rows lie in another range of threads per row (12,000 / 45,000 / 200,000 rows
of the finest level) than each instance's own give the bits of the instances'
single solves, in FP64, FP32 and mixed precision."""
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


@pytest.mark.parametrize("count,smin,smax,edge", [(4, 18, 20, 12000), (12, 18, 20, 45000), (4, 28, 30, 45000),
                                                  (8, 38, 40, 200000)])
@pytest.mark.parametrize("prec", [0, 1, 4])
def test_bits_do_not_depend_on_the_neighbours(count, smin, smax, edge, prec):
    systems = [synth.generate(sp) for sp in synth.batch(count=count, seed=5, smin=smin, smax=smax)]
    assert max(d["n_nodes"] for d in systems) < edge <= sum(d["n_nodes"] for d in systems) / 2
    B = BatchSolver(systems, precision=prec)
    B.setup()
    xs, infos = B.solve([_t(d["b"]) for d in systems])
    B.close()
    for d, x, info in zip(systems, xs, infos):
        s = Solver(d, precision=prec)
        s.setup()
        x1, info1 = s.solve(_t(d["b"]))
        assert torch.equal(x, x1)
        assert info["A_iters"] == info1["A_iters"] and info["I_iters"] == info1["I_iters"]
        s.close()
