"""Cycles and solves on levels that keep the prolongation and the full product:
a row of A P with more than 64 coarse columns leaves its level without it.  One
node coupled with every other has such a row on the finest level of both
hierarchies.  FP64 cycles against the oracle's to the 1e-10 of the other cycle
tests, solves in every precision and both loops to the requested residual."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1911_10814_gb300 import Solver  # noqa: E402
from test_gpu_setup_paths import with_dense_row  # noqa: E402

AP_CAPACITY = 64
RTOL = 1e-9


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda:0")


@pytest.fixture(scope="module")
def dense():
    d = synth.generate(synth.MeshSpec(11, 11, 11, Re=100.0, seed=3, R=(1e3, 1e4)))
    return with_dense_row(d, 6 * 144 + 6 * 12 + 6)


@pytest.mark.parametrize("opts", [dict(amg_coarse_max=20), dict(amg_cycle=0), dict(amg_cycle=2, cheb_degree=1, amg_coarse_max=20),
                                  dict(amg_coarse_max=20, cheb_degree=3, cheb_degree_S=2)])
def test_cycles_and_solves(dense, opts):
    d = dense
    o = oracle.Oracle(d, **opts)
    o.setup()
    rng = np.random.default_rng(5)
    s = Solver(d, **opts)
    s.setup()
    for which, n in ((0, 3 * d["n_nodes"]), (1, d["n_nodes"])):
        L = s.amg_levels(which)[0]
        coarse = [np.unique(L["agg"][L["col"][a:b]]) for a, b in zip(L["rowptr"], L["rowptr"][1:])]
        assert max((c >= 0).sum() for c in coarse) > AP_CAPACITY
        b = rng.standard_normal(n)
        ref = o.vcycle(which, b)
        for _ in range(2):   # the second replays the captured graph
            x = s.vcycle(which, _t(b)).cpu().numpy()
            assert np.linalg.norm(x - ref) <= 1e-10 * np.linalg.norm(ref)
    s.close()
    for precision in (0, 1, 4):
        s = Solver(d, precision=precision, **opts)
        s.setup()
        for loop in (1, 0):
            x, _ = s.solve(_t(d["b"]), device_loop=loop, rtol=RTOL)
            r = d["b"] - o.apply_full(x.cpu().numpy())
            assert np.linalg.norm(r) <= 1.01 * RTOL * np.linalg.norm(d["b"])
        s.close()
