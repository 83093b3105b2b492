"""The numbers of A-, S- and inner solves in the information of a solve: both
loops count them, two intermediate A-solves and one S-solve to an outer
iteration, one inner solve to an application of S."""
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1911_10814_gb300 import BatchSolver, Solver  # noqa: E402


def test_solves_are_counted_by_both_loops():
    d = synth.generate(synth.MeshSpec(6, 5, 7, Re=200.0, seed=8, R=(1e3,)))
    b = torch.as_tensor(d["b"], device="cuda:0")
    s = Solver(d, precision=1)
    s.setup()
    B = BatchSolver([d, d], precision=1)
    B.setup()
    for info in (s.solve(b, device_loop=0)[1], s.solve(b, device_loop=1)[1], *B.solve([b, b], device_loop=1)[1]):
        assert info["outer_iters"] > 0
        assert info["n_A_solves"] == 2 * info["outer_iters"]
        assert info["n_S_solves"] == info["outer_iters"]
        assert info["n_I_solves"] == info["S_iters"]
    s.close()
    B.close()
