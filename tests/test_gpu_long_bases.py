"""Device-driven Arnoldi steps on bases that are known to be long: the mean
number of steps of an A-solve is above the edge, so some basis is past it.

Grid kernels on vectors longer than the cluster step's (32,768 doubles, 65,536
floats) past the 64 columns that the Givens update stages in shared memory, and
bases past the 256 coefficients that the norm pass keeps there (bases that long
never take the cluster), one and two Gram-Schmidt passes in the inner solves.
Large time steps make the A-solves of point Jacobi long.

Both loops are the same GMRES in other summation orders: each reaches the
requested residual, and a step that lost orthogonality would cost steps: the
mean numbers agree within two, one for a residual estimate within rounding of
the tolerance and one for a right-hand side from other inexact inner solves."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1911_10814_gb300 import Solver  # noqa: E402

RTOL = 1e-9


def _solves(d, precision, **opts):
    b = torch.as_tensor(d["b"], device="cuda:0")
    s = Solver(d, precision=precision, pc_A=1, **opts)
    s.setup()
    o = oracle.Oracle(d)
    infos = []
    for loop in (1, 0):
        x, info = s.solve(b, device_loop=loop, rtol=RTOL)
        r = d["b"] - o.apply_full(x.cpu().numpy())
        assert np.linalg.norm(r) <= 1.01 * RTOL * np.linalg.norm(d["b"])
        infos.append(info)
    s.close()
    mean = [i["A_iters"] / i["n_A_solves"] for i in infos]
    assert abs(mean[0] - mean[1]) <= 2
    return min(mean), infos


@pytest.mark.parametrize("precision,n,dt,rtol_A,passes", [(0, (22, 22, 22), 0.2, 1e-9, 2), (1, (28, 27, 28), 1.0, 1e-6, 1)])
def test_past_the_staged_columns_on_the_grid(precision, n, dt, rtol_A, passes):
    d = synth.generate(synth.MeshSpec(*n, Re=10.0 if precision else 100.0, dt=dt, seed=3, R=(1e3, 1e2)))
    assert 3 * d["n_nodes"] > (65536 if precision else 32768)
    steps, _ = _solves(d, precision, rtol_A=rtol_A, gs_passes_I=passes)
    assert steps > 64


@pytest.mark.parametrize("precision", [0, 1])
def test_past_the_kept_coefficients(precision):
    """No tolerance at all (the residual estimate, a product of sines, goes on
    falling where the residual no longer does): every A-solve takes all 320 steps."""
    d = synth.generate(synth.MeshSpec(5, 4, 6, Re=100.0, seed=3, R=(1e3, 1e2)))
    steps, infos = _solves(d, precision, rtol_A=0.0, atol=0.0, m_A=320, nmax_A=320)
    assert steps == 320
    assert all(i["A_iters"] == 320 * i["n_A_solves"] for i in infos)
