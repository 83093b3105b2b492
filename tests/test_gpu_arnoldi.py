"""The device-driven Arnoldi step at the edges of its kernels: bases longer
than the 32 columns of the one-warp triangular solve and the 64 columns that
the Givens update stages in shared memory, restarts, one and two Gram-Schmidt
passes, and every precision mode; vector lengths that are not multiples of a
16-byte piece.

Both loops (device- and host-driven) are the same GMRES in other summation
orders, so each must reach the requested residual, and their solutions, solved
to rtol, agree to a small multiple of it: 100 rtol covers the ratio of error to
residual of these tangents (measured below 20 in test_conditioning.py) on both
sides."""
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


def _check(d, s, b, min_its=0, **kw):
    xs = []
    for loop in (1, 0):
        x, info = s.solve(b, device_loop=loop, rtol=RTOL, **kw)
        xs.append(x.cpu().numpy())
        r = d["b"] - oracle.Oracle(d).apply_full(xs[-1])
        assert np.linalg.norm(r) <= 1.01 * RTOL * np.linalg.norm(d["b"])
        assert info["A_iters"] >= min_its
    assert np.linalg.norm(xs[0] - xs[1]) <= 100 * RTOL * np.linalg.norm(xs[1])


@pytest.mark.parametrize("precision", [0, 1])
def test_long_bases(precision):
    """Point Jacobi and a tight A tolerance: A-solves of more than 64 steps."""
    d = synth.generate(synth.MeshSpec(9, 7, 11, Re=300.0, seed=3, R=(1e3, 1e2)))
    s = Solver(d, precision=precision, pc_A=1, rtol_A=1e-5 if precision else 1e-9)
    s.setup()
    _check(d, s, torch.as_tensor(d["b"], device="cuda:0"), min_its=2 * 65)
    s.close()


@pytest.mark.parametrize("nx,ny,nz", [(2, 2, 3), (5, 4, 6), (13, 12, 17)])
@pytest.mark.parametrize("precision,passes", [(0, 1), (0, 2), (4, 1), (1, 2)])
def test_odd_lengths(nx, ny, nz, precision, passes):
    d = synth.generate(synth.MeshSpec(nx, ny, nz, Re=400.0, seed=nx, R=(1e3,)))
    s = Solver(d, precision=precision, gs_passes_I=passes)
    s.setup()
    _check(d, s, torch.as_tensor(d["b"], device="cuda:0"))
    s.close()


@pytest.mark.parametrize("nx,ny,nz,precision", [(21, 21, 21, 0), (22, 21, 21, 0), (26, 27, 27, 1), (27, 27, 27, 4)])
def test_cluster_length(nx, ny, nz, precision):
    """Either side of the longest vector (32,768 doubles, 65,536 floats) whose
    step runs in one cluster: A-vectors of 31,944 / 33,396 and 63,504 / 65,856."""
    d = synth.generate(synth.MeshSpec(nx, ny, nz, Re=400.0, seed=nx, R=(1e3,)))
    s = Solver(d, precision=precision)
    s.setup()
    _check(d, s, torch.as_tensor(d["b"], device="cuda:0"))
    s.close()
