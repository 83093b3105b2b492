"""Setup kernels at the edges of their sizes.

Matching: graphs larger than the one-cluster kernel takes start with rounds
over the whole GPU; the aggregates must equal the oracle's whichever kernel ran.

Dense coarsest inverse (blocked Gauss-Jordan): a hierarchy of one level is
that inverse, so a cycle solves A x = b.  Backward error of Gauss-Jordan with
partial pivoting: ||A x - b|| <= c n eps kappa_1(A) ||b|| with a modest c; the
bar is c = 10.  Sizes: not multiples of the 8-column panel, one panel and a
bit, and beyond 3,300, where panels have 4 columns."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1911_10814_gb300 import Solver  # noqa: E402


@pytest.mark.parametrize("nx,ny,nz", [(3, 2, 5), (23, 25, 27), (27, 26, 28)])
def test_aggregates_match_oracle(nx, ny, nz):
    d = synth.generate(synth.MeshSpec(nx, ny, nz, Re=700.0, seed=nx, R=(1e3, 1e2)))
    s = Solver(d)
    s.setup()
    o = oracle.Oracle(d)
    o.setup()
    for which in (0, 1):
        got, ref = s.amg_levels(which), o.amg_levels(which)
        assert len(got) == len(ref)
        for lg, lo in zip(got, ref):
            assert np.array_equal(lg["rowptr"], lo["rowptr"])
            if lo["agg"] is not None:
                assert np.array_equal(lg["agg"], lo["agg"])
    s.close()


@pytest.mark.parametrize("nx,ny,nz", [(1, 1, 1), (2, 2, 2), (4, 3, 3), (9, 9, 12)])
def test_dense_inverse(nx, ny, nz):
    d = synth.generate(synth.MeshSpec(nx, ny, nz, Re=200.0, seed=2, R=(1e3,)))
    N = d["n_nodes"]
    s = Solver(d, amg_max_levels=1)
    s.setup()
    n = 3 * N
    A = np.zeros((N, 3, N, 3))
    rows = np.repeat(np.arange(N), np.diff(d["rowptr"]))
    A[rows, :, d["col"], :] = d["A"]
    A = A.reshape(n, n)
    kappa = np.abs(A).sum(0).max() * np.abs(np.linalg.inv(A)).sum(0).max()
    b = np.random.default_rng(1).uniform(-1, 1, n)
    x = s.vcycle(0, torch.as_tensor(b, device="cuda:0")).cpu().numpy()
    assert np.linalg.norm(A @ x - b) <= 10 * n * 2.0**-53 * kappa * np.linalg.norm(b)
    s.close()
