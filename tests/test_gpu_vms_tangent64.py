"""The FP64 tangent of the tets (k_tan_tet64, four lanes per tet) against the
oracle at its edges: few tets (blocks with idle lanes), any vertex order of a
tet (both signs of its determinant), and tau frozen at another velocity.
Both sides sum the same FP64 terms in another order; the bar is that of the
other FP64 assembly tests, 1e-12 of each array's largest entry."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1911_10814_gb300 import Solver, Vms  # noqa: E402


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda:0")


@pytest.mark.parametrize("nx,ny,nz", [(2, 2, 2), (3, 2, 2), (3, 5, 7)])
@pytest.mark.parametrize("frozen", [False, True])
def test_tangent64(nx, ny, nz, frozen):
    spec = synth.MeshSpec(nx, ny, nz, Lz=1.3, Re=300.0, seed=5, R=(1e3,))
    d, m = synth.generate(spec), synth.mesh(spec)
    rng = np.random.default_rng(nx + 10 * ny + 100 * nz)
    m = dict(m, tets=np.stack([t[rng.permutation(4)] for t in m["tets"]]))
    N = d["n_nodes"]
    v = rng.standard_normal(3 * N)
    vd, p = 40.0 * rng.standard_normal(3 * N), 80.0 * rng.standard_normal(N)
    vt = rng.standard_normal(3 * N) if frozen else None
    ref = oracle.vms_assemble(m, d, oracle.vms_phys(spec), vd, v, p, vtau=vt, residual=False)
    s = Solver(d)
    vm = Vms(s, m, spec.rho, spec.mu, spec.dt, spec.rho_inf, tangent_fp32=False)
    got = vm.tangent(_t(vd), _t(v), _t(p), vtau=_t(vt) if frozen else None)
    for k in "ABCD":
        a, b = got[k].cpu().numpy(), np.ravel(ref[k])
        assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max(), k
    vm.close()
    s.close()
