"""What the tuners time is what runs.  A coarse level's product kernel is chosen for the work that the level does:
a context with another cycle or smoothing degree times it anew, one with the
same options and shapes does not.  The Gram-Schmidt grids are timed per loop,
and not for vectors whose device-driven steps run in one cluster."""
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1911_10814_gb300 import Solver, load  # noqa: E402


def test_choices_belong_to_the_cycle_they_were_timed_in():
    d = synth.generate(synth.MeshSpec(15, 16, 17, Re=300.0, seed=21, R=(1e3,)))
    counts = [load().nbp_tuned_shapes(0)]
    for opts in (dict(amg_cycle=0), dict(amg_cycle=0), dict(amg_cycle=2), dict(amg_cycle=2), dict(amg_cycle=2, cheb_degree=3)):
        s = Solver(d, precision=1, amg_kdepth=1, **opts)
        s.setup()
        levels = [len(s.amg_levels(w)) for w in (0, 1)]
        s.close()
        counts.append(load().nbp_tuned_shapes(0))
    new = [b - a for a, b in zip(counts, counts[1:])]
    # tuned: the levels between the finest and the coarsest (dense) one
    assert all(n >= 3 for n in levels), levels
    assert new[0] == sum(n - 2 for n in levels)
    assert new[1] == 0
    assert new[2] == 2          # level 1 of both hierarchies runs a K-cycle now
    assert new[3] == 0
    assert new[4] == levels[0] - 2   # another degree on AMG(A)


def _tuned_by(s, b, loop):
    before = load().nbp_tuned_shapes(1)
    s.solve(b, device_loop=loop)
    return load().nbp_tuned_shapes(1) - before


@pytest.mark.parametrize("nx,ny,nz,device", [(7, 9, 10, 0), (27, 27, 28, 2)])
def test_gram_schmidt_grids_of_the_kernels_that_run(nx, ny, nz, device):
    """FP64 outer vectors of 4N, FP32 inner ones of 3N and N: all below the
    cluster's 32,768 doubles and 65,536 floats (880 nodes), or the last alone
    (22,736 nodes)."""
    d = synth.generate(synth.MeshSpec(nx, ny, nz, Re=300.0, seed=22, R=(1e3,)))
    b = torch.as_tensor(d["b"], device="cuda:0")
    for loops, new in (((1, 1), (device, 0)), ((0, 0), (3, 0))):
        s = Solver(d, precision=1)
        s.setup()
        assert tuple(_tuned_by(s, b, loop) for loop in loops) == new
        s.close()
