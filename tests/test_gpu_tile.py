"""FP64 tile kernels with fewer elements per CTA than a full tile (batches
smaller than the chip): residual and steps against the oracle at element
counts whose tiles are one element, a few, and not a divisor of the batch.
The bound is the FP64 path's, 1e-12 relative L2."""
import pytest

from tests import fr_cases as FC
from oracle import timestep as T
from synth import meshes as M

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("viscous", [False, True])
@pytest.mark.parametrize("shape,p", [((3, 3), 4), ((17, 9), 1), ((31, 29), 2), ((3, 3, 4), 2), ((5, 7, 5), 1)])
def test_small_tiles(shape, p, viscous):
    dim = len(shape)
    mesh = M.reorient(M.periodic_box(dim, shape, (0.0,) * dim, (1.0,) * dim, jitter=0.2), 7)
    case = FC.Case("tile", [mesh], p, viscous, 0.01 if viscous else 0.0, 0.3, dt=1e-4,
                   v_inf=(1.0, 0.0, 0.0)[:dim])
    sol, disc = FC.lib_solver(case, "fp64"), FC.oracle_disc(case)
    u = FC.initial_state(case, disc.sol_coords())
    sol.set_state(0, u)
    assert FC.rel_l2(sol.residual(0), disc.residual(u)) < 1e-12
    sol.rk_step(2)
    for _ in range(2):
        u = T.lsrk45_step(disc.residual, u, case.dt)
    assert FC.rel_l2(sol.get_state(0), u) < 1e-12
