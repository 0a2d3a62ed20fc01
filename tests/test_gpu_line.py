"""The line kernels of FP32 BR2 stages (one thread per element line of every
direction) against the FP64 oracle at the edges of their tiles: element counts
around one warp and one CTA, every degree, neighbouring faces in every
orientation, both interface fluxes.

Residuals: the standard forward error bound of the FP32 sums on the path's own
FP32 input (16 roundings of the terms' magnitude).  Steps: 1e-6 of the state,
the bound of the mixed path's short horizons."""
import numpy as np
import pytest

from tests import fr_cases as FC
from oracle import timestep as T
from synth import meshes as M

pytestmark = pytest.mark.gpu

EPS32 = 2.0 ** -24


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _case(shape, p, flux="rusanov", rk="lsrk45"):
    dim = len(shape)
    mesh = M.reorient(M.periodic_box(dim, shape, (0.0,) * dim, (1.0, 0.9, 1.1)[:dim], jitter=0.2), 5)
    return FC.Case("line", [mesh], p, True, 0.01, 0.3, dt=1e-4, flux=flux, rk=rk, v_inf=(1.0, 0.0, 0.0)[:dim])


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("shape", [(3, 3), (8, 4), (11, 3), (5, 13), (3, 3, 3), (4, 4, 3), (3, 5, 7)])
def test_residual_at_tile_edges(shape, p):
    case = _case(shape, p, flux="roe" if shape[0] in (8, 4) else "rusanov")
    sol = FC.lib_solver(case, "fp32")
    assert "stage=fused" in sol.schedule()[0]
    disc = FC.oracle_disc(case)
    u = FC.initial_state(case, disc.sol_coords())
    sol.set_state(0, u)
    R32, mag = disc.residual(FC.fp32_input(case, u), magnitude=True)
    err = FC.rel_l2(sol.residual(0), R32)
    bound = 16 * EPS32 * np.linalg.norm(mag) / np.linalg.norm(R32)
    print(f"p={p} {shape}: {err:.2e} (bound {bound:.2e})")
    assert err < bound


@pytest.mark.parametrize("rk", ["rk4", "lsrk45"])
@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("shape", [(11, 3), (3, 3, 5)])
def test_steps_follow_the_oracle(shape, p, rk):
    case = _case(shape, p, rk=rk)
    sol = FC.lib_solver(case, "fp32")
    assert "stage=fused" in sol.schedule()[0]
    disc = FC.oracle_disc(case)
    u = FC.initial_state(case, disc.sol_coords())
    sol.set_state(0, u)
    sol.rk_step(5)
    step = T.rk4_step if rk == "rk4" else T.lsrk45_step
    for _ in range(5):
        u = step(disc.residual, u, case.dt)
    assert FC.rel_l2(sol.get_state(0), u) < 1e-6


@pytest.mark.parametrize("flux", ["rusanov", "roe"])
@pytest.mark.parametrize("degrees", [(0, 1, 2, 3), (1, 4), (0, 4), (2, 3)])
def test_mortar_faces(degrees, flux):
    """Several degrees in one mesh: every degree group's line kernel and the
    mortar faces between them (most faces here), residual and steps."""
    from oracle.fr_var import VarFRDiscretisation
    from paper_2312_14167_gb300 import fr
    case = _case((11, 7), 3, flux=flux)
    mesh = case.meshes[0]
    ep = M.checker_degrees(mesh, degrees, seed=3)
    disc = VarFRDiscretisation(mesh, ep, FC.oracle_disc(case).phys)
    sol = fr.Solver([fr.Mesh(mesh, ep)], FC.lib_config(case, "fp32"))
    assert "stage=fused" in sol.schedule()[0]
    u = FC.initial_state(case, disc.sol_coords())
    sol.set_state(0, u)
    ref = disc.residual(FC.fp32_input(case, u))
    assert FC.rel_l2(sol.residual(0), ref) < 1e-5
    sol.rk_step(5)
    for _ in range(5):
        u = T.lsrk45_step(disc.residual, u, case.dt)
    assert FC.rel_l2(sol.get_state(0), u) < 1e-6


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("shape,flux", [((3, 3), "rusanov"), ((11, 3), "roe"), (None, "rusanov"), (None, "roe")])
def test_ldg_lines(shape, flux, p):
    """LDG in the line kernels: one tile edge each, and (shape None) small
    airfoils with walls and far field, the second one off the tile grid."""
    if shape is None:
        case, inst = FC.airfoil_case(n_inst=2, p=p), 1
        case.flux = flux
    else:
        case, inst = _case(shape, p, flux=flux), 0
    case.viscous_scheme = "ldg"
    sol = FC.lib_solver(case, "fp32")
    for i in range(len(case.meshes)):
        disc = FC.oracle_disc(case, i)
        u = FC.initial_state(case, disc.sol_coords(), i)
        sol.set_state(i, u)
    R32, mag = disc.residual(FC.fp32_input(case, u), magnitude=True)
    err = FC.rel_l2(sol.residual(inst), R32)
    bound = 16 * EPS32 * np.linalg.norm(mag) / np.linalg.norm(R32)
    print(f"p={p} {shape} {flux}: {err:.2e} (bound {bound:.2e})")
    assert err < bound
    sol.rk_step(3)
    for _ in range(3):
        u = T.lsrk45_step(disc.residual, u, case.dt)
    assert FC.rel_l2(sol.get_state(inst), u) < 1e-6
