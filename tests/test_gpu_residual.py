"""Residuals and conservation sums of FP32 batches whose stages run line
kernels: the values of the gradient + flux kernels, bit for bit, whatever the
schedule; and evaluating them leaves the following steps as they are.

One step of the line kernels at the edges of their tiles: the change of the
state against the oracle's, within the roundings of the step (16 of the
residual's terms per stage, twice for the five stages' weights, and one of the
stored perturbation per stage)."""
import json

import numpy as np
import pytest

from tests import fr_cases as FC
from oracle import timestep as T
from synth import meshes as M, states as S

pytestmark = pytest.mark.gpu

EPS32 = 2.0 ** -24


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _case(shape, p):
    dim = len(shape)
    mesh = M.reorient(M.periodic_box(dim, shape, (0.0,) * dim, (1.0, 0.9, 1.1)[:dim], jitter=0.2), 5)
    return FC.Case("residual", [mesh], p, True, 0.01, 0.1, dt=1e-4, v_inf=(1.0, 0.0, 0.0)[:dim])


def _solver(case, degrees=None):
    from paper_2312_14167_gb300 import fr
    mesh = case.meshes[0]
    p = case.p if degrees is None else M.checker_degrees(mesh, degrees, seed=3)
    return fr.Solver([fr.Mesh(mesh, p)], FC.lib_config(case, "fp32"))


def _force(sol, schedule, tmp_path):
    cache = tmp_path / "schedule.json"
    cache.write_text(json.dumps({sol.schedule()[1]: schedule + ";ms=1.0"}))
    assert schedule in sol.tune(str(cache), mode=2)


@pytest.mark.parametrize("shape,p,degrees", [((3, 3, 5), 1, None), ((3, 3, 5), 2, None), ((4, 3, 3), 3, None),
                                             ((3, 3, 3), 4, None), ((5, 13), 0, None), ((5, 13), 3, None),
                                             ((11, 7), 3, (0, 1, 2, 3)), ((11, 7), 4, (1, 4))])
def test_residual_does_not_depend_on_the_schedule(shape, p, degrees, tmp_path):
    case = _case(shape, p)
    line, split = _solver(case, degrees), _solver(case, degrees)
    assert "stage=fused" in line.schedule()[0]
    _force(split, "stage=split;regs=0;contract=simt", tmp_path)
    x = line.meshes[0].sol_coords()
    u = S.smooth_perturbed(x, case.dim, case.mach, amp=0.05, seed=100)
    for sol in (line, split):
        sol.set_state(0, u)
    assert np.array_equal(line.residual(0), split.residual(0))
    assert np.array_equal(line.conservation(0), split.conservation(0))
    plain = _solver(case, degrees)
    plain.set_state(0, u)
    for _ in range(2):
        plain.rk_step(1)
        line.rk_step(1)
        line.residual(0)
        line.conservation(0)
    assert np.array_equal(line.get_state(0), plain.get_state(0))


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("shape", [(3, 3), (8, 4), (11, 3), (5, 13), (3, 3, 3), (4, 4, 3), (3, 5, 7)])
def test_one_step_at_tile_edges(shape, p):
    case = _case(shape, p)
    sol, disc = _solver(case), FC.oracle_disc(case)
    assert "stage=fused" in sol.schedule()[0]
    u = FC.fp32_input(case, FC.initial_state(case, disc.sol_coords()))
    sol.set_state(0, u)
    sol.rk_step(1)
    got, want = sol.get_state(0), T.lsrk45_step(disc.residual, u, case.dt)
    ref = S.reference_conserved(case.dim, 1.0, case.v_inf, case.p_inf, FC.GAMMA)
    mag = disc.residual(u, magnitude=True)[1]
    bound = EPS32 * (32 * case.dt * np.linalg.norm(mag) + 5 * np.linalg.norm(u - ref))
    err = np.linalg.norm(got - want)
    print(f"p={p} {shape}: {err:.2e} (bound {bound:.2e}, step {np.linalg.norm(want - u):.2e})")
    assert err < bound
