"""The gradient + flux kernels of FP32 batches as chosen by the tuner (stages
run line kernels by default): every register level on hexes and on mortar
faces, and the tensor-core contraction of 2-D LDG.  Residual within the forward
error bound of its FP32 sums (16 roundings of the terms); one step within the
roundings of its stages (twice that for their weights, and one of the stored
perturbation per stage)."""
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


@pytest.mark.parametrize("shape,p,degrees,scheme,schedule", [
    ((3, 4, 3), p, None, "br2", f"split;regs={r};contract=simt") for p in (2, 3, 4) for r in (0, 1, 2)] + [
    ((11, 7), 3, (0, 1, 2, 3), "br2", f"split;regs={r};contract={c}") for r in (0, 1, 2) for c in ("simt", "tc")] + [
    ((7, 5), p, None, "ldg", f"split;regs={r};contract=tc") for p in (1, 3, 4) for r in (0, 2)] + [
    ((7, 5), 0, None, "ldg", "split;regs=0;contract=simt")])
def test_tile_schedule_matches_the_oracle(shape, p, degrees, scheme, schedule, tmp_path):
    from oracle.fr_var import VarFRDiscretisation
    from paper_2312_14167_gb300 import fr
    dim = len(shape)
    mesh = M.reorient(M.periodic_box(dim, shape, (0.0,) * dim, (1.0, 0.9, 1.1)[:dim], jitter=0.2), 5)
    case = FC.Case("tiles", [mesh], p, True, 0.01, 0.3, dt=1e-4, v_inf=(1.0, 0.0, 0.0)[:dim], viscous_scheme=scheme)
    disc, deg = FC.oracle_disc(case), p
    if degrees:
        deg = M.checker_degrees(mesh, degrees, seed=3)
        disc = VarFRDiscretisation(mesh, deg, disc.phys)
    sol = fr.Solver([fr.Mesh(mesh, deg)], FC.lib_config(case, "fp32"))
    cache = tmp_path / "schedule.json"
    cache.write_text(json.dumps({sol.schedule()[1]: f"stage={schedule};ms=1.0"}))
    assert schedule in sol.tune(str(cache), mode=2)
    u = FC.fp32_input(case, FC.initial_state(case, disc.sol_coords()))
    sol.set_state(0, u)
    R, mag = disc.residual(u, magnitude=True)
    err, bound = FC.rel_l2(sol.residual(0), R), 16 * EPS32 * np.linalg.norm(mag) / np.linalg.norm(R)
    print(f"residual {err:.2e} (bound {bound:.2e})")
    assert err < bound
    sol.rk_step(1)
    ref = S.reference_conserved(dim, 1.0, case.v_inf, case.p_inf, FC.GAMMA)
    bound = EPS32 * (32 * case.dt * np.linalg.norm(mag) + 5 * np.linalg.norm(u - ref))
    err = np.linalg.norm(sol.get_state(0) - T.lsrk45_step(disc.residual, u, case.dt))
    print(f"step {err:.2e} (bound {bound:.2e})")
    assert err < bound
