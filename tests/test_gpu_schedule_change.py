"""A schedule that fr_tune takes up when states are already set (a cached entry,
or the winner of a measurement): the next residual and steps are those of a
solver that had the schedule before its state was set.  What the face buffers
hold, and how they are laid out, depends on the schedule."""
import json

import numpy as np
import pytest

from tests import fr_cases as FC
from synth import meshes as M, states as S

pytestmark = pytest.mark.gpu

LINE, SPLIT = "stage=fused;regs=0;contract=simt", "stage=split;regs=0;contract=simt"
TC = "stage=fused;regs=0;contract=tc"


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _solver(case, degrees=None):
    from paper_2312_14167_gb300 import fr
    ps = [case.p if degrees is None else M.checker_degrees(m, degrees, seed=3) for m in case.meshes]
    return fr.Solver([fr.Mesh(m, p) for m, p in zip(case.meshes, ps)], FC.lib_config(case, "fp32"))


def _force(sol, schedule, tmp_path, mode=2):
    cache = tmp_path / "schedule.json"
    cache.write_text(json.dumps({sol.schedule()[1]: schedule + ";ms=1.0"}))
    assert schedule in sol.tune(str(cache), mode=mode)


def _box(shape):
    dim = len(shape)
    mesh = M.periodic_box(dim, shape, (0.0,) * dim, (1.0, 0.9, 1.1)[:dim], jitter=0.2)
    return FC.Case("change", [mesh], 3, True, 0.01, 0.3, dt=1e-4, v_inf=(1.0, 0.0, 0.0)[:dim])


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("shape,degrees,before,after", [
    ((3, 4, 3), None, LINE, SPLIT), ((3, 4, 3), None, LINE, TC), ((3, 4, 3), None, SPLIT, LINE),
    ((3, 4, 3), None, TC, LINE), ((7, 5), None, SPLIT, LINE), ((7, 5), (0, 1, 2, 3), LINE, SPLIT),
    ((7, 5), (0, 1, 2, 3), SPLIT, LINE)])
def test_cached_schedule_after_the_state(shape, degrees, before, after, mode, tmp_path):
    case = _box(shape)
    late, early = _solver(case, degrees), _solver(case, degrees)
    u = S.smooth_perturbed(late.meshes[0].sol_coords(), case.dim, case.mach, amp=0.05, seed=100)
    _force(late, before, tmp_path)
    late.set_state(0, u)
    _force(late, after, tmp_path, mode)
    _force(early, after, tmp_path)
    early.set_state(0, u)
    assert np.array_equal(late.residual(0), early.residual(0))
    late.rk_step(2)
    early.rk_step(2)
    assert np.array_equal(late.get_state(0), early.get_state(0))


@pytest.mark.parametrize("name", ["tandem", "airfoil"])
def test_measured_schedule_without_a_new_state(name, tmp_path):
    """A measurement leaves every instance some steps after the free stream;
    going on from there is going on from the same states set anew (to the
    rounding of the perturbation's way through FP64: 1e-6 of the state)."""
    case = FC.tandem_case(n_inst=2, n_hex=300, n_span=3, p=2) if name == "tandem" else FC.airfoil_case(n_inst=2)
    degrees = None if name == "tandem" else (2, 3)
    sol = _solver(case, degrees)
    sol.tune(str(tmp_path / "measured.json"), mode=1)
    u = sol.get_states()
    again = _solver(case, degrees)
    again.tune(str(tmp_path / "measured.json"), mode=0)
    again.set_states(u)
    for i in range(2):
        a, b = sol.residual(i), again.residual(i)
        assert np.all(np.isfinite(b)) and np.linalg.norm(a - b) < 1e-3 * np.linalg.norm(b)
    sol.rk_step(2)
    again.rk_step(2)
    a, b = sol.get_states(), again.get_states()
    assert np.linalg.norm(a - b) < 1e-6 * np.linalg.norm(b)


def test_measured_time_is_the_steps_time(tmp_path):
    """The tuner times steps as fr_rk_step runs them: on a batch of four small
    degree groups (parallel branches of the captured step; one by one they take
    over twice as long) its time per step is that of the steps that follow,
    within a half.  The least of five on both sides."""
    import torch
    sol = _solver(_box((11, 7)), (0, 1, 2, 3))
    told = []
    for _ in range(5):
        sol.tune(None, mode=1)
        told.append(float(dict(kv.split("=", 1) for kv in sol.schedule()[0].split(";"))["ms"]))
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    took = []
    sol.rk_step(3)
    for _ in range(5):
        torch.cuda.synchronize()
        a.record(sol.stream)
        sol.rk_step(3)
        b.record(sol.stream)
        torch.cuda.synchronize()
        took.append(a.elapsed_time(b) / 3)
    print(f"told {min(told):.4f} ms, took {min(took):.4f} ms")
    assert min(told) < 1.5 * min(took)


@pytest.mark.parametrize("scheme", ["br2", "ldg"])
def test_no_kernel_is_measured_twice(scheme):
    """The fused kernel of hexes and the 2-D LDG kernels have one register level."""
    case = _box((3, 4, 3) if scheme == "br2" else (7, 5))
    case.viscous_scheme = scheme
    choice = _solver(case).tune(None, mode=1)
    told = [c.split("=")[0] for c in choice.split("candidates=")[1].split(",")]
    tc = [f"{s}/{r}/tc" for s in (("split", "fused") if scheme == "br2" else ("split",)) for r in (0, 1, 2)]
    assert told == (["split/0/simt", "split/1/simt", "split/2/simt", "fused/0/simt"] if scheme == "br2"
                    else ["split/0/simt"]) + tc
