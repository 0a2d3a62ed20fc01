"""Workspace sizes (CPU): the tables of the line kernels are in the workspace of
the batches that can run them, and in no other."""
import ctypes as C
import os

import pytest

from synth import meshes as M


@pytest.fixture(scope="module")
def fr():
    from paper_2312_14167_gb300 import build, fr as module
    if not os.path.exists(os.path.join(os.path.dirname(module.__file__), "libfr.so")):
        build.build()
    return module


def _bytes(fr, meshes, **cfg):
    arr = (C.c_void_p * len(meshes))(*[m.handle for m in meshes])
    n = fr.lib().fr_workspace_bytes(arr, len(meshes), C.byref(fr.make_config(cfg.pop("dim"), p_inf=1.0, **cfg)))
    assert n > 0
    return n


def test_line_kernel_tables_are_sized_where_they_are_used(fr):
    n, p = 4, 3
    slots = 4 * 256                                        # alignment, and the slots of unused buffers
    for dim in (2, 3):
        mesh = fr.Mesh(M.periodic_box(dim, (n,) * dim, (0.0,) * dim, (1.0,) * dim), p)
        e, nsp, nfp, v = n ** dim, (p + 1) ** dim, 2 * dim * (p + 1) ** (dim - 1), dim + 2
        common = dict(dim=dim, viscous=True, mu=0.01, dt=1e-3, precision=fr.FR_FP32)
        record = e * nfp * 4 * dim * 4                     # face geometry of the line kernels
        metric = e * nsp * (dim * dim + 1) * 4 if dim == 3 else 0
        br2 = _bytes(fr, [mesh], **common)
        ldg = _bytes(fr, [mesh], viscous_scheme=fr.FR_VISC_LDG, **common)
        adaptive = _bytes(fr, [mesh], rk=fr.FR_BS32, rtol=1e-6, **common)
        if dim == 2:
            assert ldg == br2                              # both run line kernels
        else:
            assert abs(br2 - ldg - (record + metric)) <= slots
        assert abs(br2 - adaptive - (record + metric - e * nsp * v * 4 - e * 8)) <= slots
    # 3-D mortar faces: no line kernels (two degrees against each alone)
    mesh = M.periodic_box(3, (n,) * 3, (0.0,) * 3, (1.0,) * 3)
    degrees = M.checker_degrees(mesh, (2, 3), seed=3)
    common = dict(dim=3, viscous=True, mu=0.01, dt=1e-3, precision=fr.FR_FP32)
    mixed = [fr.Mesh(mesh, degrees)]
    assert _bytes(fr, mixed, **common) == _bytes(fr, mixed, viscous_scheme=fr.FR_VISC_LDG, **common)
    both = _bytes(fr, mixed, **common) - _bytes(fr, mixed, rk=fr.FR_BS32, rtol=1e-6, **common)
    points = sum(int((degrees == q).sum()) * (q + 1) ** 3 for q in (2, 3))
    assert abs(both + points * 5 * 4 + n ** 3 * 8) <= slots
